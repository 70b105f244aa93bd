"""shci_select_alloc at its ends: an allocator that returns NULL, one that raises
(through the Python call), a selection without new determinants, no allocator;
the context stays usable and selects what it selected before."""
import ctypes

import numpy as np
import pytest

import shci_synth as S
from paper_1809_04600_gb300 import binding
from tests import gpu_common as G

pytestmark = pytest.mark.gpu


def _context(P):
    cfg, h, eri, ec, dets = G.system("sel_24o_6a6b_1m", 600)
    B = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta, mode=P.SHCI_ON_THE_FLY)
    return B, G.dev(S.random_vectors(B.n, 1, 3))


@pytest.mark.parametrize("host", [False, True])
def test_allocators(monkeypatch, host):
    P = G.lib()
    B, c = _context(P)
    c = c.cpu().numpy() if host else c
    want = P.shci_select(B.ctx.handle, c, 1e-3)
    as_host = lambda x: np.asarray(x if host else x.cpu().numpy().view(np.uint64))
    assert want.shape[0] > 0

    def call(alloc, eps1):
        lib = P.load_library()
        pc, mem, keep = binding._ptr(c, np.float64)
        n = ctypes.c_int64(-1)
        return lib.shci_select_alloc(B.ctx.handle, 1, pc, eps1, alloc, None, ctypes.byref(n), mem), n.value

    asked = []
    null = binding.ALLOC_ROWS(lambda user, rows: asked.append(rows))       # returns NULL
    assert call(null, 1e-3) == (binding.SHCI_ERR_OOM, want.shape[0]) and asked == [want.shape[0]]
    assert call(null, 1e6) == (binding.SHCI_OK, 0) and len(asked) == 1     # nothing to place: not called
    assert call(ctypes.cast(None, binding.ALLOC_ROWS), 1e-3)[0] == binding.SHCI_ERR_INVALID
    assert P.shci_select(B.ctx.handle, c, 1e6).shape == (0, 2)

    # an exception in the allocator reaches the caller as itself
    class Full(Exception):
        pass

    def empty(*a, **k):
        raise Full()

    with monkeypatch.context() as m:
        m.setattr(np if host else __import__("torch"), "empty", empty)
        with pytest.raises(Full):
            P.shci_select(B.ctx.handle, c, 1e-3)
    assert np.array_equal(as_host(P.shci_select(B.ctx.handle, c, 1e-3)), as_host(want))
    B.close()
