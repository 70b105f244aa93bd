"""Two contexts in two host threads (the calls release the interpreter's lock),
one with a table of opposite-spin words of a few hundred bytes, one of more
than 48 KB: the kernels' launch limits are the process's, and neither context's
may fail or change the other's results."""
import threading

import numpy as np
import pytest
import torch

import shci_synth as S
from tests import gpu_common as G
from tests.test_gpu_opposite import _dets, _strings

pytestmark = pytest.mark.gpu

ROUNDS = 300


def test_contexts_with_small_and_large_tables():
    P = G.lib()
    # 20,475 beta strings (80 KB of words) and 70 (280 bytes)
    b = _strings(range(28), 4)
    large = _dets(np.repeat(np.array([1, 2], dtype=object), b.size), np.tile(b, 2), 1)
    small = S.fci_dets(8, 1, 4)
    built, x, want = [], [], []
    for n_orb, na, nb, dets in ((28, 1, 4, large), (8, 1, 4, small)):
        h, eri, ec = S.integrals(n_orb, 4, 3)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            B = G.Built(P, h, eri, ec, dets, na, nb, mode=P.SHCI_ON_THE_FLY)
            built.append(B)
            x.append(G.dev(S.random_vectors(B.n, 1, 5)))
            want.append(B.sigma(x[-1].cpu().numpy()))
    failed = []
    start = threading.Barrier(2)

    def run(t):
        try:
            y = torch.empty_like(x[t])
            start.wait()
            for _ in range(ROUNDS if t == 0 else 8 * ROUNDS):
                P.shci_sigma(built[t].ctx.handle, x[t], y)
            if not np.array_equal(y.cpu().numpy(), want[t]):
                failed.append((t, "another product"))
        except Exception as e:  # reported by the main thread
            failed.append((t, e))

    threads = [threading.Thread(target=run, args=(t,)) for t in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for B in built:
        B.close()
