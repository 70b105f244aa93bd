"""The screen of a group's members at its edges: groups of a tile of 1024 and one
more or less, of a warp and one more or less, strings that use one to four
32-bit words with electrons in the highest orbitals; pairs exact and elements
within 1e-12 of the oracle, upper triangle and products on the fly alike."""
import numpy as np
import pytest

import oracle
import shci_synth as S
from tests import gpu_common as G
from tests.test_gpu_opposite import _dets, _strings

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_orb", [32, 33, 64, 65, 96, 97])
@pytest.mark.parametrize("size", [1, 31, 33, 1023, 1025])
def test_groups_at_tile_edges(n_orb, size):
    P = G.lib()
    rng = np.random.default_rng(size)
    words = S.n_words(n_orb)
    # three electrons among the lowest four and the highest fifteen orbitals
    s = _strings(list(range(4)) + list(range(n_orb - 15, n_orb)), 3)[::-1]
    big = s[rng.permutation(969)] if size > 969 else s
    b = (np.concatenate([big, _strings(range(4, 17), 3)]) if size > 969 else s[rng.permutation(969)])[:size]
    b = np.array(sorted(set(b)), dtype=object)
    a = np.repeat(np.array([s[0], s[1], s[400]], dtype=object), [b.size, min(b.size, 40), min(b.size, 7)])
    dets = _dets(a, np.concatenate([b, b[:40], b[:7]]), words)
    h, eri, ec = S.integrals(n_orb, 3, 12)
    ii, jj = oracle.pairs_allpairs(dets)
    v = oracle.System(h, eri, ec).hij_list(dets, ii, jj)
    for swap in (False, True):                             # the beta groups' screen too
        d = np.ascontiguousarray(np.concatenate([dets[:, words:], dets[:, :words]], axis=1)) if swap else dets
        B = G.Built(P, h, eri, ec, d, 3, 3)
        gi, gj, gv = B.pairs()
        assert np.array_equal(gi, ii) and np.array_equal(gj, jj)
        assert (np.max(np.abs(gv - v)) if v.size else 0.0) < 1e-12
        x = S.random_vectors(B.n, 2, 4)
        want = B.sigma(x)
        for mode in (P.SHCI_STORED_UPPER, P.SHCI_ON_THE_FLY):
            C = G.Built(P, h, eri, ec, d, 3, 3, mode=mode)
            assert C.nnz == B.nnz
            assert np.max(np.abs(C.sigma(x) - want)) < 1e-12 * max(1.0, np.max(np.abs(want)))
            C.close()
        B.close()
