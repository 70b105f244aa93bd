"""Sort keys of more than one word: digits that no key differs in cost no pass,
and the edges of the tiles of two- and four-word keys (1,280 and 768 elements)."""
import numpy as np
import pytest

import oracle
import shci_synth as S
from tests import gpu_common as G
from tests.test_gpu_opposite import _dets, _strings
from tests.test_gpu_sort_edges import BAND, _rows

pytestmark = pytest.mark.gpu


def test_constant_digits_are_not_sorted_by():
    """V within 17 of 70 orbitals: two spins of three digits, where 70 orbitals have nine."""
    P = G.lib()
    s = _strings(range(17), 3)
    pick = np.random.default_rng(1).choice(s.size * s.size, 2000, replace=False)
    dets = _dets(s[pick // s.size], s[pick % s.size], 2)
    h, eri, ec = S.integrals(70, 4, 9)
    B = G.Built(P, h, eri, ec, dets, 3, 3, mode=P.SHCI_ON_THE_FLY)
    c = G.dev(S.random_vectors(B.n, 1, 2)[0])
    launches = []
    for _ in range(2):                            # the first call builds the sorted lists
        before = B.stats()["kernel_launches"]
        assert P.shci_pt2(B.ctx.handle, c, -1e3, 1e6) == (0.0, 0)
        launches.append(B.stats()["kernel_launches"] - before)
    # a pass is a histogram, a scan of up to three launches and a scatter; besides: the screen
    # and its scan, the keys, the reduction
    assert launches[1] <= 6 * 5 + 6, launches
    B.close()


@pytest.mark.parametrize("n_orb,tile", [(40, 1280), (70, 768)])
@pytest.mark.parametrize("off", [-1, 0, 1])
def test_tile_edges_of_long_keys(n_orb, tile, off):
    """As many determinants of V as a tile holds, one fewer and one more."""
    P = G.lib()
    n = tile + off
    s = _strings(list(range(6)) + list(range(n_orb - 6, n_orb)), 2)
    pick = np.random.default_rng(n).choice(s.size * s.size, n, replace=False)
    dets = _dets(s[pick // s.size], s[pick % s.size], 1 if n_orb <= 64 else 2)
    h, eri, ec = S.integrals(n_orb, 4, 9)
    O = oracle.System(h, eri, ec)
    c = np.zeros(n)
    used = np.random.default_rng(2).choice(n, 5, replace=False)
    c[used] = [0.7, -0.5, 0.3, -0.2, 0.1]
    B = G.Built(P, h, eri, ec, dets, 2, 2, mode=P.SHCI_ON_THE_FLY)
    got = P.shci_select(B.ctx.handle, G.dev(c), 2e-2).cpu().numpy().view(np.uint64)
    ref, best = O.select(dets, c, 2e-2 * (1 - BAND), with_best=True)
    assert _rows(ref[best >= 2e-2 * (1 + BAND)]) <= _rows(got) <= _rows(ref)
    order = [tuple(int(x) for x in r[::-1]) for r in got]
    assert order == sorted(order) and len(set(order)) == len(order) and len(order) > 100
    B.close()
