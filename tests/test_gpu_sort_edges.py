"""The radix sort and scan at the edges of their tiles, through the calls that
use them: the helper lists (and so the pairs and the product) of spaces whose
sizes straddle a tile or the scan's two forms, and the selection's and
second-order energy's sort keys in one word, two words and four."""
import numpy as np
import pytest
import torch

import oracle
import shci_synth as S
from tests import gpu_common as G

pytestmark = pytest.mark.gpu

TILE = 2048                # radix sort (one-word keys) and scan tile


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, TILE - 1, TILE, TILE + 1, 2 * TILE + 1])
def test_pairs_at_tile_edges(n):
    P = G.lib()
    cfg, h, eri, ec, dets = G.system("sel_24o_6a6b_1m", n)
    B = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta)
    ii, jj = oracle.pairs_allpairs(dets)
    gi, gj, gv = B.pairs()
    assert np.array_equal(gi, ii) and np.array_equal(gj, jj)
    if ii.size:
        assert np.max(np.abs(gv - oracle.System(h, eri, ec).hij_list(dets, ii, jj))) < 1e-12
    B.close()


@pytest.mark.parametrize("n", [512 * TILE - 1, 512 * TILE + 1])
def test_scan_both_forms(n):
    """Row offsets of n rows: up to 512 tiles each block sums the totals before
    it, above that they are scanned first.  Rows sampled against the oracle."""
    P = G.lib()
    cfg = S.config("sel_24o_6a6b_1m_standin")
    h, eri, ec = S.integrals(cfg.n_orb, cfg.rank, cfg.seed)
    dets = S.selected_dets(cfg.n_orb, cfg.n_alpha, cfg.n_beta, np.diag(h), n, cfg.seed)
    B = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta, mode=P.SHCI_ON_THE_FLY)
    x = np.zeros((1, n))
    rows = [0, 1, n // 2, n - 1]
    O = oracle.System(h, eri, ec)
    x[0, rows] = 1.0
    y = B.sigma(x)[0]
    want = np.zeros(n)
    d = O.hdiag(dets[rows])
    for t, i in enumerate(rows):
        cols, vals = O.row(dets, i)
        want[cols] += vals                                 # H is symmetric: column i is row i
        want[i] += d[t]
    assert np.max(np.abs(y - want)) < 1e-12 * max(1.0, np.max(np.abs(want)))
    B.close()


BAND = 1e-12               # products this close to a threshold may fall on either side of it


def _rows(a):
    return {tuple(int(x) for x in r) for r in np.asarray(a).view(np.uint64)}


@pytest.mark.parametrize("tabulated", [False, True])
@pytest.mark.parametrize("n_orb,na,nb", [(32, 2, 2), (33, 2, 2), (64, 2, 2), (65, 2, 2)])
def test_keys_of_every_width(n_orb, na, nb, tabulated):
    """One sort word (2 n_orb <= 64), two and four: the selected set with its
    order, the second-order energy and one stochastic sample against the
    oracle's brute force.  Single moves are evaluated for a small V and read
    from the per-string tables for a large one of few strings (its coefficients
    zero but for a few determinants, so that the oracle stays cheap)."""
    P = G.lib()
    h, eri, ec = S.integrals(n_orb, 6, 77 + n_orb)
    O = oracle.System(h, eri, ec)
    dets = S.fci_dets(17, na, nb)                          # 136^2 determinants of the lowest 17 orbitals
    if S.n_words(n_orb) == 2:
        dets = np.ascontiguousarray(np.stack([dets[:, 0], 0 * dets[:, 0], dets[:, 1], 0 * dets[:, 0]], axis=1))
    rng = np.random.default_rng(n_orb)
    used = np.sort(rng.choice(dets.shape[0], 8, replace=False))
    if not tabulated:
        dets, used = np.ascontiguousarray(dets[used]), np.arange(8)
    c = np.zeros(dets.shape[0])
    c[used] = rng.normal(size=8)
    B = G.Built(P, h, eri, ec, dets, na, nb, mode=P.SHCI_ON_THE_FLY)
    cd = G.dev(c)
    got = P.shci_select(B.ctx.handle, cd, 2e-2).cpu().numpy().view(np.uint64)
    ref, best = O.select(dets, c, 2e-2 * (1 - BAND), with_best=True)
    assert _rows(ref[best >= 2e-2 * (1 + BAND)]) <= _rows(got) <= _rows(ref)
    order = [tuple(int(x) for x in r[::-1]) for r in got]
    assert order == sorted(order) and len(set(order)) == len(order) and len(order) > 100
    e_var = float(O.hdiag(dets[used]).min()) - 1.0
    e2, npert = P.shci_pt2(B.ctx.handle, cd, e_var, 1e-2)
    refs = [O.pt2(dets, c, e_var, 1e-2 * f) for f in (1 - BAND, 1 + BAND)]
    assert any(abs(e2 - r[0]) <= 1e-10 * abs(r[0]) and npert == r[1] for r in refs), (e2, npert, refs)
    draws = used[rng.integers(0, 8, size=(1, 40))].astype(np.int64)
    v = P.shci_pt2_samples(B.ctx.handle, cd, e_var, 1e-2, 3e-2, G.dev(draws))[0]
    refs = [O.pt2_sample(dets, c, e_var, 1e-2 * f, 3e-2 * f, draws[0]) for f in (1 - BAND, 1 + BAND)]
    assert any(all(abs(v[j] - r[j]) <= 1e-10 * max(1e-8, abs(r[j])) for j in (0, 1)) for r in refs), (v, refs)
    with pytest.raises(P.ShciError):                       # a draw with a zero coefficient, or outside V
        P.shci_pt2_samples(B.ctx.handle, cd, e_var, 1e-2, 3e-2, G.dev(np.full((1, 4), dets.shape[0], np.int64)))
    B.close()


def _vose(q):
    """Vose's table, one column at a time."""
    n = q.size
    q, alias = q.copy(), np.arange(n)
    small, large = [i for i in range(n) if q[i] < 1.0], [i for i in range(n) if q[i] >= 1.0]
    prob = q.copy()
    while small and large:
        l, g = small.pop(), large.pop()
        prob[l], alias[l] = q[l], g
        q[g] = (q[g] + q[l]) - 1.0
        (small if q[g] < 1.0 else large).append(g)
    for i in small + large:
        prob[i] = 1.0
    return prob, alias


@pytest.mark.parametrize("kind", ["decaying", "two_values", "one_large", "single"])
def test_alias_draws_are_voses(kind):
    """The draws are those of Vose's table built column by column."""
    P = G.lib()
    cfg, h, eri, ec, dets = G.system("sel_24o_6a6b_1m", 1 if kind == "single" else 1500)
    n = dets.shape[0]
    rng = np.random.default_rng(9)
    c = {"decaying": (np.arange(n) + 3.0) ** -0.9 * rng.normal(size=n),
         "two_values": np.where(np.arange(n) % 2 == 0, 0.3, -0.1),
         "one_large": np.where(np.arange(n) == 0, 0.999, 1e-5),
         "single": np.ones(n)}[kind]
    B = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta, mode=P.SHCI_ON_THE_FLY)
    m = 20000
    got = P.shci_alias_draw(B.ctx.handle, G.dev(c), m, 77).cpu().numpy()
    # the library's sum of |c| (its order is its own) is within 1e-13 of this one; a
    # draw can differ only where a probability moves past a 32-bit uniform number
    prob, alias = _vose(np.abs(c) * (n / np.sum(np.abs(c))))
    z = (np.uint64(77) + (np.arange(1, m + 1, dtype=np.uint64)) * np.uint64(0x9E3779B97F4A7C15))
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z ^= z >> np.uint64(31)
    col = ((z >> np.uint64(32)) * np.uint64(n) >> np.uint64(32)).astype(np.int64)
    u = (z & np.uint64(0xFFFFFFFF)).astype(np.float64) / 2.0 ** 32
    assert np.array_equal(got, np.where(u < prob[col], col, alias[col]))
    B.close()
