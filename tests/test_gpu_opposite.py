"""The opposite-spin pass (words of 32 alpha singles over tables of beta
strings) against the general path that scans the alpha singles' groups
(SHCI_OPP_SPIN=scan), where its tables and queues have edges: more than 32
alpha singles, beta strings over more than one table, strings of two words, no
alpha singles, one determinant; with and without tabulated single moves.

An opposite-spin element is one entry of the integrals with a sign, and the
singles are summed alike on both paths, so the stored H agrees bit for bit.
Products and gradients add the same terms in another order: with at most m
terms per sum the two differ by less than 2 m 2^-53 of the sum of the terms'
magnitudes, which is below 1e-12 of it for the m < 4500 of these spaces."""
import itertools

import numpy as np
import pytest

import oracle
import shci_synth as S
from tests import gpu_common as G
from tests.test_gpu_adjoint import gpu_gradient
from tests.test_gpu_extend import _extend

pytestmark = pytest.mark.gpu


def _strings(orbs, n_elec):
    return np.array([sum(1 << o for o in s) for s in itertools.combinations(orbs, n_elec)], dtype=object)


def _dets(alpha, beta, words):
    """Determinants of the paired string lists (Python integers)."""
    cols = []
    for s in (alpha, beta):
        cols += [np.array([(int(v) >> (64 * w)) & (2 ** 64 - 1) for v in s], dtype=np.uint64) for w in range(words)]
    return np.ascontiguousarray(np.stack(cols, axis=1))


def _space(name):
    rng = np.random.default_rng(5)
    if name == "fci":                                     # 36 alpha singles a string: 32 and 4
        n_orb, na, nb = 20, 2, 2
        return n_orb, na, nb, S.fci_dets(n_orb, na, nb)[::3].copy()
    if name == "two_beta_tables":                         # 35,960 beta strings > 24,576
        n_orb, na, nb = 32, 1, 4
        b = _strings(range(n_orb), nb)
        b = np.concatenate([rng.permutation(b), rng.permutation(b)[:9000]])
        a = np.array([1 << int(k) for k in np.concatenate([rng.integers(0, 3, 35960), np.full(9000, 3)])], dtype=object)
        return n_orb, na, nb, _dets(a, b, 1)
    if name == "two_words":                               # strings across the word boundary, too many to tabulate
        n_orb, na, nb = 70, 3, 3
        s = _strings(range(58, 70), 3)
        pick = rng.choice(s.size * s.size, 3001, replace=False)
        return n_orb, na, nb, _dets(s[pick // s.size], s[pick % s.size], 2)
    n_orb, na, nb = 12, 3, 3
    if name == "no_alpha_singles":                        # alpha strings that differ by doubles
        b = _strings(range(n_orb), nb)
        return n_orb, na, nb, _dets(np.repeat(np.array([0b111, 0b11001], dtype=object), b.size), np.tile(b, 2), 1)
    return n_orb, na, nb, _dets([0b111], [0b111], 1)      # one determinant


def _paths(monkeypatch, P, sys_, mode):
    n_orb, na, nb, dets, h, eri, ec = sys_
    out = []
    for opp in ("scan", "auto"):
        monkeypatch.setenv("SHCI_OPP_SPIN", opp)
        out.append(G.Built(P, h, eri, ec, dets, na, nb, mode=mode))
    return out


def _system(name):
    n_orb, na, nb, dets = _space(name)
    h, eri, ec = S.integrals(n_orb, 6, 31)
    return n_orb, na, nb, dets, h, eri, ec


SPACES = ["fci", "two_beta_tables", "two_words", "no_alpha_singles", "one"]


@pytest.mark.parametrize("name", SPACES)
def test_stored_matrix_is_the_same(monkeypatch, name):
    P = G.lib()
    sys_ = _system(name)
    dets, (h, eri, ec) = sys_[3], sys_[4:]
    A, B = _paths(monkeypatch, P, sys_, P.SHCI_STORED)
    assert A.nnz == B.nnz
    for x, y in zip(A.pairs(), B.pairs()):
        assert np.array_equal(x, y)
    O = oracle.System(h, eri, ec)
    n = dets.shape[0]
    for i in sorted({0, n // 2, n - 1}) if n > 1 else []:       # an empty row is refused
        for x, y in zip(A.row(i), B.row(i)):
            assert np.array_equal(x, y)
        cols, vals = O.row(dets, i)
        gc, gv = (np.asarray(t) for t in B.row(i))
        keep = np.asarray(cols) != i
        o, g = np.argsort(np.asarray(cols)[keep]), np.argsort(gc)
        assert np.array_equal(np.asarray(cols)[keep][o], gc[g])
        assert np.all(np.abs(np.asarray(vals)[keep][o] - gv[g]) < 1e-12)
    A.close()
    B.close()


@pytest.mark.parametrize("name", SPACES)
@pytest.mark.parametrize("upper", [False, True])
def test_products_and_gradient(monkeypatch, name, upper):
    """On the fly, or from the upper triangle."""
    P = G.lib()
    sys_ = _system(name)
    A, B = _paths(monkeypatch, P, sys_, P.SHCI_STORED_UPPER if upper else P.SHCI_ON_THE_FLY)
    assert A.nnz == B.nnz
    monkeypatch.setenv("SHCI_OPP_SPIN", "scan")
    F = G.Built(P, *sys_[4:], sys_[3], sys_[1], sys_[2])
    for k in (1, 2, 3, 5, 8):
        x = S.random_vectors(A.n, k, 3 + k)
        # sum_j |H_ij x_j| <= |H|_row max|x|; |H| by rows from the stored matrix
        ya, yb, yf = A.sigma(x), B.sigma(x), F.sigma(x)
        if k == 1:
            ii, jj, vv = F.pairs()
            rows = np.abs(F.diag())
            np.add.at(rows, ii, np.abs(vv))
            np.add.at(rows, jj, np.abs(vv))
        bound = 1e-12 * rows * np.max(np.abs(x))
        assert np.all(np.abs(ya - yb) <= bound)
        assert np.all(np.abs(yf - yb) <= bound)
    c = S.random_vectors(A.n, 1, 9)[0]
    c /= np.linalg.norm(c)
    per_row = np.bincount(np.concatenate([ii, jj]), minlength=1).max(initial=1)
    for x, y in zip(gpu_gradient(P, A, c), gpu_gradient(P, B, c)):
        # the terms of an entry: at most 4 |c_i c_j| per pair, sum over pairs <= per_row / 2
        assert np.all(np.abs(x - y) <= 1e-12 * 4.0 * per_row)
    for t in (A, B, F):
        t.close()


@pytest.mark.parametrize("name", ["fci", "two_beta_tables", "two_words"])
def test_grown_space_is_the_same(monkeypatch, name):
    """Old rows take the new pairs only, new rows all of theirs."""
    P = G.lib()
    sys_ = _system(name)
    dets = sys_[3][np.random.default_rng(2).permutation(sys_[3].shape[0])]
    n_old = dets.shape[0] - dets.shape[0] // 17
    A, B = _paths(monkeypatch, P, sys_[:3] + (dets[:n_old],) + sys_[4:], P.SHCI_STORED)
    for opp, T in (("scan", A), ("auto", B)):
        monkeypatch.setenv("SHCI_OPP_SPIN", opp)
        _extend(P, T, dets[n_old:])
    assert A.nnz == B.nnz
    for x, y in zip(A.pairs(), B.pairs()):
        assert np.array_equal(x, y)
    A.close()
    B.close()
