"""The opposite-spin pass where its tables and its lookups in the occupancy
bitmap meet: spaces whose alpha singles are looked up one by one (few of them,
beside many beta strings), sparse groups, spaces over several tables, spaces
that mix both, singles without members, growth by one determinant, by a few and
by a third; against the path that scans the alpha singles'
groups (SHCI_OPP_SPIN=scan), bit for bit.  Products and gradients add the same
terms in another order: they differ by less than 2 m 2^-53 of the sum of the
terms' magnitudes, below 1e-12 of it for the m < 4500 terms of a row here."""
import numpy as np
import pytest

import shci_synth as S
from tests import gpu_common as G
from tests.test_gpu_adjoint import gpu_gradient
from tests.test_gpu_extend import _extend
from tests.test_gpu_opposite import _dets, _strings

pytestmark = pytest.mark.gpu


def _space(name):
    rng = np.random.default_rng(7)
    if name == "sparse":                                  # 14,950 strings a spin, some 1.3 members a group
        a = _strings(range(26), 4)
        pick = rng.choice(a.size * a.size, 20_011, replace=False)
        return 26, 4, 4, _dets(a[pick // a.size], a[pick % a.size], 1)
    if name == "few_alpha":                               # 2 alpha singles, 35,960 beta strings
        b = _strings(range(32), 4)
        pick = rng.choice(3 * b.size, 60_013, replace=False)
        return 32, 1, 4, _dets(np.array([1, 2, 4], dtype=object)[pick // b.size], b[pick % b.size], 1)
    if name == "tables":
        # one alpha string with all 35,960 beta strings, the 31 others with 100: two tables for the
        # large group's items of 16 rows, lookups for the small groups' (the rule in opposite.cuh)
        b = _strings(range(32), 4)
        rest = np.concatenate([rng.permutation(b)[:100] for _ in range(31)])
        a = np.array([1 << k for k in np.concatenate([np.zeros(b.size, int), np.repeat(np.arange(1, 32), 100)])],
                     dtype=object)
        return 32, 1, 4, _dets(a, np.concatenate([b, rest]), 1)
    n_orb = 70                                            # "words": two-word strings, sparse
    s = _strings(range(54, 70), 3)
    pick = rng.choice(s.size * s.size, 3001, replace=False)
    return n_orb, 3, 3, _dets(s[pick // s.size], s[pick % s.size], 2)


SPACES = ["sparse", "few_alpha", "tables", "words"]


def _both(monkeypatch, P, name, mode, head=None):
    n_orb, na, nb, dets = _space(name)
    h, eri, ec = S.integrals(n_orb, 5, 41)
    out = []
    for opp in ("scan", "auto"):
        monkeypatch.setenv("SHCI_OPP_SPIN", opp)
        out.append(G.Built(P, h, eri, ec, dets if head is None else dets[:head], na, nb, mode=mode))
    return dets, out


def _same_pairs(A, B):
    assert A.nnz == B.nnz
    for x, y in zip(A.pairs(), B.pairs()):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("name", SPACES)
@pytest.mark.parametrize("upper", [False, True])
def test_stored_matrix_is_the_same(monkeypatch, name, upper):
    P = G.lib()
    dets, (A, B) = _both(monkeypatch, P, name, P.SHCI_STORED_UPPER if upper else P.SHCI_STORED)
    _same_pairs(A, B)
    if not upper:
        n = dets.shape[0]
        for i in (0, n // 3, n - 1):
            for x, y in zip(A.row(i), B.row(i)):
                assert np.array_equal(x, y)
    A.close()
    B.close()


@pytest.mark.parametrize("name", SPACES)
def test_products_and_gradient(monkeypatch, name):
    P = G.lib()
    dets, (A, B) = _both(monkeypatch, P, name, P.SHCI_ON_THE_FLY)
    assert A.nnz == B.nnz
    monkeypatch.setenv("SHCI_OPP_SPIN", "scan")
    F = G.Built(P, A.h, A.eri, A.e_core, dets, A.n_alpha, A.n_beta)
    ii, jj, vv = F.pairs()
    rows = np.abs(F.diag())
    np.add.at(rows, ii, np.abs(vv))
    np.add.at(rows, jj, np.abs(vv))
    for k in (1, 2, 7):
        x = S.random_vectors(A.n, k, 3 + k)
        bound = 1e-12 * rows * np.max(np.abs(x))
        want = F.sigma(x)
        assert np.all(np.abs(A.sigma(x) - want) <= bound)
        assert np.all(np.abs(B.sigma(x) - want) <= bound)
    c = S.random_vectors(A.n, 1, 9)[0]
    c /= np.linalg.norm(c)
    per_row = np.bincount(np.concatenate([ii, jj]), minlength=1).max(initial=1)
    for x, y in zip(gpu_gradient(P, A, c), gpu_gradient(P, B, c)):
        assert np.all(np.abs(x - y) <= 1e-12 * 4.0 * per_row)
    for t in (A, B, F):
        t.close()


@pytest.mark.parametrize("name", SPACES)
@pytest.mark.parametrize("new", ["one", "few", "third"])
@pytest.mark.parametrize("upper", [False, True])
def test_grown_space_is_the_same(monkeypatch, name, new, upper):
    P = G.lib()
    n = _space(name)[3].shape[0]
    head = n - {"one": 1, "few": 23, "third": n // 3}[new]
    dets, (A, B) = _both(monkeypatch, P, name, P.SHCI_STORED_UPPER if upper else P.SHCI_STORED, head)
    for opp, T in (("scan", A), ("auto", B)):
        monkeypatch.setenv("SHCI_OPP_SPIN", opp)
        _extend(P, T, dets[head:])
    _same_pairs(A, B)
    A.close()
    B.close()
