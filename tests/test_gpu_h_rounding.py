"""h symmetric to rounding only (the library takes up to 1e-12): an element H_ij
carries h_pq of the particle p in D_i and the hole q in D_j, whether V is large
enough to tabulate its single moves or not.

An element is a sum of at most 12 terms below 8: within 12 x 2^-53 x 96 = 1.3e-13
of its value; h_pq and h_qp differ by 9e-13 here."""
import numpy as np
import pytest

import oracle
import shci_synth as S
from tests import gpu_common as G

pytestmark = pytest.mark.gpu

TOL = 1.3e-13


def _integrals(n):
    h, eri, ec = S.integrals(n, 2 * n, 77)
    return h + np.triu(np.full((n, n), 9e-13), 1), eri, ec


@pytest.mark.parametrize("mode", ["SHCI_STORED", "SHCI_STORED_UPPER"])
@pytest.mark.parametrize("step", [1, 40])                 # 3,136 determinants, enough for tables, and 79
def test_stored_elements(mode, step):
    P = G.lib()
    h, eri, ec = _integrals(8)
    dets = np.ascontiguousarray(S.fci_dets(8, 3, 3)[::step])
    B = G.Built(P, h, eri, ec, dets, 3, 3, mode=getattr(P, mode))
    O = oracle.System(h, eri, ec)
    ii, jj, vv = B.pairs()
    want = O.hij_list(dets, ii, jj)
    assert np.max(np.abs(vv - want)) <= TOL
    if mode == "SHCI_STORED":                             # and the rows' lower parts
        for i in (1, ii.max(), dets.shape[0] - 1):
            cols, vals = (np.asarray(t) for t in B.row(i))
            want = O.hij_list(dets, np.full(cols.size, i), cols.astype(np.int64))
            assert np.max(np.abs(vals - want)) <= TOL
    B.close()


def test_products_on_the_fly():
    P = G.lib()
    h, eri, ec = _integrals(8)
    dets = S.fci_dets(8, 3, 3)
    B = G.Built(P, h, eri, ec, dets, 3, 3, mode=P.SHCI_ON_THE_FLY)
    O = oracle.System(h, eri, ec)
    for j in (0, 17, 3135):
        x = np.zeros((1, 3136))
        x[0, j] = 1.0
        y = B.sigma(x)[0]
        rows = np.flatnonzero(y)
        rows = rows[rows != j]
        want = O.hij_list(dets, rows, np.full(rows.size, j))
        assert np.max(np.abs(y[rows] - want)) <= TOL
    B.close()
