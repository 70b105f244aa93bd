"""Products over the upper triangle with a row per warp (small spaces) and with
groups of rows, on both sides of the sizes where the form changes, against the
product over both triangles: the same m terms per row in another order differ by
less than 2 m 2^-53 of the sum of their magnitudes, below 2e-12 of it for the
at most 7,875 excitations of a determinant here."""
import numpy as np
import pytest
import torch

import shci_synth as S
from tests import gpu_common as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("side", [-1, 0, 1])
def test_both_sides_of_the_change_of_form(k, side):
    P = G.lib()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    edge = sms * {1: 128 * 4, 2: 64 * 4, 3: 64 * 2, 4: 64 * 2}.get(k, 64)
    cfg, h, eri, ec, dets = G.system("sel_20o_5a5b_1m", edge + side)
    x = S.random_vectors(edge + side, k, 3 + k)
    U = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta, mode=P.SHCI_STORED_UPPER)
    got = U.sigma(x)
    U.close()
    F = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta)
    want = F.sigma(x)
    ii, jj, vv = F.pairs()
    a = np.abs(x)
    scale = np.abs(F.diag()) * a
    F.close()
    for q in range(k):
        scale[q] += np.bincount(ii, np.abs(vv) * a[q, jj], edge + side)
        scale[q] += np.bincount(jj, np.abs(vv) * a[q, ii], edge + side)
    assert np.all(np.abs(got - want) <= 2e-12 * scale)
