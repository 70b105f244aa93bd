"""The subspace eigensolver at its corners, through the Davidson solves that use
it: one to eight roots (subspaces up to 64 vectors and over several restarts),
starts whose new vectors have no coupling to the subspace (deflation), exactly
degenerate spectra, and a batch; eigenvalues against the oracle's dense matrix."""
import numpy as np
import pytest
import torch

import oracle
import shci_synth as S
from tests import gpu_common as G

pytestmark = pytest.mark.gpu


def _check(H, e, v, k):
    """e ascending eigenvalues of H, v orthonormal with small residuals."""
    w = np.linalg.eigvalsh(H)
    assert np.all(np.diff(e) > -1e-11)
    assert max(np.min(np.abs(w - x)) for x in e) < 1e-9
    assert np.max(np.abs(v @ v.T - np.eye(k))) < 1e-10
    assert np.max(np.linalg.norm(v @ H - e[:, None] * v, axis=1)) < 2e-6
    return w


@pytest.mark.parametrize("mode", ["SHCI_STORED", "SHCI_ON_THE_FLY"])
@pytest.mark.parametrize("k", [1, 2, 3, 5, 8])
def test_roots_over_restarts(k, mode):
    P = G.lib()
    h, eri, ec = S.integrals(9, 18, 321)
    dets = S.fci_dets(9, 3, 3)[::5]
    B = G.Built(P, h, eri, ec, dets, 3, 3, mode=getattr(P, mode))
    H = oracle.System(h, eri, ec).dense_h(dets)
    e, v, it = B.davidson(k)
    w = _check(H, e, v, k)
    assert abs(e[0] - w[0]) < 1e-9
    # a start that is already converged: the first subspace is diagonal
    e2, v2, it2 = B.davidson(k, guess=v)
    assert it2 <= 3 and np.max(np.abs(e2 - e)) < 1e-10
    _check(H, e2, v2, k)
    B.close()


@pytest.mark.parametrize("k", [1, 4])
def test_degenerate_spectrum(k):
    """No two-electron term: the spectrum is sums of orbital energies, with
    repeated orbital energies (poles that coincide, borders that vanish)."""
    P = G.lib()
    n = 8
    h, eri, ec = S.integrals(n, 4, 5)
    q = np.linalg.qr(np.random.default_rng(2).normal(size=(n, n)))[0]
    h = q @ np.diag([-2.0, -2.0, -1.0, -1.0, 0.5, 0.5, 1.0, 2.0]) @ q.T
    h = 0.5 * (h + h.T)
    eri = np.zeros_like(eri)
    dets = S.fci_dets(n, 3, 2)
    B = G.Built(P, h, eri, ec, dets, 3, 2)
    H = oracle.System(h, eri, ec).dense_h(dets)
    e, v, it = B.davidson(k)
    _check(H, e, v, k)
    B.close()


@pytest.mark.parametrize("k", [1, 4])
def test_batch_of_uneven_systems(k):
    """Vector slices of one block to several: sizes below, at and above them."""
    P = G.lib()
    systems, want = [], []
    for s, n in enumerate((5, 255, 256, 257, 1400)):
        h, eri, ec = S.integrals(9, 18, 400 + s)
        dets = np.ascontiguousarray(S.fci_dets(9, 3, 3)[:n])
        systems.append({"n_orb": 9, "n_alpha": 3, "n_beta": 3, "h": G.dev(h), "eri": G.dev(eri), "dets": G.dev(dets)})
        want.append(np.linalg.eigvalsh(oracle.System(h, eri, ec).dense_h(dets)))
    ctx = P.Context(0, torch.cuda.current_stream())
    b = P.shci_batch_create(ctx.handle, systems)
    e, it, cv, rc = P.shci_batch_davidson(ctx.handle, b, len(systems), k)
    assert cv.all()
    for s in range(len(systems)):
        assert max(np.min(np.abs(want[s] - x)) for x in e[s]) < 1e-9
    P.shci_batch_destroy(b)
    ctx.close()
