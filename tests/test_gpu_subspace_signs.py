"""The subspace eigensolver in solves (the lowest roots) and by itself: bordered
matrices whose leading block is decomposed first, then the whole vector by vector
with signs, against the Jacobi iteration from the same start and against numpy.

Both end with off-diagonal elements below 1e-14 of the diagonal's magnitudes, so
eigenvalues and residuals are within 64 x 2e-14 |G| = 1.3e-12 |G| (2e-12 here); the
vectors are products of at most 2,000 rotations or 64 vector updates, each
orthogonal to a few 1e-16: 1e-12.  Eigenvectors a gap g apart are defined to about
1e-15 |G| / g, at least 1e-5 here, so that corresponding ones overlap by 1 and not
-1 when their signs agree."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle
import shci_synth as S
from tests import gpu_common as G
from paper_1809_04600_gb300 import build_lib

pytestmark = pytest.mark.gpu

LD = 64


@pytest.fixture(scope="module")
def solver(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("subspace") / "subspace_eig.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "subspace_eig.cu")
    cmd = [build_lib._nvcc(), *build_lib.ARCH, *build_lib.NVCC_FLAGS, "-I", build_lib.CSRC, "-I", build_lib.INCLUDE,
           "-shared", "-o", so, src, "-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(so)

    def solve(A, m_prev, how):
        m = A.shape[0]
        a = np.zeros((LD, LD))
        a[:m, :m] = A
        e, v, did = np.zeros(LD), np.zeros((LD, LD)), ctypes.c_int(0)
        p = lambda x: x.ctypes.data_as(ctypes.c_void_p)
        assert lib.subspace_eig_test(p(a), m, m_prev, how, p(e), p(v), ctypes.byref(did)) == 0
        return e[:m], v[:m, :m], did.value

    return solve


def _check(A, e, v):
    norm = np.abs(np.linalg.eigvalsh(A)).max()
    assert np.max(np.abs(e - np.linalg.eigvalsh(A))) <= 2e-12 * norm
    assert np.max(np.linalg.norm(v @ A - e[:, None] * v, axis=1)) <= 2e-12 * norm
    assert np.max(np.abs(v @ v.T - np.eye(e.size))) <= 1e-12


def _symmetric(m, seed):
    g = np.random.default_rng(seed).normal(size=(m, m))
    return g + g.T


SIZES = [(1, 2), (2, 3), (7, 8), (31, 32), (32, 33), (33, 34), (62, 63), (63, 64), (1, 5), (24, 32), (56, 64)]


@pytest.mark.parametrize("m_prev,m", SIZES)
@pytest.mark.parametrize("kind", ["dense", "shifted", "weak", "uncoupled"])
def test_appended_vectors(solver, m_prev, m, kind):
    """Every append is taken, and the signs are the Jacobi iteration's."""
    A = _symmetric(m, 100 * m + m_prev)
    if kind == "shifted":                                 # as Ritz values far from zero are
        A += -75.0 * np.eye(m) + np.diag(np.arange(m))
    elif kind == "weak":                                  # a nearly converged subspace
        A[:m_prev, m_prev:] *= 1e-7
        A[m_prev:, :m_prev] *= 1e-7
    elif kind == "uncoupled":                             # a border without elements
        A[:m - 1, m - 1] = A[m - 1, :m - 1] = 0.0
    _, _, taken = solver(A, m_prev, 2)
    assert taken == m - m_prev
    e, v, _ = solver(A, m_prev, 0)
    ej, vj, _ = solver(A, m_prev, 1)
    _check(A, e, v)
    _check(A, ej, vj)
    assert np.all((v * vj).sum(1) > 0.9)


def _close(m_prev, gap, seed):
    """A leading block with pairs of eigenvalues `gap` apart, coupled to one more vector."""
    rng = np.random.default_rng(seed)
    d = np.sort(rng.uniform(-3.0, 3.0, m_prev))
    d[1::2] = d[0:2 * (m_prev // 2):2] + gap
    A = np.diag(np.append(d, 0.3))
    A[:m_prev, m_prev] = A[m_prev, :m_prev] = rng.normal(size=m_prev)
    return A


@pytest.mark.parametrize("m_prev", [2, 9, 40])
@pytest.mark.parametrize("gap", [1e-6, 1e-8, 1e-10])
def test_eigenvalues_that_fp32_cannot_tell_apart(solver, m_prev, gap):
    """Taken or refused, the signs are the Jacobi iteration's."""
    for seed in range(8):
        A = _close(m_prev, gap, seed)
        e, v, _ = solver(A, m_prev, 0)
        ej, vj, _ = solver(A, m_prev, 1)
        _check(A, e, v)
        assert np.all((v * vj).sum(1) > 0.9)


@pytest.mark.parametrize("m_prev", [4, 9, 40])
@pytest.mark.parametrize("late", [False, True])
def test_refused_appends(solver, m_prev, late):
    """Poles closer than 1e-12 that are both coupled: refused, at once or after another
    vector was appended; the result is the Jacobi iteration's, bit for bit."""
    A = _close(m_prev, 0.0, 3)
    if late:                                              # a first vector that leaves one such pair alone
        first = np.zeros((m_prev + 2, m_prev + 2))
        first[:m_prev, :m_prev] = A[:m_prev, :m_prev]
        d = np.diag(first).copy()
        rest = np.arange(2, m_prev)
        d[rest] = np.linspace(-2.0, 2.5, rest.size)
        np.fill_diagonal(first, d)
        first[rest, m_prev] = first[m_prev, rest] = -A[rest, m_prev]
        first[m_prev, m_prev] = 0.7
        first[:m_prev, m_prev + 1] = first[m_prev + 1, :m_prev] = A[:m_prev, m_prev]
        first[m_prev + 1, m_prev + 1] = -0.2
        A = first
    assert solver(A, m_prev, 2)[2] == (1 if late else 0)
    e, v, _ = solver(A, m_prev, 0)
    ej, vj, _ = solver(A, m_prev, 1)
    _check(A, e, v)
    assert np.array_equal(e, ej) and np.array_equal(v, vj)


def _space(step):
    dets = np.ascontiguousarray(S.fci_dets(9, 3, 3)[::step])
    h, eri, ec = S.integrals(9, 18, 321)
    return h, eri, ec, dets, np.linalg.eigvalsh(oracle.System(h, eri, ec).dense_h(dets))


@pytest.mark.parametrize("k", [2, 5, 8])
def test_the_lowest_roots_of_a_solve(k):
    """All k of them (to the solves' 1e-9), over restarts: k = 8 fills 64 vectors in at most 8 steps."""
    P = G.lib()
    h, eri, ec, dets, want = _space(5)
    B = G.Built(P, h, eri, ec, dets, 3, 3)
    e, v, it = B.davidson(k)
    assert np.max(np.abs(e - want[:k])) < 1e-9
    assert k < 8 or it > 8
    B.close()


@pytest.mark.parametrize("k", [1, 4])
def test_the_lowest_root_of_each_system_of_a_batch(k):
    P = G.lib()
    systems, want = [], []
    for step in (3, 7, 11):
        h, eri, ec, dets, w = _space(step)
        systems.append({"n_orb": 9, "n_alpha": 3, "n_beta": 3, "e_core": ec, "h": G.dev(h), "eri": G.dev(eri),
                        "dets": G.dev(dets)})
        want.append(w[0])
    ctx = P.Context(0, torch.cuda.current_stream())
    b = P.shci_batch_create(ctx.handle, systems)
    e, it, cv, rc = P.shci_batch_davidson(ctx.handle, b, len(systems), k)
    assert cv.all() and np.max(np.abs(e[:, 0] - want)) < 1e-9
    P.shci_batch_destroy(b)
    ctx.close()
