"""Performance cases: the work this library does for its users, each through
the calls of ``paper_1809_04600_gb300.binding``.

A case is a plain dict with a ``kind`` (which call or sequence of calls is one
pass), a ``space`` (where its determinants come from) and sizes:

* ``sigma``    one product H c of the user's own eigen-solver, over a stored H
  (both triangles, or the upper one) or on the fly;
* ``solve``    integrals, connectivity and the lowest roots: a whole
  variational calculation on a given space;
* ``gradient`` dE/dh and dE/d(pq|rs) of a root (a geometry or orbital step);
* ``grow``     connectivity of a space, then of the space grown by the next
  selection, and the first product over it;
* ``select``   the next heat-bath selection;
* ``pt2``      the deterministic second-order energy;
* ``pt2_sampled`` the semistochastic one;
* ``batch``    many small systems solved in one launch.

Spaces are the heat-bath-selected ones stored with the tests (any prefix is an
earlier stage of the selection), the 76-orbital band shape, full-CI spaces of a
few orbitals, and the uneven systems of the batched workload.  They are fixed;
the integrals (another geometry of the same molecule) and the coefficients are
drawn from the seed.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

import paper_1809_04600_gb300 as P
import shci_synth as S

SPACES = {"24o": "sel_24o_6a6b_1m", "20o": "sel_20o_5a5b_1m", "76o": "sel_76o_14a14b_50m"}
MODES = {"stored": P.SHCI_STORED, "upper": P.SHCI_STORED_UPPER, "fly": P.SHCI_ON_THE_FLY}
MAX_DETS = {"24o": 1_000_000, "20o": 1_000_000, "76o": 400_003}
PRODUCTS = 40                # products of a solve counted as unavoidable by work()
EXACT_PAIRS = 4.5e10         # determinant pairs that exact() goes through at most


def listed():
    return [
        # an early selection stage, where the call's latency is the cost
        {"name": "sigma_small", "kind": "sigma", "space": "24o", "n": 2053, "k": 1, "mode": "stored"},
        # the stored product at the size the library is built for, two roots
        {"name": "sigma_stored", "kind": "sigma", "space": "24o", "n": 1_000_000, "k": 2, "mode": "stored"},
        # half the memory: the upper triangle, four roots, a ragged size
        {"name": "sigma_upper", "kind": "sigma", "space": "24o", "n": 200_003, "k": 4, "mode": "upper"},
        # two-word strings, where H is not stored
        {"name": "sigma_fly", "kind": "sigma", "space": "76o", "n": 400_003, "k": 1, "mode": "fly"},
        # a full-CI calculation (44,100 determinants, one root)
        {"name": "solve_fci", "kind": "solve", "space": "fci", "n_orb": 10, "na": 4, "nb": 4, "k": 1},
        # the benchmark's calculation: two roots of a heat-bath space
        {"name": "solve_selected", "kind": "solve", "space": "24o", "n": 1_000_000, "k": 2},
        # the adjoint of an energy
        {"name": "gradient", "kind": "gradient", "space": "20o", "n": 200_003},
        # a late selection step: 5 % new determinants
        {"name": "grow", "kind": "grow", "space": "24o", "n": 1_000_000, "new": 50_000},
        # the selection that follows a solve for one root
        {"name": "select", "kind": "select", "space": "24o", "n": 200_003, "k": 1, "eps1": 1e-4},
        # the perturbative stage, deterministic
        {"name": "pt2", "kind": "pt2", "space": "24o", "n": 200_003, "eps2": 1e-5},
        # and semistochastic, at a tighter screen
        {"name": "pt2_sampled", "kind": "pt2_sampled", "space": "24o", "n": 100_003, "eps2": 1e-6, "eps2_d": 1e-4,
         "n_d": 10_000, "samples": 4},
        # a screening over uneven small systems, four roots of each
        {"name": "batch", "kind": "batch", "first": 0, "count": 8, "n_max": 40_000, "k": 4},
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["sigma", "sigma", "sigma", "solve", "gradient", "grow", "select", "pt2", "pt2_sampled",
                       "batch"])
    if kind == "batch":
        return {"kind": kind, "first": rng.randrange(64), "count": rng.randint(2, 8),
                "n_max": _log_int(rng, 12_000, 40_000), "k": rng.randint(1, 4)}
    if kind == "solve" and rng.random() < 0.4:
        n_orb = rng.randint(7, 10)
        return {"kind": kind, "space": "fci", "n_orb": n_orb, "na": rng.randint(2, 4), "nb": rng.randint(2, 4),
                "k": rng.randint(1, 3)}
    space = rng.choice(["24o", "20o", "76o"])
    if kind == "sigma":
        mode = rng.choice(["stored", "upper", "fly"])
        return {"kind": kind, "space": space, "n": _log_int(rng, 1_000, MAX_DETS[space]), "k": rng.randint(1, 8),
                "mode": mode}
    if kind == "solve":
        return {"kind": kind, "space": space, "n": _log_int(rng, 2_000, MAX_DETS[space] // 2), "k": rng.randint(1, 2)}
    if kind == "gradient":
        return {"kind": kind, "space": space, "n": _log_int(rng, 1_000, MAX_DETS[space])}
    if kind == "grow":
        n = _log_int(rng, 2_000, MAX_DETS[space])
        return {"kind": kind, "space": space, "n": n, "new": max(1, int(n * rng.uniform(0.01, 0.19)))}
    if kind == "select":
        large = space == "76o"
        return {"kind": kind, "space": space, "n": _log_int(rng, 1_000, 50_000 if large else 400_003),
                "k": rng.randint(1, 3), "eps1": 10.0 ** (rng.uniform(-4.0, -3.0) + (1.0 if large else 0.0))}
    space = rng.choice(["24o", "20o"])
    if kind == "pt2":
        return {"kind": kind, "space": space, "n": _log_int(rng, 1_000, 200_003), "eps2": 10.0 ** rng.uniform(-5.0, -3.5)}
    eps2 = 10.0 ** rng.uniform(-6.0, -5.0)
    return {"kind": kind, "space": space, "n": _log_int(rng, 2_000, 100_003), "eps2": eps2,
            "eps2_d": eps2 * rng.uniform(20.0, 100.0), "n_d": _log_int(rng, 500, 10_000), "samples": rng.randint(2, 4)}


# ---------------------------------------------------------------- inputs

class System:
    """A system's fixed part: shape, reference integrals and determinants."""

    def __init__(self, n_orb, na, nb, rank, band, h, eri, dets):
        self.n_orb, self.na, self.nb, self.rank, self.band = n_orb, na, nb, rank, band
        self.h, self.eri, self.dets = h, eri, dets

    def integrals(self, seed):
        """Another geometry: nine tenths of the reference integrals and one tenth of a draw from the seed."""
        h, eri, _ = S.integrals(self.n_orb, self.rank, seed, self.band, self.na)
        return 0.9 * self.h + 0.1 * h, 0.9 * self.eri + 0.1 * eri


@functools.lru_cache(maxsize=16)
def _space(space, n):
    cfg = S.config(SPACES[space])
    h, eri, _ = S.integrals(cfg.n_orb, cfg.rank, cfg.seed, cfg.band, cfg.n_alpha)
    if cfg.space == "heat-bath":
        dets = S.load_selected_space(cfg.name, check_hash=False, n_det=n)
    else:
        hw, pw, ml = cfg.window
        dets = S.selected_dets(cfg.n_orb, cfg.n_alpha, cfg.n_beta, np.diag(h), n, cfg.seed, hole_window=hw,
                               particle_window=pw, max_level=ml)
    return System(cfg.n_orb, cfg.n_alpha, cfg.n_beta, cfg.rank, cfg.band, h, eri, dets)


@functools.lru_cache(maxsize=16)
def _fci(n_orb, na, nb):
    h, eri, _ = S.integrals(n_orb, 2 * n_orb, 1001)
    return System(n_orb, na, nb, 2 * n_orb, 0, h, eri, S.fci_dets(n_orb, na, nb))


@functools.lru_cache(maxsize=8)
def _batch(first, count, n_max):
    out = []
    for cfg in S.batch_configs(count, 5000 + first, n_max, 10_000):
        h, eri, _, dets = S.make_system(cfg)
        out.append(System(cfg.n_orb, cfg.n_alpha, cfg.n_beta, cfg.rank, 0, h, eri, dets))
    return out


def _system(case):
    if case["space"] == "fci":
        return _fci(case["n_orb"], case["na"], case["nb"])
    return _space(case["space"], case["n"])


def _gpu(a):
    a = np.ascontiguousarray(a)
    return torch.from_numpy(a.view(np.int64) if a.dtype == np.uint64 else a.copy()).cuda()


def _coefficients(n, k, seed):
    """[k, n] unit vectors that decay along the generation order as a root's coefficients do, with random signs."""
    rng = np.random.default_rng(seed)
    c = (np.arange(n) + 10.0) ** -0.8 * np.exp(0.7 * rng.normal(size=(k, n))) * rng.choice([-1.0, 1.0], size=(k, n))
    return c / np.linalg.norm(c, axis=1, keepdims=True)


def _reference_energy(s, h, eri):
    """Energy of the aufbau determinant: the scale of the variational energy handed to the perturbative calls."""
    slot = lambda p, q, r, t: _pair(_pair(p, q), _pair(r, t))
    e = 2.0 * h[range(s.na), range(s.na)].sum() if s.na == s.nb else h.diagonal()[:s.na].sum() + h.diagonal()[:s.nb].sum()
    for na, nb, same in ((s.na, s.na, 1), (s.nb, s.nb, 1), (s.na, s.nb, 0), (s.nb, s.na, 0)):
        for p in range(na):
            for q in range(nb):
                e += 0.5 * (eri[slot(p, p, q, q)] - (eri[slot(p, q, q, p)] if same else 0.0))
    return float(e)


def _pair(p, q):
    return p * (p + 1) // 2 + q if p >= q else q * (q + 1) // 2 + p


def prepare(case, seed):
    kind = case["kind"]
    ctx = P.Context(torch.cuda.current_device(), torch.cuda.current_stream())
    st = {"kind": kind, "ctx": ctx, "case": case}
    if kind == "batch":
        keep = []
        for i, s in enumerate(_batch(case["first"], case["count"], case["n_max"])):
            h, eri = s.integrals(seed + i)
            keep.append({"n_orb": s.n_orb, "n_alpha": s.na, "n_beta": s.nb, "h": _gpu(h), "eri": _gpu(eri),
                         "dets": _gpu(s.dets)})
        st["handle"] = _Batch(ctx, keep)
        st["count"] = len(keep)
        return st
    s = _system(case)
    n = s.dets.shape[0]
    h, eri = s.integrals(seed)
    st.update(s=s, n=n, h=_gpu(h), eri=_gpu(eri), dets=_gpu(s.dets))
    if kind != "solve":
        P.shci_load_integrals(ctx.handle, s.n_orb, 0.0, st["h"], st["eri"])
    if kind == "sigma":
        P.shci_build_connectivity(ctx.handle, s.na, s.nb, st["dets"], MODES[case["mode"]])
        st["c"] = _gpu(_coefficients(n, case["k"], seed))
        st["y"] = torch.empty_like(st["c"])
    elif kind == "solve":
        st["vecs"] = torch.empty((case["k"], n), dtype=torch.float64, device="cuda")
    elif kind == "gradient":
        P.shci_build_connectivity(ctx.handle, s.na, s.nb, st["dets"], P.SHCI_STORED)
        st["c"] = _gpu(_coefficients(n, 1, seed)[0])
        st["dh"], st["deri"] = torch.empty_like(st["h"]), torch.empty_like(st["eri"])
    elif kind == "grow":
        st["head"], st["tail"] = st["dets"][:n - case["new"]], st["dets"][n - case["new"]:]
        st["c"] = _gpu(_coefficients(n, 1, seed)[0])
        st["y"], st["diag"] = torch.empty_like(st["c"]), torch.empty_like(st["c"])
    else:
        P.shci_build_connectivity(ctx.handle, s.na, s.nb, st["dets"], P.SHCI_STORED)
        c = _coefficients(n, case.get("k", 1), seed)
        st["c"] = _gpu(c if kind == "select" else c[0])
        st["e_var"] = _reference_energy(s, h, eri) - 0.5
        st["seed"] = seed
    if kind == "select":
        # the next space, with room for what is selected
        st["grown"] = torch.empty((max(2_000_000, 64 * n), st["dets"].shape[1]), dtype=torch.int64, device="cuda")
    return st


class _Batch:
    """Owns a batch handle (and the context it belongs to)."""

    def __init__(self, ctx, systems):
        self.ctx, self.systems = ctx, systems
        self.handle = P.shci_batch_create(ctx.handle, systems)

    def __del__(self):
        P.shci_batch_destroy(self.handle)


# ---------------------------------------------------------------- one pass

def run(st):
    kind, case, H = st["kind"], st["case"], st["ctx"].handle
    if kind == "sigma":
        return P.shci_sigma(H, st["c"], st["y"])
    if kind == "solve":
        s = st["s"]
        P.shci_load_integrals(H, s.n_orb, 0.0, st["h"], st["eri"])
        P.shci_build_connectivity(H, s.na, s.nb, st["dets"], P.SHCI_STORED)
        e, _, _ = P.shci_davidson(H, case["k"], 1e-10, 400, vecs=st["vecs"])
        return {"energies": e, "vectors": st["vecs"]}
    if kind == "gradient":
        P.shci_energy_backward(H, st["c"], 1.0, st["dh"], st["deri"])
        return {"dh": st["dh"], "deri": st["deri"]}
    if kind == "grow":
        s = st["s"]
        P.shci_build_connectivity(H, s.na, s.nb, st["head"], P.SHCI_STORED)
        pairs = P.shci_extend_connectivity(H, st["tail"])
        return {"pairs": pairs, "diag": P.shci_get_diag(H, st["diag"]), "y": P.shci_sigma(H, st["c"], st["y"])}
    if kind == "select":
        new = P.shci_select(H, st["c"], case["eps1"])
        grown, n, m = st["grown"], st["n"], new.shape[0]
        grown[:n].copy_(st["dets"])
        grown[n:n + m].copy_(new)
        grown[n + m:].zero_()
        return {"grown": grown, "count": m}
    if kind == "pt2":
        e2, n_pert = P.shci_pt2(H, st["c"], st["e_var"], case["eps2"])
        return {"e2": e2, "n_pert": n_pert}
    if kind == "pt2_sampled":
        e2, err = P.shci_pt2_semistochastic(H, st["c"], st["e_var"], case["eps2"], case["eps2_d"], case["n_d"],
                                            case["samples"], st["seed"])
        return {"e2": e2, "err": err}
    e, _, converged, _ = P.shci_batch_davidson(H, st["handle"].handle, st["count"], case["k"])
    return {"energies": e, "converged": converged}


# ---------------------------------------------------------------- the work of one pass

@functools.lru_cache(maxsize=64)
def _n_pairs(space, n):
    """Connected pairs of a space (counted by the library, on its reference integrals)."""
    s = _fci(*n) if space == "fci" else _space(space, n)
    return _count(s)


def _count(s):
    with P.Context(torch.cuda.current_device(), torch.cuda.current_stream()) as ctx:
        P.shci_load_integrals(ctx.handle, s.n_orb, 0.0, _gpu(s.h), _gpu(s.eri))
        return P.shci_build_connectivity(ctx.handle, s.na, s.nb, _gpu(s.dets), P.SHCI_ON_THE_FLY)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        pairs, inputs = 0, 0
        for s in _batch(case["first"], case["count"], case["n_max"]):
            pairs += _count(s)
            inputs += s.dets.nbytes + s.eri.nbytes
        return {"bytes": inputs + 12 * pairs, "flops": 4.0 * pairs * case["k"] * PRODUCTS}
    s = _system(case)
    n = s.dets.shape[0]
    inputs = s.dets.nbytes + s.eri.nbytes + s.h.nbytes
    if kind in ("select", "pt2", "pt2_sampled"):
        # every single move of every determinant has to be evaluated; the doubles come from sorted lists
        rows = n if kind != "pt2_sampled" else n + case["samples"] * case["n_d"]
        singles = s.na * (s.n_orb - s.na) + s.nb * (s.n_orb - s.nb)
        return {"bytes": inputs + 8 * n * case.get("k", 1), "flops": float(rows) * singles * (s.na + s.nb) * 2}
    pairs = _n_pairs(case["space"], (case["n_orb"], case["na"], case["nb"]) if case["space"] == "fci" else case["n"])
    k = case.get("k", 1)
    if kind == "sigma":
        stored = {"stored": 24, "upper": 12, "fly": 0}[case["mode"]] * pairs
        return {"bytes": (stored or inputs) + 8 * n * (2 * k + 1), "flops": 4.0 * pairs * k + 2.0 * n * k}
    if kind == "solve":
        # H is larger than the caches: each product reads it
        return {"bytes": inputs + 24 * pairs * (PRODUCTS + 1) + 8 * n * k, "flops": 4.0 * pairs * k * PRODUCTS}
    if kind == "gradient":
        return {"bytes": 2 * inputs + 8 * n, "flops": 4.0 * pairs}
    return {"bytes": inputs + 48 * pairs + 24 * n, "flops": 8.0 * pairs}


# ---------------------------------------------------------------- 64-bit values in plain torch

class Plain:
    """Matrix elements in the spin-orbital form: orbital p of spin s is s * n_orb + p, alpha first."""

    def __init__(self, s, h, eri):
        n = self.n = s.n_orb
        self.s = s
        p = torch.arange(n, device="cuda")
        pq = torch.maximum(p[:, None], p) * (torch.maximum(p[:, None], p) + 1) // 2 + torch.minimum(p[:, None], p)
        pq = pq.reshape(-1)
        hi, lo = torch.maximum(pq[:, None], pq), torch.minimum(pq[:, None], pq)
        self.slot = (hi * (hi + 1) // 2 + lo).reshape(n, n, n, n)
        self.h = _gpu(h)
        self.eri = _gpu(eri)[self.slot]
        self.occ = self.unpack(_gpu(s.dets))
        self.before = torch.cumsum(self.occ, 1, dtype=torch.int16) - self.occ      # electrons before each spin orbital

    def unpack(self, dets):
        w = dets.shape[1] // 2
        o = torch.arange(self.n, device="cuda")
        return torch.cat([(dets[:, spin * w + (o >> 6)] >> (o & 63)) & 1 for spin in (0, 1)], 1).to(torch.uint8)

    def coulomb(self):
        J = torch.einsum("pqkk->pqk", self.eri)
        K = torch.einsum("pkkq->pqk", self.eri)
        return J, K

    def diag(self, occ):
        Jd, Kd = torch.einsum("kkll->kl", self.eri), torch.einsum("kllk->kl", self.eri)
        a, b = occ[:, :self.n].double(), occ[:, self.n:].double()
        two = ((a + b) @ Jd * (a + b)).sum(1) - (a @ Kd * a).sum(1) - (b @ Kd * b).sum(1)
        return (a + b) @ torch.diagonal(self.h) + 0.5 * two

    def pairs(self):
        """Chunks (i, j) of the connected ordered pairs, singles apart from doubles."""
        f = self.occ.to(torch.float16)
        n, electrons = f.shape[0], self.s.na + self.s.nb
        rows = max(1, min(n, int(2e9) // n))
        for r in range(0, n, rows):
            common = f[r:r + rows] @ f.T
            for degree in (1, 2):
                at = torch.nonzero(common == electrons - degree)
                for c in range(0, at.shape[0], 2_000_000):
                    yield degree, at[c:c + 2_000_000, 0] + r, at[c:c + 2_000_000, 1]

    def element(self, degree, i, j):
        oi, oj = self.occ[i], self.occ[j]
        p = torch.nonzero(oi > oj)[:, 1].reshape(-1, degree)
        q = torch.nonzero(oj > oi)[:, 1].reshape(-1, degree)
        odd = (self.before[i[:, None], p].sum(1) + self.before[j[:, None], q].sum(1)) & 1
        sign = 1.0 - 2.0 * odd
        P_, Q_ = p % self.n, q % self.n
        if degree == 1:
            core = (oi & oj).double()
            up, dn = core[:, :self.n], core[:, self.n:]
            J, K = self.coulomb()
            p0, q0 = P_[:, 0], Q_[:, 0]
            same = torch.where((p[:, :1] < self.n), up, dn)
            v = self.h[p0, q0] + ((up + dn) * J[p0, q0]).sum(1) - (same * K[p0, q0]).sum(1)
        else:
            # p and q ascend: with one particle in each spin the holes pair off in the same order
            a, b, c, d = P_[:, 0], P_[:, 1], Q_[:, 0], Q_[:, 1]
            same = ((p[:, 0] < self.n) == (p[:, 1] < self.n)).double()
            v = self.eri[a, c, b, d] - same * self.eri[a, d, b, c]
        return sign * v

    def sigma(self, c):
        y = self.diag(self.occ) * c
        for degree, i, j in self.pairs():
            y.index_add_(1, i, self.element(degree, i, j) * c[:, j])
        return y

    def matrix(self):
        n = self.occ.shape[0]
        ii, jj, vv = [torch.arange(n, device="cuda")], [torch.arange(n, device="cuda")], [self.diag(self.occ)]
        for degree, i, j in self.pairs():
            ii.append(i)
            jj.append(j)
            vv.append(self.element(degree, i, j))
        return torch.sparse_coo_tensor(torch.stack([torch.cat(ii), torch.cat(jj)]), torch.cat(vv), (n, n)).to_sparse_csr()

    def lowest(self, k):
        """The k lowest eigenvalues that the usual start reaches: Lanczos with full reorthogonalisation from the k
        lowest eigenvectors within the 64 determinants of lowest diagonal (a start stays in its symmetry sectors)."""
        A = self.matrix()
        n = A.shape[0]
        steps = min(n, 400)
        first = torch.argsort(self.diag(self.occ))[:64]
        block = torch.zeros((n, first.numel()), dtype=torch.float64, device="cuda")
        block[first, torch.arange(first.numel(), device="cuda")] = 1.0
        vec = torch.linalg.eigh((A @ block)[first])[1][:, :k]
        q = torch.zeros(n, dtype=torch.float64, device="cuda")
        q[first] = vec.sum(1)
        Q = torch.zeros((steps, n), dtype=torch.float64, device="cuda")
        alpha, beta = [], []
        q = q / q.norm()
        for m in range(steps):
            Q[m] = q
            r = torch.mv(A, q)
            alpha.append(torch.dot(q, r).item())
            for _ in range(2):
                r = r - Q[:m + 1].T @ (Q[:m + 1] @ r)
            b = r.norm().item()
            T = np.diag(alpha) + np.diag(beta, 1) + np.diag(beta, -1)
            values, vectors = np.linalg.eigh(T)
            if b < 1e-10 or (m >= k and b * np.abs(vectors[-1, :k]).max() < 1e-8):
                break
            beta.append(b)
            q = r / b
        return torch.from_numpy(values[:k])

    def gradient(self, c):
        self.h.requires_grad_(True)
        self.eri.requires_grad_(True)
        (self.diag(self.occ) * c * c).sum().backward()
        for degree, i, j in self.pairs():
            (self.element(degree, i, j) * c[i] * c[j]).sum().backward()
        n_slots = int(self.slot.max()) + 1
        deri = torch.zeros(n_slots, dtype=torch.float64, device="cuda")
        deri.index_add_(0, self.slot.reshape(-1), self.eri.grad.reshape(-1))
        return self.h.grad, deri

    def excitations(self, lo, hi):
        """Every excitation of determinants [lo, hi): chunks (row, determinant key, matrix element).  The key is the
        bit string over the 2 n_orb spin orbitals."""
        n, s = self.n, self.s
        occ = self.occ[lo:hi]
        m = occ.shape[0]
        J, K = self.coulomb()
        bit = torch.ones(2 * n, dtype=torch.int64, device="cuda") << torch.arange(2 * n, device="cuda")
        key = (occ.long() * bit).sum(1)
        up, dn = occ[:, :n].double(), occ[:, n:].double()
        full, empty = [], []
        for spin, ne in ((0, s.na), (1, s.nb)):
            o = occ[:, spin * n:(spin + 1) * n]
            full.append(torch.nonzero(o)[:, 1].reshape(m, ne) + spin * n)
            empty.append(torch.nonzero(o == 0)[:, 1].reshape(m, n - ne) + spin * n)
        before = self.before[lo:hi].long()
        at = lambda t, x: torch.gather(t, 1, x)
        row = lambda x: torch.arange(lo, hi, device="cuda")[:, None].expand_as(x)
        for spin, ne in ((0, s.na), (1, s.nb)):
            q, p = full[spin].repeat_interleave(n - ne, 1), empty[spin].repeat(1, ne)
            sign = 1.0 - 2.0 * ((at(before, q) + at(before, p) - (q < p).long()) & 1)
            P_, Q_ = p - spin * n, q - spin * n
            same = (up, dn)[spin]
            v = self.h[P_, Q_] + torch.einsum("mk,mxk->mx", up + dn, J[P_, Q_]) - J[P_, Q_, Q_]
            v = v - torch.einsum("mk,mxk->mx", same, K[P_, Q_]) + K[P_, Q_, Q_]
            yield row(v), key[:, None] ^ bit[p] ^ bit[q], sign * v
            if ne > 1 and n - ne > 1:
                fo = torch.tensor(list(itertools.combinations(range(ne), 2)), device="cuda")
                em = torch.tensor(list(itertools.combinations(range(n - ne), 2)), device="cuda")
                for x, y in fo.tolist():
                    q1, q2 = full[spin][:, x:x + 1], full[spin][:, y:y + 1]
                    p1, p2 = empty[spin][:, em[:, 0]], empty[spin][:, em[:, 1]]
                    odd = x + y + at(before, p1) + at(before, p2) - sum((a < b).long() for a in (q1, q2)
                                                                          for b in (p1, p2)) + 1
                    b_, d_, a_, c_ = q1 - spin * n, q2 - spin * n, p1 - spin * n, p2 - spin * n
                    v = self.eri[a_, b_, c_, d_] - self.eri[a_, d_, c_, b_]
                    yield row(v), key[:, None] ^ bit[q1] ^ bit[q2] ^ bit[p1] ^ bit[p2], (1.0 - 2.0 * (odd & 1)) * v
        for x in range(s.na):
            qa, pa = full[0][:, x:x + 1], empty[0]
            odd_a = at(before, qa) + at(before, pa) - (qa < pa).long()
            for y in range(s.nb):
                qb, pb = full[1][:, y:y + 1], empty[1]
                odd_b = at(before, qb) + at(before, pb) - (qb < pb).long()
                odd = (odd_a[:, :, None] + odd_b[:, None, :]).reshape(m, -1)
                v = self.eri[pa[:, :, None], qa[:, :, None], pb[:, None, :] - n, qb[:, None, :] - n].reshape(m, -1)
                k2 = (key[:, None, None] ^ (bit[pa] ^ bit[qa])[:, :, None] ^ (bit[pb] ^ bit[qb])[:, None, :]).reshape(m, -1)
                yield row(v), k2, (1.0 - 2.0 * (odd & 1)) * v

    def pt2(self, c, e_var, eps2):
        bit = torch.ones(2 * self.n, dtype=torch.int64, device="cuda") << torch.arange(2 * self.n, device="cuda")
        own = torch.sort((self.occ.long() * bit).sum(1))[0]
        keys, terms = [], []
        for lo in range(0, self.occ.shape[0], 20_000):
            for row, key, v in self.excitations(lo, min(lo + 20_000, self.occ.shape[0])):
                t = v * c[row]
                kept = t.abs() >= eps2
                keys.append(key[kept])
                terms.append(t[kept])
        keys, terms = torch.cat(keys), torch.cat(terms)
        place = torch.searchsorted(own, keys).clamp_(max=own.numel() - 1)
        out = own[place] != keys
        keys, inverse = torch.unique(keys[out], return_inverse=True)
        total = torch.zeros(keys.numel(), dtype=torch.float64, device="cuda").index_add_(0, inverse, terms[out])
        e2 = 0.0
        for r in range(0, keys.numel(), 4_000_000):
            occ = ((keys[r:r + 4_000_000, None] >> torch.arange(2 * self.n, device="cuda")) & 1).to(torch.uint8)
            e2 += float((total[r:r + 4_000_000] ** 2 / (e_var - self.diag(occ))).sum())
        return e2


def exact(case, seed):
    kind = case["kind"]
    if kind in ("select", "pt2_sampled"):
        return None
    if kind == "batch":
        systems = _batch(case["first"], case["count"], case["n_max"])
        if sum(float(s.dets.shape[0]) ** 2 for s in systems) > EXACT_PAIRS:
            return None
        e = [Plain(s, *s.integrals(seed + i)).lowest(case["k"]) for i, s in enumerate(systems)]
        return {"energies": torch.stack(e), "converged": None}
    s = _system(case)
    n = s.dets.shape[0]
    if float(n) * n > EXACT_PAIRS or (kind == "solve" and n > 60_000):
        return None
    h, eri = s.integrals(seed)
    plain = Plain(s, h, eri)
    if kind == "sigma":
        return plain.sigma(_gpu(_coefficients(n, case["k"], seed)))
    if kind == "solve":
        return {"energies": plain.lowest(case["k"]), "vectors": None}
    if kind == "gradient":
        dh, deri = plain.gradient(_gpu(_coefficients(n, 1, seed)[0]))
        return {"dh": dh, "deri": deri}
    c = _gpu(_coefficients(n, 1, seed))
    if kind == "grow":
        return {"pairs": None, "diag": plain.diag(plain.occ), "y": plain.sigma(c)[0]}
    if 2 * s.n_orb > 62:
        return None
    return {"e2": plain.pt2(c[0], _reference_energy(s, h, eri) - 0.5, case["eps2"]), "n_pert": None}
