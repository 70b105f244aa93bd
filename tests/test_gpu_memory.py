"""Calls at the limit of the device's memory: growth beside a large occupancy
bitmap (the bitmap of the new members alone would not fit), and a build without
room for a bitmap.  Results as with room to spare, bit for bit."""
import numpy as np
import pytest
import torch

import shci_synth as S
from tests import gpu_common as G
from tests.test_gpu_extend import _extend
from tests.test_gpu_opposite import _dets, _strings

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _leave(nbytes):
    """Take all free memory but nbytes."""
    return torch.empty(max(_free() - int(nbytes), 0), dtype=torch.uint8, device="cuda")


def _sparse():
    """26 orbitals, 5 electrons a spin, random strings: a bitmap of some 65,000 x 900 cells, 0.9 GB."""
    rng = np.random.default_rng(3)
    s = _strings(range(26), 5)
    pick = rng.choice(s.size * s.size, 150_011, replace=False)
    h, eri, ec = S.integrals(26, 5, 41)
    return h, eri, ec, _dets(s[pick // s.size], s[pick % s.size], 1)


@pytest.mark.parametrize("upper", [False, True])
def test_growth_beside_a_large_bitmap(upper):
    P = G.lib()
    h, eri, ec, dets = _sparse()
    head = dets.shape[0] - 29
    mode = P.SHCI_STORED_UPPER if upper else P.SHCI_STORED
    B = G.Built(P, h, eri, ec, dets[:head], 5, 5, mode=mode)
    taken = _leave(600 * MB)
    try:
        _extend(P, B, dets[head:])
    finally:
        del taken
        _free()
    assert B.stats()["extend_incremental"] == 1
    F = G.Built(P, h, eri, ec, dets, 5, 5, mode=mode)
    assert F.nnz == B.nnz
    for x, y in zip(F.pairs(), B.pairs()):
        assert np.array_equal(x, y)
    x = S.random_vectors(dets.shape[0], 2, 4)
    # the same terms in another order: below 1e-12 of the largest sum of magnitudes for m < 4500 terms
    ii, jj, vv = F.pairs()
    rows = np.abs(F.diag())
    np.add.at(rows, ii, np.abs(vv))
    np.add.at(rows, jj, np.abs(vv))
    assert np.all(np.abs(F.sigma(x) - B.sigma(x)) <= 1e-12 * rows * np.max(np.abs(x)))
    F.close()
    B.close()


def test_build_without_room_for_a_bitmap():
    P = G.lib()
    h, eri, ec, dets = _sparse()
    F = G.Built(P, h, eri, ec, dets, 5, 5)
    want = F.pairs()
    F.close()
    taken = _leave(600 * MB)
    try:
        B = G.Built(P, h, eri, ec, dets, 5, 5)
    finally:
        del taken
        _free()
    for x, y in zip(want, B.pairs()):
        assert np.array_equal(x, y)
    B.close()


@pytest.mark.parametrize("upper", [False, True])
def test_matrix_without_room_for_the_move_tables(upper):
    """A matrix asked for is stored where it fits beside the lists, with the tables
    of single moves or without."""
    P = G.lib()
    cfg, h, eri, ec, dets = G.system("sel_24o_6a6b_1m", 120_000)
    mode = P.SHCI_STORED_UPPER if upper else P.SHCI_STORED
    dh, de, dd = G.dev(h), G.dev(eri), G.dev(dets)
    x = G.dev(S.random_vectors(dets.shape[0], 1, 4))
    y = [torch.empty_like(x), torch.empty_like(x)]

    def build():
        ctx = P.Context(0, torch.cuda.current_stream())
        P.shci_load_integrals(ctx.handle, cfg.n_orb, ec, dh, de)
        return ctx, P.shci_build_connectivity(ctx.handle, cfg.n_alpha, cfg.n_beta, dd, mode)

    build()[0].close()                            # the library's modules are loaded
    before = _free()
    ctx, pairs = build()
    used = before - _free()
    stats = P.shci_get_stats(ctx.handle)
    tables = 16 * (stats["n_alpha_strings"] + stats["n_beta_strings"]) * 300
    assert tables > 16 * MB
    P.shci_sigma(ctx.handle, x, y[0])
    ctx.close()
    taken = _leave(used - tables // 2)
    try:
        ctx, again = build()
    finally:
        del taken
        _free()
    assert again == pairs
    P.shci_sigma(ctx.handle, x, y[1])
    ctx.close()
    if upper:                                     # atomic sums: 2 m 2^-53 of magnitudes below 1e3, m < 4500
        assert (y[0] - y[1]).abs().max() < 1e-9
    else:
        assert torch.equal(y[0], y[1])


def test_a_batch_holds_nothing_of_the_opposite_spin_pass(monkeypatch):
    """Beyond what it holds when every pair of singles is looked up: the lists
    of the pass (8 bytes per beta single, 12 per determinant) are released."""
    P = G.lib()
    cfg, h, eri, ec, dets = G.system("sel_24o_6a6b_1m", 800_000)
    dh, de, dd = G.dev(h), G.dev(eri), G.dev(dets)
    system = {"n_orb": cfg.n_orb, "n_alpha": cfg.n_alpha, "n_beta": cfg.n_beta, "h": dh, "eri": de, "dets": dd}
    ctx = P.Context(0, torch.cuda.current_stream())
    used = {}
    for opp in ("auto", "lookup", "auto"):        # the first loads the library's modules
        monkeypatch.setenv("SHCI_OPP_SPIN", opp)
        before = _free()
        b = P.shci_batch_create(ctx.handle, [system], 0.0)
        used[opp] = before - _free()
        P.shci_batch_destroy(b)
    ctx.close()
    # allocations below 1 MB share blocks of 2 MB: at most a few blocks more
    assert used["auto"] <= used["lookup"] + 6 * MB, used


def test_a_stored_batch_neither_holds_nor_counts_what_it_does_not_read():
    """The bitmap and the tables of single moves serve a member's build: a batch that
    stores H releases them, and plans its storage with their memory."""
    P = G.lib()
    cfg, h, eri, ec, dets = G.system("sel_24o_6a6b_1m", 400_000)
    n = dets.shape[0]
    dh, de, dd = G.dev(h), G.dev(eri), G.dev(dets)
    system = {"n_orb": cfg.n_orb, "n_alpha": cfg.n_alpha, "n_beta": cfg.n_beta, "h": dh, "eri": de, "dets": dd}
    ctx = P.Context(0, torch.cuda.current_stream())
    P.shci_load_integrals(ctx.handle, cfg.n_orb, ec, dh, de)
    pairs = P.shci_build_connectivity(ctx.handle, cfg.n_alpha, cfg.n_beta, dd, P.SHCI_ON_THE_FLY)
    stats = P.shci_get_stats(ctx.handle)
    ctx.close()
    ua, ub = stats["n_alpha_strings"], stats["n_beta_strings"]
    tables, matrix = 16 * (ua + ub) * 300, 24 * pairs
    assert 300 * (ua + ub) <= 24 * n and tables > 32 * MB      # a batch's member takes them
    ctx = P.Context(0, torch.cuda.current_stream())
    used, modes = {}, {}
    for budget in (0.0, -1.0, 0.0, -1.0):                       # the first two load the library's modules
        before = _free()
        b = P.shci_batch_create(ctx.handle, [system], budget)
        used[budget] = before - _free()
        modes[budget] = int(P.shci_batch_get_modes(b, 1)[0])
        P.shci_batch_destroy(b)
    assert modes == {0.0: P.SHCI_ON_THE_FLY, -1.0: P.SHCI_STORED}
    # blocks of 2 MB: at most a few more
    assert used[-1.0] <= used[0.0] + matrix - tables + 8 * MB, (used, matrix, tables)
    # 80 % of the free memory is short of both triangles by 0.4 of the tables, and
    # beyond them by as much with the tables released
    taken = _leave(used[0.0] + matrix / 0.8 - tables // 2)
    try:
        b = P.shci_batch_create(ctx.handle, [system])
        mode = int(P.shci_batch_get_modes(b, 1)[0])
        P.shci_batch_destroy(b)
    finally:
        del taken
        _free()
    ctx.close()
    assert mode == P.SHCI_STORED


def test_the_choice_of_form_does_not_count_tables_of_an_earlier_build():
    """SHCI_AUTO after a build on the fly: its tables of single moves make way for H."""
    P = G.lib()
    cfg, h, eri, ec, dets = G.system("sel_24o_6a6b_1m", 400_000)
    dh, de, dd = G.dev(h), G.dev(eri), G.dev(dets)

    def build(ctx, mode):
        return P.shci_build_connectivity(ctx.handle, cfg.n_alpha, cfg.n_beta, dd, mode)

    modes = []
    for short in (0.0, 1.0):                                    # the first loads the library's modules
        ctx = P.Context(0, torch.cuda.current_stream())
        P.shci_load_integrals(ctx.handle, cfg.n_orb, ec, dh, de)
        pairs = build(ctx, P.SHCI_ON_THE_FLY)
        stats = P.shci_get_stats(ctx.handle)
        tables = 16 * (stats["n_alpha_strings"] + stats["n_beta_strings"]) * 300
        assert tables > 32 * MB
        # 80 % of the free memory is short of the upper triangle by 0.4 of the tables,
        # and beyond it by as much without them
        taken = _leave(12 * pairs / 0.8 - short * tables // 2) if short else None
        try:
            build(ctx, P.SHCI_AUTO)
            modes.append(P.shci_get_stats(ctx.handle)["mode"])
        finally:
            del taken
            _free()
        ctx.close()
    assert modes == [P.SHCI_STORED, P.SHCI_STORED_UPPER]


def test_products_without_room_for_their_grouped_vectors():
    """Eight vectors on the fly with room for the two layouts of the vectors and no third."""
    P = G.lib()
    cfg, h, eri, ec, dets = G.system("sel_24o_6a6b_1m", 400_000)
    n, k = dets.shape[0], 8
    x = G.dev(S.random_vectors(n, k, 4))
    want, got = torch.empty_like(x), torch.empty_like(x)
    F = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta, mode=P.SHCI_ON_THE_FLY)
    P.shci_sigma(F.ctx.handle, x, want)
    B = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta, mode=P.SHCI_ON_THE_FLY)
    taken = _leave(2.5 * 8 * k * n)
    try:
        P.shci_sigma(B.ctx.handle, x, got)
    finally:
        del taken
        _free()
    # the same m <= 16470 terms in another order: 2 m 2^-53 of sums of magnitudes below 1e3
    assert (want - got).abs().max() < 4e-9
    F.close()
    B.close()


def test_gradient_without_room_for_its_grouped_vector():
    P = G.lib()
    cfg, h, eri, ec, dets = G.system("sel_24o_6a6b_1m", 1_000_000)
    c = G.dev(S.random_vectors(dets.shape[0], 1, 4))[0]
    B = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta, mode=P.SHCI_STORED_UPPER)
    out = [[torch.empty((24, 24), dtype=torch.float64, device="cuda"),
            torch.empty(eri.size, dtype=torch.float64, device="cuda")] for _ in range(2)]
    # 32 copies of the gradient, 12 and 2 MB, and not 8 MB more
    taken = _leave(19 * MB)
    try:
        P.shci_energy_backward(B.ctx.handle, c, 1.0, *out[0])
    finally:
        del taken
        _free()
    P.shci_energy_backward(B.ctx.handle, c, 1.0, *out[1])
    for a, b in zip(*out):
        assert (a - b).abs().max() <= 1e-7 * b.abs().max()
    B.close()


def test_build_without_room_for_the_lists_of_the_pass(monkeypatch):
    P = G.lib()
    cfg, h, eri, ec, dets = G.system("sel_24o_6a6b_1m", 1_000_000)
    x = G.dev(S.random_vectors(dets.shape[0], 1, 4))
    dd = G.dev(dets)
    y = [torch.empty_like(x), torch.empty_like(x)]
    F = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta, mode=P.SHCI_ON_THE_FLY)
    P.shci_sigma(F.ctx.handle, x, y[0])
    monkeypatch.setenv("SHCI_OPP_SPIN", "lookup")               # everything but the pass's lists
    B = G.Built(P, h, eri, ec, dets, cfg.n_alpha, cfg.n_beta, mode=P.SHCI_ON_THE_FLY)
    P.shci_sigma(B.ctx.handle, x, y[1])
    monkeypatch.delenv("SHCI_OPP_SPIN")
    taken = _leave(5 * MB)                                      # 4 MB for the members' indices, more for the singles
    try:
        pairs = P.shci_build_connectivity(B.ctx.handle, cfg.n_alpha, cfg.n_beta, dd, P.SHCI_ON_THE_FLY)
        P.shci_sigma(B.ctx.handle, x, y[1])
    finally:
        del taken
        _free()
    assert pairs == F.nnz
    # the same m <= 16470 terms in another order: 2 m 2^-53 of sums of magnitudes below 1e3
    assert (y[0] - y[1]).abs().max() < 4e-9
    F.close()
    B.close()
