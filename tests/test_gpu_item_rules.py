"""Where the rules for work items and their routes change (needs a GB300): blocks of rows taken by one
warp each while items are made. References are the float64 oracle with the same table.

Bars, of the largest cell. Float64 1e-12 (sums of up to 1e5 terms of 53-bit rounding). Float32:
a term carries at most six roundings of 2^-24 (two interpolated weights, their product with the
visibility), 3.6e-7, and a plain chain of n terms of one sign drifts by about 2^-25 sqrt(n / 3) of its
sum, 8e-7 for the 2000 records that chains end with here: 4e-6 for plain sums (four times both),
1e-6 for compensated ones, whose chains add no more than the last rounding.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import imaging as I  # noqa: E402
from paper_1906_07102_gb300 import lmg  # noqa: E402
from paper_1906_07102_gb300 import synthetic as S  # noqa: E402
from tests.cases import INTERP, caller_table  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {"plain": 4e-6, "compensated": 1e-6}


def clusters(N, spread, dense, seed):
    """spread positions over the disk, and dense ones in four pairs of rows of one block around a
    strip's edge (two next to each other, two apart)."""
    g = np.random.default_rng(seed)
    a = S.disk_uniform(spread, 0.45 * N, seed) if spread else np.zeros((0, 2))
    row = g.choice([4.0, 6.0, 12.0, 20.0], dense)
    b = np.stack([g.uniform(-1.5, 1.5, dense), row + g.uniform(0.1, 1.9, dense)], 1)
    uv = np.concatenate([a, b])
    return np.ascontiguousarray(uv[g.permutation(len(uv))])


def check(N, W, interp, dtype, accum, uv, max_vis=None, Ms=200):
    """Gridding and degridding against the oracle; returns the plan's info."""
    T = caller_table(W, Ms)
    p = lmg.Plan(lmg.Table(W, 0.5, Ms, interp, values=T), N // 2, 1.0 / N, max_vis or len(uv), dtype)
    p.bin(torch.from_numpy(uv).cuda())
    assert p.status() == (0, 0)
    vis = 1.0 + 0.3 * S.complex_normal(len(uv), 5)
    cd, tol = (torch.complex64, TOL[accum]) if dtype == "c64" else (torch.complex128, 1e-12)
    op = I.Plan(uv[:, 0], uv[:, 1], W, N)
    ref = I.grid(op, T, Ms, INTERP[interp], vis)
    g = p.grid(torch.from_numpy(vis).to("cuda", cd), accum=accum).cpu().numpy()
    assert np.abs(g - ref).max() <= tol * np.abs(ref).max()
    G = S.random_image(N, 6)
    d = p.degrid(torch.from_numpy(G).to("cuda", cd)).cpu().numpy()
    dref = I.degrid(op, T, Ms, INTERP[interp], G)
    assert np.abs(d - dref).max() <= (1e-5 if dtype == "c64" else 1e-12) * np.abs(dref).max()
    return p.info()


@pytest.mark.parametrize("dtype,accum,N", [
    ("c64", "plain", 1536), ("c64", "plain", 1600), ("c64", "compensated", 1600),  # 576 and 625 blocks
    ("c128", "plain", 1088), ("c128", "plain", 1152)])                              # 578 and 648
def test_blocks_of_rows_in_one_warp(dtype, accum, N):
    """Above 608 blocks, few visibilities on average: a warp makes a block's items, several cut pairs of
    rows among them."""
    check(N, 6, "linear", dtype, accum, clusters(N, 3000, 20000, N))


@pytest.mark.parametrize("N,spread,dense", [(64, 31, 0), (64, 40, 3000), (512, 4001, 20000), (1152, 3000, 33)])
@pytest.mark.parametrize("interp", ["nearest", "linear", "cubic"])
def test_float64_one_cell_supports(N, interp, spread, dense):
    """W = 1 in float64: a lane a record, several of one warp in one cell, rows with few records."""
    check(N, 1, interp, "c128", "plain", clusters(N, spread, dense, N + dense))


@pytest.mark.parametrize("N,W,max_vis,stored", [
    (512, 7, 511, True), (512, 7, 513, False),              # N^3 / 2^18 = 512
    (2048, 7, 32767, True), (2048, 7, 32769, False),        # 32768
    (2176, 9, 200000, False), (2240, 9, 200000, True),      # W >= 9: 1156 and 1225 blocks of rows
    (2496, 8, 200000, False), (2560, 8, 200000, True)])     # 48 MB
def test_route_of_gridding(N, W, max_vis, stored):
    """Rows stored once (every block of rows has an item, empty ones too) or added into a zeroed grid."""
    info = check(N, W, "linear", "c64", "plain", clusters(N, 0, 30, N), max_vis)
    assert (info["items"] >= (N // 64) ** 2) == stored


@pytest.mark.parametrize("accum", ["plain", "compensated"])
@pytest.mark.parametrize("N,W,max_vis,stored", [
    (2496, 8, 0, False), (2560, 8, 0, True), (2560, 3, 0, True), (2240, 16, 0, True), (2048, 16, 0, False),
    (2560, 8, 200000, True)])  # a plan for more visibilities has smaller items
def test_cut_pairs_of_both_routes(accum, N, W, max_vis, stored):
    uv = clusters(N, 2000, 25000, N + W)
    info = check(N, W, "linear", "c64", accum, uv, max_vis)
    assert info["items"] >= (N // 64) ** 2 or not stored


def test_memory_of_a_plan_for_many_visibilities():
    """Records (two of 16 bytes a visibility) and ranks (8 bytes); items, bucket counts and the transforms
    of a 256^2 grid take a few MB. Sums of cut pairs' chains need nothing of their own at this count."""
    nvis = 16 << 20
    tab = lmg.Table(12, 0.5, 200, "linear", values=caller_table(12, 200))
    lmg.Plan(tab, 128, 1.0 / 256, 1000, "c64")  # the library's own first allocations
    used = []
    for _ in range(5):  # other processes' allocations show in the device's free memory too
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        p = lmg.Plan(tab, 128, 1.0 / 256, nvis, "c64")
        used.append(before - torch.cuda.mem_get_info()[0])
        assert p.info()["N"] == 256
        del p
    assert 0 < min(u for u in used if u > 0) <= 40 * nvis + (32 << 20)


@pytest.mark.parametrize("accum", ["plain", "compensated"])
@pytest.mark.parametrize("N,W", [(64, 16), (64, 3), (256, 8), (2560, 7), (2560, 2)])
def test_plan_without_room_for_short_items(monkeypatch, accum, N, W):
    """The sizes a plan falls back to when memory is short: few places for merged chains, several parts of a
    dense pair in each, and on the stored route no spill rows for items below 512 records."""
    monkeypatch.setenv("LMG_INJECT_FAULT", "roomy_plan")
    check(N, W, "linear", "c64", accum, clusters(N, 3000, 40000, N + W), 1 << 17)


@pytest.mark.parametrize("W", [1, 2, 3])
@pytest.mark.parametrize("accum", ["plain", "compensated"])
@pytest.mark.parametrize("N,nvis", [(64, 20000), (64, 300000), (2560, 100000)])
def test_dense_pairs_of_narrow_supports_sum_in_one_order(W, accum, N, nvis):
    """Items are pairs of rows at least, so that with W <= 3 two of them meet in a cell: the same bits on
    every call, however many parts a pair is swept in."""
    tab = lmg.Table(W, 0.5, 200, "linear", values=caller_table(W, 200))
    p = lmg.Plan(tab, N // 2, 1.0 / N, nvis, "c64")
    p.bin(torch.from_numpy(clusters(N, nvis // 2, nvis // 2, W)).cuda())
    vis = torch.from_numpy(S.complex_normal(nvis, 3)).to("cuda", torch.complex64)
    first = torch.view_as_real(p.grid(vis, accum=accum))
    assert p.status() == (0, 0)
    for _ in range(6):
        assert torch.equal(first, torch.view_as_real(p.grid(vis, accum=accum)))
