"""Work items and the sweeps' two ways to finish rows, at the sizes where they change (needs a
GB300): counts around a target, dense row pairs cut into parts (with plain and compensated sums
and in float64), grids that are added into and grids whose rows are stored once, and supports
that cross strips. References are the float64 oracle with the same table.

Bars: float64 1e-12 of the largest cell (the parity tests' bar for a shared table: sums of up to
1e5 terms of 53-bit rounding). Float32 1e-5 of the largest cell: the table and the products are
rounded to 2^-24 and a plain chain of n terms of one sign drifts by about 2^-25 sqrt(n / 3) of its
sum, 4e-6 for the longest chain here (5e4 terms).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import imaging as I  # noqa: E402
from paper_1906_07102_gb300 import lmg  # noqa: E402
from paper_1906_07102_gb300 import synthetic as S  # noqa: E402
from tests.cases import INTERP, caller_table  # noqa: E402

pytestmark = pytest.mark.gpu


def positions(N, spread, dense, seed):
    """spread positions over the disk, and dense ones within 3 x 2 cells around a strip's edge
    (cells; one pair of rows holds most of them)."""
    g = np.random.default_rng(seed)
    a = S.disk_uniform(spread, 0.45 * N, seed) if spread else np.zeros((0, 2))
    b = np.stack([g.uniform(-1.5, 1.5, dense), g.uniform(0.1, 1.9, dense)], 1)
    uv = np.concatenate([a, b])
    return np.ascontiguousarray(uv[g.permutation(len(uv))])


def check(N, W, interp, Ms, dtype, accum, uv, tol):
    T = caller_table(W, Ms)
    tab = lmg.Table(W, 0.5, Ms, interp, values=T)
    p = lmg.Plan(tab, N // 2, 1.0 / N, len(uv), dtype)
    p.bin(torch.from_numpy(uv).cuda())
    vis = 1.0 + 0.3 * S.complex_normal(len(uv), 5)
    cd = torch.complex64 if dtype == "c64" else torch.complex128
    op = I.Plan(uv[:, 0], uv[:, 1], W, N)
    v = torch.from_numpy(vis).to("cuda", cd)
    ref = I.grid(op, T, Ms, INTERP[interp], vis)
    g = p.grid(v, accum=accum).cpu().numpy()
    assert np.abs(g - ref).max() <= tol * np.abs(ref).max()
    G = S.random_image(N, 6)
    d = p.degrid(torch.from_numpy(G).to("cuda", cd)).cpu().numpy()
    dref = I.degrid(op, T, Ms, INTERP[interp], G)
    assert np.abs(d - dref).max() <= tol * np.abs(dref).max()
    assert p.status() == (0, 0)


@pytest.mark.parametrize("accum", ["plain", "compensated"])
@pytest.mark.parametrize("spread,dense", [(0, 255), (0, 513), (300, 1025), (5000, 6000), (2000, 50000)])
def test_dense_pairs_float32(accum, spread, dense):
    check(256, 7, "linear", 200, "c64", accum, positions(256, spread, dense, dense), 1e-5)


@pytest.mark.parametrize("accum", ["plain", "compensated"])
@pytest.mark.parametrize("W", [3, 12, 16])
def test_dense_pairs_float32_stored_rows(accum, W):
    """A grid too large to be added into (2496^2): rows stored once, spill rows added."""
    check(2496, W, "linear", 200, "c64", accum, positions(2496, 3000, 20000, W), 1e-5)


@pytest.mark.parametrize("W,interp", [(1, "nearest"), (3, "linear"), (8, "quadratic"), (9, "linear"), (14, "cubic"),
                                      (16, "linear")])
@pytest.mark.parametrize("N", [96, 1760])
def test_dense_pairs_float64(W, interp, N):
    """Added into (96^2, three strips) and stored rows (1760^2)."""
    check(N, W, interp, 200, "c128", "plain", positions(N, 700, 5000, W), 1e-12)
