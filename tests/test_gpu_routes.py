"""Routes chosen by size, at the sizes where they change (needs a GB300): bucket counts in shared
memory against one counter update a record, the one-CTA scan, float64 sweeps of every support, and
batches with 4096^2 channels, few visibilities in them (mostly empty work items).

Bars, of the largest value: float64 1e-12 and float32 1e-5, as for the work items (sums of up to 1e5
terms of 53-bit rounding; table and products rounded to 2^-24 and chains of up to 5e4 terms).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import imaging as I  # noqa: E402
from paper_1906_07102_gb300 import lmg  # noqa: E402
from paper_1906_07102_gb300 import synthetic as S  # noqa: E402
from tests.cases import INTERP, caller_table  # noqa: E402
from tests.test_gpu_work_items import check, positions  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,N,nvis", [
    ("c64", 256, 65535), ("c64", 256, 65536), ("c64", 512, 262144 + 4097),  # 1024 and 4096 buckets, 64 each
    ("c64", 576, 70000), ("c64", 1024, 3000), ("c64", 1088, 3000),         # 16,384 buckets scanned in one CTA; more
    ("c128", 96, 18432), ("c128", 352, 3872 * 64 + 1)])
def test_bucket_counts_and_scan(dtype, N, nvis):
    """With positions that are dropped among them."""
    W, Ms = 4, 50
    uv = positions(N, nvis - 2000, 2000, nvis % 97)
    uv[[0, 77, nvis - 1]] = [[np.nan, 1.0], [1.0, np.inf], [1e12, 0.0]]
    keep = np.ones(nvis, bool)
    keep[[0, 77, nvis - 1]] = False
    T = caller_table(W, Ms)
    p = lmg.Plan(lmg.Table(W, 0.5, Ms, "linear", values=T), N // 2, 1.0 / N, nvis, dtype)
    p.bin(torch.from_numpy(uv).cuda())
    assert p.dropped() == 3 and p.status() == (0, 0)
    vis = 1.0 + 0.3 * S.complex_normal(nvis, 5)
    cd, tol = (torch.complex64, 1e-5) if dtype == "c64" else (torch.complex128, 1e-12)
    op = I.Plan(uv[keep, 0], uv[keep, 1], W, N)
    ref = I.grid(op, T, Ms, INTERP["linear"], vis[keep])
    assert np.abs(p.grid(torch.from_numpy(vis).to("cuda", cd)).cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
    G = S.random_image(N, 6)
    d = p.degrid(torch.from_numpy(G).to("cuda", cd)).cpu().numpy()
    dref = I.degrid(op, T, Ms, INTERP["linear"], G)
    assert np.abs(d[keep] - dref).max() <= tol * np.abs(dref).max() and not d[~keep].any()


@pytest.mark.parametrize("W", [2, 4, 5, 6, 7, 10, 11, 12, 13, 15])
@pytest.mark.parametrize("interp", ["linear", "cubic"])
def test_float64_supports(W, interp):
    check(64, W, interp, 100, "c128", "plain", positions(64, 37, 300, W), 1e-12)


@pytest.mark.parametrize("x0s", [(0.5, 0.5), (0.5, 0.5 + 4 / 4096)])
def test_batch_with_4096_channels(x0s):
    """Fused transforms where every 4096^2 channel keeps a multiple of 8 pixels, the library's for the
    class otherwise; a 1024^2 channel beside them."""
    W, Ms, sizes = 4, 50, [(4096, x0s[0]), (1024, 0.5), (4096, x0s[1])]
    T = caller_table(W, Ms)
    tabs = [lmg.Table(W, x0, Ms, "linear", values=T) for _, x0 in sizes]
    n = [int(round(N * x0)) for N, x0 in sizes]
    uv = [torch.from_numpy(S.disk_uniform(3001 + 7 * i, 0.45 * N, i)).cuda() for i, (N, _) in enumerate(sizes)]
    b = lmg.Batch(tabs, n, [1.0 / N for N, _ in sizes], [u.shape[0] for u in uv])
    b.bin(uv)
    vis = [torch.from_numpy(S.complex_normal(u.shape[0], 3)).to("cuda", torch.complex64) for u in uv]
    model = [torch.from_numpy(S.random_image(k, 4)).to("cuda", torch.complex64) for k in n]
    for _ in range(2):  # captured, then replayed
        img, pred = b.dirty_image(vis), b.predict_vis(model)
    for c in range(3):
        p = lmg.Plan(tabs[c], n[c], 1.0 / sizes[c][0], uv[c].shape[0], "c128")
        p.bin(uv[c])
        for got, ref in ((img[c], p.dirty_image(vis[c].to(torch.complex128))),
                         (pred[c], p.predict_vis(model[c].to(torch.complex128)))):
            assert float((got - ref).abs().max()) <= 1e-5 * float(ref.abs().max())
        q = lmg.Plan(tabs[c], n[c], 1.0 / sizes[c][0], uv[c].shape[0], "c64")
        q.bin(uv[c])
        assert q.status() == (0, 0)
