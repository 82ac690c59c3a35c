"""Replayed graphs of a batch with 4096^2 channels (needs a GB300): their fused transforms share one
scratch, and the caller's image pointers are arguments of the captured launches. The outputs of a
second call on the same buffers follow the buffers' new contents, without another capture.

Bar: 1e-5 of the largest value, as for the batch tests (order of float32 sums, transforms).
"""
import pytest

torch = pytest.importorskip("torch")

from paper_1906_07102_gb300 import lmg  # noqa: E402
from paper_1906_07102_gb300 import synthetic as S  # noqa: E402
from tests.cases import caller_table  # noqa: E402

pytestmark = pytest.mark.gpu


def test_replay_follows_the_buffers():
    W, sides = 4, [4096, 1024, 4096]
    tab = lmg.Table(W, 0.5, 50, "linear", values=caller_table(W, 50))
    uv = [torch.from_numpy(S.disk_uniform(3001 + 7 * i, 0.45 * N, i)).cuda() for i, N in enumerate(sides)]
    b = lmg.Batch([tab] * 3, [N // 2 for N in sides], [1.0 / N for N in sides], [u.shape[0] for u in uv])
    b.bin(uv)
    plans = []
    for N, u in zip(sides, uv):
        plans.append(lmg.Plan(tab, N // 2, 1.0 / N, u.shape[0], "c64"))
        plans[-1].bin(u)
        assert plans[-1].status() == (0, 0)
    vis = [torch.empty(u.shape[0], dtype=torch.complex64, device="cuda") for u in uv]
    model = [torch.empty(N // 2, N // 2, dtype=torch.complex64, device="cuda") for N in sides]
    img, pred = [torch.empty_like(m) for m in model], [torch.empty_like(v) for v in vis]
    captured = []
    for seed in (1, 2, 3):
        for i, (v, m) in enumerate(zip(vis, model)):
            v.copy_(torch.from_numpy(S.complex_normal(v.numel(), seed + 10 * i)))
            m.copy_(torch.from_numpy(S.random_image(m.shape[0], seed + 20 * i)))
        b.dirty_image(vis, out=img)
        b.predict_vis(model, out=pred)
        captured.append(b.info()["graphs_captured"])
        for p, v, m, x, y in zip(plans, vis, model, img, pred):
            for got, ref in ((x, p.dirty_image(v)), (y, p.predict_vis(m))):
                assert float((got - ref).abs().max()) <= 1e-5 * float(ref.abs().max())
    assert captured[1] == captured[0] and captured[2] == captured[0]
