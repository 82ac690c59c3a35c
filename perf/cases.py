"""Performance cases of the library: what a program that images with it has it do, from the
smallest call to the largest, through the public entry points of ``lmg.py``.

``listed()`` names the cases and ``draw(rng)`` gives further ones of the same ranges;
``prepare`` makes the inputs and the plan, ``run`` is one pass, ``work`` counts the bytes and
operations a pass cannot do without, and ``exact`` is the same result in 64 bits with torch.

Kinds of pass:

* ``step``    positions binned, dirty image of the visibilities, prediction of a model image:
              one imaging step on new positions (a new snapshot, facet or pointing).
* ``sweeps``  gridding and degridding with positions binned before: the inner work of an
              iterative reconstruction, which keeps its plan and changes only the values.
* ``fit``     forward and backward of the differentiable prediction of a real image
              (gradient of 1/2 ||P I - V||^2).
* ``static``  binning and gridding through the call that allocates nothing.
* ``batch``   dirty images and predictions of several channels of uneven sizes as one batch,
              with positions binned before and output buffers kept, as its graphs want.

Positions are Earth-rotation tracks of a random array (time-major, one block per channel) or
uniform in a disk; visibilities are those of a few point sources with noise, models sums of
Gaussian blobs. The gridding function is handed over as table values (Kaiser-Bessel window),
which costs the kernels exactly what the library's own least-misfit table does and lets
``exact`` use the same numbers without the library.
"""
import math

import numpy as np
import torch

from paper_1906_07102_gb300 import lmg

C_LIGHT = 299792458.0
DEC = LAT = math.radians(-30.0)
MAX_EXACT_POINTS = 8.0e9  # grid points touched; beyond this the 64-bit sums take too long


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------
def _case(kind, N, x0, W, Ms, interp="linear", dtype="c64", accum="plain", weights=False, layout="disk", nvis=0,
          n_ant=0, n_times=0, n_chan=1, cut=0, hint=False, size_seed=0):
    """A case: grid side N, kept fraction x0, support W, table rate Ms, and the positions (a
    disk of nvis, or n_ant antennas x n_times samples x n_chan channels less the last cut)."""
    return dict(kind=kind, N=N, x0=x0, W=W, Ms=Ms, interp=interp, dtype=dtype, accum=accum, weights=weights,
                layout=layout, nvis=nvis, n_ant=n_ant, n_times=n_times, n_chan=n_chan, cut=cut, hint=hint,
                size_seed=size_seed)


def listed():
    cases = {
        # the smallest problem of the tests, double precision: every launch and host call counts
        "tiny_f64": _case("step", 512, 0.5, 3, 100, "nearest", "c128", nvis=10000),
        # a small facet in single precision (the size of the smoke run): latency again
        "facet_small": _case("step", 256, 0.5, 7, 1000, nvis=20000),
        # a real-time snapshot through the call that allocates nothing, weighted, last sample row partial
        "snapshot_static": _case("static", 1024, 0.5, 7, 1000, weights=True, layout="tracks", n_ant=24, n_times=724,
                                 cut=37),
        # positions in no order, an odd count, a grid side that is no power of two, weighted
        "ragged_odd": _case("step", 1600, 0.625, 5, 400, weights=True, nvis=777777),
        # one iteration of a small differentiable fit
        "fit_small": _case("fit", 1024, 0.5, 8, 1000, layout="tracks", n_ant=24, n_times=89, n_chan=5),
        # the benchmark's step: 64 antennas, 6 h, 4.1M visibilities, 4096^2, W = 7
        "tracks_step": _case("step", 4096, 0.5, 7, 1000, layout="tracks", n_ant=64, n_times=2048, hint=True),
        # the same data in an iterative reconstruction: gridding and degridding on a kept plan
        "tracks_sweeps": _case("sweeps", 4096, 0.5, 7, 1000, weights=True, layout="tracks", n_ant=64, n_times=2048,
                               hint=True),
        # the same visibilities on a coarse grid, compensated: dense cells, high accuracy in single precision
        "dense_core": _case("step", 256, 0.5, 12, 1000, accum="compensated", layout="tracks", n_ant=64, n_times=2048),
        # double precision in earnest: wide support and a cubic table
        "f64_cubic": _case("step", 2048, 0.5, 14, 20000, "cubic", "c128", layout="tracks", n_ant=64, n_times=512,
                           hint=True),
        # frequency channels of uneven visibility counts, grid sizes and supports as one batch
        "channels_batch": _case("batch", 4096, 0.5, 8, 1000, layout="tracks", n_ant=64, n_chan=24, size_seed=2024),
        # differentiable imaging at full size: 64 channels x 384 samples, 49.5M visibilities
        "fit_large": _case("fit", 4096, 0.5, 8, 1000, layout="tracks", n_ant=64, n_times=384, n_chan=64),
        # large and accurate: 8192^2, W = 12, compensated, 128 antennas, 49.9M visibilities
        "large_w12": _case("step", 8192, 0.5, 12, 1000, accum="compensated", layout="tracks", n_ant=128, n_times=768,
                           n_chan=8, hint=True),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A further case of the listed ranges: any grid side that is a multiple of 64, counts and
    table rates spread over their logarithm, supports 3 to 14."""
    kind = rng.choice(["step"] * 5 + ["sweeps"] * 2 + ["fit"] * 2 + ["static", "batch"])
    x0 = rng.choice([0.5, 0.5, 0.5, 0.375, 0.625, 0.75])
    dtype = "c128" if kind in ("step", "sweeps") and rng.random() < 0.25 else "c64"
    interp, Ms = "linear", _log_int(rng, 100, 1000)
    if dtype == "c128":
        N, W, most = 64 * _log_int(rng, 4, 32), rng.randint(3, 14), 1.0e6
        if rng.random() < 0.5:
            interp, Ms = "cubic", _log_int(rng, 200, 20000)
    elif kind == "static":
        N, W, most = 64 * _log_int(rng, 4, 32), rng.randint(4, 10), 2.5e5
    else:
        N, W, most = 64 * _log_int(rng, 3, 64), rng.randint(3, 12), 8.0e6
    if interp == "linear" and rng.random() < 0.15:
        interp = "nearest"
    if kind == "batch":
        return _case("batch", rng.choice([2048, 4096]), 0.5, rng.choice([4, 6, 8, 9]), Ms, layout="tracks", n_ant=64,
                     n_chan=rng.randint(4, 20), size_seed=rng.randint(0, 10 ** 6))
    accum = "compensated" if dtype == "c64" and kind != "static" and W >= 9 and rng.random() < 0.5 else "plain"
    nvis = _log_int(rng, 1.0e4, most)
    c = _case(kind, N, x0, W, Ms, interp, dtype, accum if kind != "fit" else "plain",
              weights=kind != "fit" and rng.random() < 0.5)
    if kind != "fit" and rng.random() < 0.3:
        c.update(nvis=nvis)
    else:
        n_ant = rng.randint(12, 64)
        n_bl = n_ant * (n_ant - 1) // 2
        n_chan = rng.choice([1, 1, 2, 5])
        n_times = max(1, nvis // (n_bl * n_chan))
        c.update(layout="tracks", n_ant=n_ant, n_times=n_times, n_chan=n_chan, hint=rng.random() < 0.7,
                 cut=rng.randint(0, n_bl // 2))
    return c


def _channels(case):
    """Sizes of a batch's channels (plain cases): visibility counts log-uniform in 1e5 to 2e6,
    grid sides 1024 to the case's, supports up to the case's."""
    g = np.random.default_rng(case["size_seed"])
    sides = [n for n in (1024, 2048, 4096) if n <= case["N"]]
    n_bl = case["n_ant"] * (case["n_ant"] - 1) // 2
    out = []
    for _ in range(case["n_chan"]):
        nvis = int(math.exp(g.uniform(math.log(1.0e5), math.log(2.0e6))))
        n_times = -(-nvis // n_bl)
        out.append(_case("step", int(g.choice(sides)), case["x0"], int(g.choice([case["W"] - 4, case["W"] - 2, case["W"]]))
                         if case["W"] > 4 else case["W"], case["Ms"], layout="tracks", n_ant=case["n_ant"],
                         n_times=n_times, cut=n_times * n_bl - nvis))
    return out


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _window(W, Ms):
    """Kaiser-Bessel window on the table layout: row i at s = i / Ms, entry j at
    d = j - W/2 + s."""
    d = np.arange(W)[None, :] - W / 2 + (np.arange(Ms + 1) / Ms)[:, None]
    return np.i0(2.3 * W * np.sqrt(np.clip(1 - (2 * d / W) ** 2, 0, None))) / np.i0(2.3 * W)


def _positions(case, gen):
    """(u, v) in wavelengths, float64 [nvis, 2] on the GPU, and the pixel scale."""
    dev = torch.device("cuda")
    if case["layout"] == "disk":
        r = 0.45 * case["N"] * torch.sqrt(torch.rand(case["nvis"], dtype=torch.float64, device=dev, generator=gen))
        th = 2 * math.pi * torch.rand(case["nvis"], dtype=torch.float64, device=dev, generator=gen)
        return torch.stack([r * torch.cos(th), r * torch.sin(th)], 1), 1.0 / case["N"]
    en = torch.randn(2, case["n_ant"], dtype=torch.float64, device=dev, generator=gen) * 1000.0
    i, j = torch.triu_indices(case["n_ant"], case["n_ant"], 1, device=dev)
    d_e, d_n = en[0, j] - en[0, i], en[1, j] - en[1, i]
    x, y, z = -d_n * math.sin(LAT), d_e, d_n * math.cos(LAT)
    n_t, half = case["n_times"], math.radians(15.0 * 6.0) / 2
    ha = -half + (torch.arange(n_t, dtype=torch.float64, device=dev) + 0.5) * (2 * half / n_t)
    sin_h, cos_h = torch.sin(ha)[:, None], torch.cos(ha)[:, None]
    u = sin_h * x + cos_h * y
    v = -math.sin(DEC) * cos_h * x + math.sin(DEC) * sin_h * y + math.cos(DEC) * z
    m = torch.stack([u, v], -1).reshape(-1, 2)
    if case["n_chan"] == 1:
        f = torch.tensor([1.4e9], dtype=torch.float64, device=dev)
    else:
        f = torch.linspace(0.95e9, 1.05e9, case["n_chan"], dtype=torch.float64, device=dev)
    uv = torch.cat([m * (g / C_LIGHT) for g in f])
    scale = 0.45 / float(uv.abs().max())
    return uv[:uv.shape[0] - case["cut"]].contiguous(), scale


def _values(uv, scale, case, gen):
    """Visibilities of eight point sources in the kept field, with noise."""
    n = uv.shape[0]
    half = 0.45 * case["N"] * case["x0"] * scale
    lm = (torch.rand(8, 2, dtype=torch.float64, device=uv.device, generator=gen) * 2 - 1) * half
    flux = torch.exp(torch.rand(8, dtype=torch.float64, device=uv.device, generator=gen) * math.log(1e-3))
    real = torch.float32 if case["dtype"] == "c64" else torch.float64
    out = torch.randn(n, 2, dtype=real, device=uv.device, generator=gen) * 0.1
    for s in range(8):
        turn = uv[:, 0] * -lm[s, 0] - uv[:, 1] * lm[s, 1]
        ph = ((turn - torch.round(turn)) * (2 * math.pi)).to(real)
        fs = float(flux[s])
        out[:, 0].add_(torch.cos(ph), alpha=fs)
        out[:, 1].add_(torch.sin(ph), alpha=fs)
    return torch.view_as_complex(out)


def _model(case, gen):
    """Real model image: 32 Gaussian blobs."""
    n = int(round(case["N"] * case["x0"]))
    r = torch.rand(4, 32, dtype=torch.float64, device="cuda", generator=gen)
    x = torch.arange(n, dtype=torch.float64, device="cuda")
    sg = torch.exp(r[2] * math.log(8.0))[:, None]
    gx = torch.exp(-((x - n * (0.1 + 0.8 * r[0][:, None])) / sg) ** 2 / 2)
    gy = torch.exp(-((x - n * (0.1 + 0.8 * r[1][:, None])) / sg) ** 2 / 2)
    return (gy * torch.exp(r[3] * math.log(1e-3))[:, None]).T @ gx


def _inputs(case, seed):
    """Everything a case's pass reads, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    uv, scale = _positions(case, gen)
    d = dict(case=case, uv=uv, scale=scale, vis=_values(uv, scale, case, gen), weights=None)
    cplx = torch.complex64 if case["dtype"] == "c64" else torch.complex128
    real = torch.float32 if case["dtype"] == "c64" else torch.float64
    if case["weights"]:
        d["weights"] = torch.rand(uv.shape[0], dtype=real, device="cuda", generator=gen) * 1.9 + 0.1
    if case["kind"] == "fit":
        d["model"] = _model(case, gen).to(real)
    elif case["kind"] == "step":
        d["model"] = _model(case, gen).to(cplx)
    elif case["kind"] == "sweeps":
        d["grid"] = torch.randn(case["N"], case["N"], dtype=cplx, device="cuda", generator=gen)
    return d


def _table(case):
    return lmg.Table(case["W"], case["x0"], case["Ms"], case["interp"], values=_window(case["W"], case["Ms"]))


def _n_image(case):
    return int(round(case["N"] * case["x0"]))


def _hint(case):
    return case["n_ant"] * (case["n_ant"] - 1) // 2 if case["hint"] else None


def prepare(case, seed):
    if case["kind"] == "batch":
        chans = [_inputs(c, seed + 1000 * i) for i, c in enumerate(_channels(case))]
        tables = {}
        for c in chans:
            w = c["case"]["W"]
            if w not in tables:
                tables[w] = _table(c["case"])
        batch = lmg.Batch([tables[c["case"]["W"]] for c in chans], [_n_image(c["case"]) for c in chans],
                          [c["scale"] for c in chans], [c["uv"].shape[0] for c in chans])
        batch.bin([c["uv"] for c in chans])
        vis, model = [c["vis"] for c in chans], [c["model"] for c in chans]
        return dict(case=case, batch=batch, vis=vis, model=model, image=[torch.empty_like(m) for m in model],
                    pred=[torch.empty_like(v) for v in vis])
    s = _inputs(case, seed)
    s["table"] = _table(case)
    if case["kind"] != "static":
        s["plan"] = lmg.Plan(s["table"], _n_image(case), s["scale"], s["uv"].shape[0], case["dtype"])
    if case["kind"] in ("sweeps", "fit"):
        s["plan"].bin(s["uv"], tracks=_hint(case))
    if case["kind"] == "fit":
        s["model"].requires_grad_(True)
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        state["batch"].dirty_image(state["vis"], out=state["image"])
        state["batch"].predict_vis(state["model"], out=state["pred"])
        return {"image": state["image"], "pred": state["pred"]}
    if kind == "static":
        return lmg.grid_static(state["table"], _n_image(case), state["scale"], state["uv"], state["vis"],
                               state["weights"])
    plan = state["plan"]
    if kind == "step":
        plan.bin(state["uv"], tracks=_hint(case))
        image = plan.dirty_image(state["vis"], state["weights"], case["accum"])
        return {"image": image, "pred": plan.predict_vis(state["model"])}
    if kind == "sweeps":
        grid = plan.grid(state["vis"], state["weights"], case["accum"])
        return {"grid": grid, "pred": plan.degrid(state["grid"])}
    pred = lmg.predict(state["model"], plan)
    (grad,) = torch.autograd.grad(pred, state["model"], pred.detach() - state["vis"])
    return {"pred": pred.detach(), "grad": grad}


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------
def _nvis(case):
    if case["layout"] == "disk":
        return case["nvis"]
    return case["n_ant"] * (case["n_ant"] - 1) // 2 * case["n_times"] * case["n_chan"] - case["cut"]


def work(case):
    """Positions, values, weights, images and grids that a pass takes or returns, each once;
    one multiply-add per part of each support point and the kept-field transforms."""
    if case["kind"] == "batch":
        each = [work(c) for c in _channels(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    n, N, m, W = _nvis(case), case["N"], _n_image(case), case["W"]
    c = 8 if case["dtype"] == "c64" else 16
    sums = 4.0 * W * W * n
    transform = 5.0 * N * math.log2(N) * (N + m)
    b = n * (16 + c + (c // 2 if case["weights"] else 0))
    if case["kind"] == "static":
        return {"bytes": b + N * N * c, "flops": sums}
    if case["kind"] == "sweeps":
        return {"bytes": b + n * c + 2 * N * N * c, "flops": 2 * sums}
    image = m * m * (c // 2 if case["kind"] == "fit" else c)
    return {"bytes": b + n * c + 2 * image, "flops": 2 * (sums + transform)}


# ---------------------------------------------------------------------------------------
# the same results in 64 bits, with torch alone
# ---------------------------------------------------------------------------------------
def _weights64(T, Ms, interp, s):
    """Table weights [n, W] at s in [0, 1): nearest row, linear or cubic Lagrange."""
    t = s * Ms
    if interp == "nearest":
        return T[torch.floor(t + 0.5).long()]
    if interp == "linear":
        k = torch.floor(t).long().clamp(max=Ms - 1)
        f = (t - k)[:, None]
        return (1 - f) * T[k] + f * T[k + 1]
    k = torch.floor(t - 1.0).long().clamp(0, Ms - 3)
    x = (t - k)[:, None]
    a, b, c, e = x, x - 1, x - 2, x - 3
    return (-b * c * e * T[k] / 6 + a * c * e * T[k + 1] / 2 - a * b * e * T[k + 2] / 2 + a * b * c * T[k + 3] / 6)


def _supports(case, uv, scale, T):
    """First grid index and weights of both axes for a block of positions."""
    out = []
    for ax in (0, 1):
        u = uv[:, ax] * (np.float64(case["N"]) * np.float64(scale))
        n0 = torch.ceil(u - case["W"] / 2)
        out.append((n0.long() + case["N"] // 2, _weights64(T, case["Ms"], case["interp"], n0 - (u - case["W"] / 2))))
    return out


def _blocks(n, W):
    step = max(1, int(2.0e8 // (W * W)))
    return ((k, min(n, k + step)) for k in range(0, n, step))


def _grid64(case, d, vis):
    N, W = case["N"], case["W"]
    T = torch.from_numpy(_window(W, case["Ms"])).cuda()
    G = torch.zeros(N * N, 2, dtype=torch.float64, device="cuda")
    for k0, k1 in _blocks(vis.shape[0], W):
        (x, cu), (y, cv) = _supports(case, d["uv"][k0:k1], d["scale"], T)
        v = vis[k0:k1].to(torch.complex128)
        if d["weights"] is not None:
            v = v * d["weights"][k0:k1].double()
        v = torch.view_as_real(v)
        for j in range(W):
            row = (y + j) % N * N
            vj = v * cv[:, j:j + 1]
            for i in range(W):
                G.index_add_(0, row + (x + i) % N, vj * cu[:, i:i + 1])
    return torch.view_as_complex(G).reshape(N, N)


def _degrid64(case, d, G):
    N, W = case["N"], case["W"]
    T = torch.from_numpy(_window(W, case["Ms"])).cuda()
    flat, out = G.reshape(-1), []
    for k0, k1 in _blocks(d["uv"].shape[0], W):
        (x, cu), (y, cv) = _supports(case, d["uv"][k0:k1], d["scale"], T)
        s = torch.zeros(k1 - k0, dtype=torch.complex128, device="cuda")
        for j in range(W):
            row = (y + j) % N * N
            r = torch.zeros_like(s)
            for i in range(W):
                r += cu[:, i] * flat[row + (x + i) % N]
            s += cv[:, j] * r
        out.append(s)
    return torch.cat(out)


def _factors64(case):
    """Correction h = c / D at the kept pixels with the centring sign (-1)^q, the integrals
    over s by 8-point Gauss-Legendre on each table piece (at most 4096 pieces)."""
    N, W, Ms, n = case["N"], case["W"], case["Ms"], _n_image(case)
    if Ms > 4096:
        edges = np.arange(4097) / 4096
    elif case["interp"] == "nearest":
        edges = np.concatenate([[0.0], (np.arange(Ms) + 0.5) / Ms, [1.0]])
    else:
        edges = np.arange(2 * Ms + 1) / (2 * Ms)
    gx, gw = np.polynomial.legendre.leggauss(8)
    s = ((edges[1:] + edges[:-1])[:, None] + (edges[1:] - edges[:-1])[:, None] * gx[None, :]).ravel() / 2
    w = ((edges[1:] - edges[:-1])[:, None] * gw[None, :]).ravel() / 2
    s, w = torch.from_numpy(s).cuda(), torch.from_numpy(w).cuda()
    C = _weights64(torch.from_numpy(_window(W, Ms)).cuda(), Ms, case["interp"], s)
    x = (torch.arange(n, dtype=torch.float64, device="cuda") - n // 2) / N
    j = torch.arange(W, dtype=torch.float64, device="cuda")
    h = []
    for xs in x.split(256):
        ph = 2 * math.pi * j[:, None] * xs
        re, im = C @ torch.cos(ph), C @ torch.sin(ph)
        ps = 2 * math.pi * (s - W / 2)[:, None] * xs
        h.append((w @ (re * torch.cos(ps) - im * torch.sin(ps))) / (w @ (re * re + im * im)))
    q = torch.arange(n, device="cuda") - n // 2
    return torch.cat(h) * (1 - 2 * (q % 2)), q % N


def _image64(case, d, vis):
    h, q = _factors64(case)
    F = torch.fft.ifft2(_grid64(case, d, vis), norm="forward")
    return F[q][:, q] * h[:, None] * h


def _predict64(case, d, image):
    h, q = _factors64(case)
    P = torch.zeros(case["N"], case["N"], dtype=torch.complex128, device="cuda")
    P[q[:, None], q] = image.detach().to(torch.complex128) * h[:, None] * h
    return _degrid64(case, d, torch.fft.fft2(P))


def exact(case, seed):
    if case["kind"] == "batch":
        chans = _channels(case)
        if sum(_nvis(c) * c["W"] ** 2 for c in chans) > MAX_EXACT_POINTS:
            return None
        got = {"image": [], "pred": []}
        for i, c in enumerate(chans):
            d = _inputs(c, seed + 1000 * i)
            got["image"].append(_image64(c, d, d["vis"]))
            got["pred"].append(_predict64(c, d, d["model"]))
        return got
    if _nvis(case) * case["W"] ** 2 > MAX_EXACT_POINTS:
        return None
    d = _inputs(case, seed)
    if case["kind"] == "static":
        return _grid64(case, d, d["vis"])
    if case["kind"] == "sweeps":
        return {"grid": _grid64(case, d, d["vis"]), "pred": _degrid64(case, d, d["grid"].to(torch.complex128))}
    pred = _predict64(case, d, d["model"])
    if case["kind"] == "step":
        return {"image": _image64(case, d, d["vis"]), "pred": pred}
    return {"pred": pred, "grad": _image64(case, d, pred - d["vis"]).real}
