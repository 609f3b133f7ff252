"""Measured cases: what a user of the imager has it do, through its Python API.

A case is a dict of plain values; `op` says which calls a pass makes:
  image   rick_dirty_image on device buffers (bin, grid, transform, reduce)
  graph   the same path captured once as a CUDA graph and launched again
  host    rick_dirty_image_host on page-locked host buffers
  planes  the three separate calls: rick_grid, rick_fft_wplanes,
          rick_phase_correct_reduce (every plane whole)
  predict rick_predict: a model image to visibilities
  lgrid   the learned kernel: bake the table, load it, rick_grid
  train   one training step of the learned kernel (LearnedKernel.train)

Observations are earth-rotation tracks of two array layouts (64 antennas within
8 km, 856-1712 MHz; 60 stations within 100 km, half in a 2 km core, 120-168 MHz)
or visibilities spread over a disk of the mesh; visibilities are a few point
sources under noise, weights U[0.5, 1.5], 5 % (8 km) or up to 40 % per channel
(100 km) flagged.  Kaiser-Bessel images are taken on a mesh padded by 2 and
Gaussian ones on the bare mesh: on the bare mesh the Kaiser-Bessel taper reaches
1e-5 at the edge, where the image is rounding noise times 1e10.

`exact` is the same method in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

from paper_2601_19714_gb300 import learned, rick

C_LIGHT = 299_792_458.0
# support S: Kaiser-Bessel shape of a mesh without oversampling; Gaussian 1e-3 at the edge
KB_BETA = {s: math.pi * math.sqrt(0.25 * s * s - 0.8) for s in range(4, 9)}
GAUSS_SIGMA = {s: 0.5 * s / math.sqrt(2.0 * math.log(1e3)) for s in range(4, 9)}

BASE = dict(op="image", layout="meerkat", N=1024, pad=1, Nw=16, S=7, kernel="gauss", C=1, rows=100_000,
            fov_deg=1.5, fold=True, w_support=0, weighting="natural", robust=0.0, budget_mb=0,
            lattice=0, hidden=0, batch=0)


def listed():
    return [
        # the smallest call: one channel, 20 k visibilities, 256^2 x 8 planes (quick looks, self-calibration steps)
        dict(BASE, name="image_tiny", layout="disk", N=256, Nw=8, rows=20_000, fov_deg=2.0, fold=False),
        # a short scan imaged with Briggs weights; a ragged row count
        dict(BASE, name="image_briggs", N=1024, pad=2, S=8, kernel="kb", C=4, rows=200_003, fov_deg=0.375,
             weighting="briggs"),
        # the ordinary spectral cube: 8 h track, 16 channels, 4096^2 mesh, 32 planes
        dict(BASE, name="image_meerkat", N=2048, pad=2, Nw=32, S=8, kernel="kb", C=16, rows=2_016_000, fov_deg=0.75),
        # wide-field, uneven channels, dense core, plane groups streamed under a memory budget, one graph
        dict(BASE, name="image_lofar", op="graph", layout="lofar", N=4096, pad=2, Nw=40, S=8, kernel="kb", C=6,
             rows=1_274_400, fov_deg=2.5, budget_mb=24_000),
        # the largest image: 16384^2, 32 planes, one channel at a time
        dict(BASE, name="image_large", N=16384, Nw=32, C=2, rows=5_846_400, fov_deg=1.5, budget_mb=36_000),
        # the same job from page-locked host buffers, copies both ways inside the call
        dict(BASE, name="image_host", op="host", N=2048, pad=2, Nw=32, S=8, kernel="kb", C=4, rows=504_001,
             fov_deg=0.75),
        # improved w-stacking: each visibility on 4 planes
        dict(BASE, name="image_wkernel", N=2048, pad=2, Nw=20, S=8, kernel="kb", C=4, rows=1_008_000, fov_deg=0.75,
             w_support=4),
        # a program that wants the planes themselves: grid, transform and reduce as separate calls
        dict(BASE, name="planes_4096", op="planes", N=4096, Nw=16, rows=504_000, fold=False),
        # the other half of a major cycle: model image to 16 M visibilities
        dict(BASE, name="predict_meerkat", op="predict", N=4096, Nw=32, S=8, kernel="kb", C=8, rows=2_016_000),
        # a small prediction with many planes unreached and an odd row count
        dict(BASE, name="predict_small", op="predict", layout="disk", N=512, Nw=9, rows=30_011, fov_deg=2.0, fold=False),
        # gridding with the learned kernel (table baked from the network, 2 M visibilities)
        dict(BASE, name="learned_grid", op="lgrid", layout="disk", N=2048, S=4, kernel="table", rows=2_000_000,
             fov_deg=2.0, fold=False, lattice=32, hidden=64),
        # one training step of the learned kernel on a batch of fields
        dict(BASE, name="learned_train", op="train", layout="disk", N=2048, S=4, kernel="table", rows=2_000_000,
             fov_deg=2.0, fold=False, lattice=32, hidden=64, batch=4),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    op = rng.choice(["image"] * 5 + ["graph", "host", "planes", "predict", "predict", "predict", "lgrid", "train"])
    if op in ("lgrid", "train"):
        N = 2 ** rng.randint(8, 11)
        c = dict(BASE, op=op, layout="disk", N=N, S=4, kernel="table", fov_deg=2.0, fold=False,
                 rows=logint(2_000, min(2_000_000, 4 * N * N)) | 1, Nw=rng.randint(2, 16))
        c.update(lattice=rng.choice([8, 16, 24, 32]), hidden=rng.choice([16, 32, 64]),
                 batch=rng.randint(1, 4) if op == "train" else 0)
        return c
    mesh = 2 ** rng.choice([8, 9, 10, 11, 11, 12, 12, 13, 13])
    pad = rng.choice([1, 2])
    # at most about 2 visibilities a cell and channel
    c = dict(BASE, op=op, rows=logint(2_000, min(2_000_000, 2 * mesh * mesh)) | 1)
    c.update(N=mesh // pad, pad=pad, Nw=logint(1, min(48, 2 ** 30 // (mesh * mesh))), layout=rng.choice(["meerkat", "lofar", "disk"]),
             fold=rng.random() < 0.6, kernel="kb" if pad == 2 else "gauss",
             S=rng.choice([4, 5, 6, 7, 8, 8]) if pad == 2 else rng.choice([5, 6, 7, 7]))
    if op != "predict":
        c["weighting"] = rng.choice(["natural"] * 4 + ["uniform", "briggs"])
        c["robust"] = rng.choice([-1.0, 0.0, 0.5])
    if c["layout"] == "disk":
        c["fov_deg"] = rng.choice([1.0, 2.0, 3.0])
        c["C"] = 1
    else:
        # field of view from the part of the mesh that the longest baseline reaches
        far = 8_000 * 1.6e9 / C_LIGHT if c["layout"] == "meerkat" else 100_000 * 1.65e8 / C_LIGHT
        c["fov_deg"] = round(math.degrees(rng.uniform(0.15, 1.0) * 0.5 * c["N"] / far), 4)
        sw = rng.choice([2, 4, 6])
        # a w-kernel needs planes close enough for the field
        turn = 2.0 * min(20_000.0 if c["layout"] == "lofar" else 46_000.0, far) / c["Nw"] * math.radians(c["fov_deg"]) ** 2 / 4.0
        if rng.random() < 0.5 and c["Nw"] >= 8 and math.pi * sw * turn < 8.0:
            c["w_support"] = sw
        planes = c["Nw"] + c["w_support"] if op == "planes" or not c["fold"] else (c["Nw"] + c["w_support"] + 1) // 2
        c["C"] = logint(1, max(1, min(16, 2 ** 30 // (planes * mesh * mesh),
                                      2 ** 22 // (c["rows"] * max(1, c["w_support"])))))
    if rng.random() < 0.3:
        c["budget_mb"] = max(16, int(8e-6 * mesh * mesh * logint(1, 64)))
    return c


# ---- inputs ---------------------------------------------------------------------


def _rand(seed, stream):
    g = torch.Generator("cuda")
    g.manual_seed(seed * 64 + stream)
    return lambda *n: torch.rand(*n, generator=g, device="cuda", dtype=torch.float64)


def _observation(case, seed):
    """uvw [rows][3] in wavelengths at the first channel, chan_scale, w extent."""
    r = _rand(seed, 1)
    rows, C, fov = case["rows"], case["C"], math.radians(case["fov_deg"])
    if case["layout"] == "disk":
        rad, t = 0.45 * case["N"] / fov * r(rows).sqrt(), 2.0 * math.pi * r(rows)
        uvw = torch.stack([rad * t.cos(), rad * t.sin(), 200.0 * (2.0 * r(rows) - 1.0)], 1)
        return uvw.contiguous(), torch.ones(1, dtype=torch.float64, device="cuda"), 200.0
    far = case["layout"] == "lofar"
    n, size, lat = (60, 50_000.0, 52.9) if far else (64, 4_000.0, -30.7)
    rad, t = size * r(n).sqrt(), 2.0 * math.pi * r(n)
    if far:
        rad[: n // 2] *= 0.02
    e, nn, up = rad * t.cos(), rad * t.sin(), 10.0 * (r(n) - 0.5)
    i, j = torch.triu_indices(n, n, 1, device="cuda")
    E, Nn, U = e[j] - e[i], nn[j] - nn[i], up[j] - up[i]
    steps = -(-rows // E.numel())
    s, c = math.sin(math.radians(lat)), math.cos(math.radians(lat))
    X, Y, Z = -s * Nn + c * U, E, c * Nn + s * U
    half = 4.0 * math.pi / 12.0
    H = torch.linspace(-half, half, steps, dtype=torch.float64, device="cuda")[:, None]
    sH, cH = H.sin(), H.cos()
    uvw = torch.stack([sH * X + cH * Y, -s * cH * X + s * sH * Y + c * Z, c * cH * X - c * sH * Y + s * Z], -1)
    lo, hi = (120e6, 168e6) if far else (856e6, 1712e6)
    f = lo + (torch.arange(C, dtype=torch.float64, device="cuda") + 0.5) * (hi - lo) / C
    uvw = (uvw.reshape(-1, 3)[:rows] * (f[0] / C_LIGHT)).contiguous()
    scale = (f / f[0]).contiguous()
    w = float(uvw[:, 2].abs().max() * scale[-1])
    return uvw, scale, min(w, 20_000.0) if far else w


def _sources(case, seed, n=4):
    """(l, m, flux) rows inside the central 70 % of the field, on the host."""
    g = np.random.Generator(np.random.Philox(key=[seed, 7]))
    lm = (g.random((n, 2)) - 0.5) * 0.7 * math.radians(case["fov_deg"])
    return np.concatenate([lm, 0.1 * (0.03 + g.random((n, 1))) ** (-1.0 / 1.5)], 1)


def _inputs(case, seed):
    uvw, scale, w = _observation(case, seed)
    r = _rand(seed, 2)
    rows, C = case["rows"], case["C"]
    vis = torch.empty(rows, C, dtype=torch.complex64, device="cuda")
    torch.view_as_real(vis).copy_(0.7 * torch.randn(rows, C, 2, device="cuda", generator=torch.Generator("cuda").manual_seed(seed)))
    for l, m, a in _sources(case, seed):
        n = math.sqrt(1.0 - l * l - m * m)
        turn = uvw @ torch.tensor([l, m, n - 1.0], dtype=torch.float64, device="cuda")
        for c in range(C):
            t = turn * scale[c]
            ph = ((t - t.round()) * (-2.0 * math.pi)).float()
            vis[:, c] += torch.polar(torch.full_like(ph, a / n), ph)
    weight = (0.5 + r(rows, C)).float()
    if case["layout"] == "disk":
        flag = None
    else:
        share = 0.05 if case["layout"] == "meerkat" else 0.4 * r(C)
        flag = (r(rows, C) < share).to(torch.uint8)
        if case["layout"] == "lofar":
            flag |= ((uvw[:, 2:3] * scale).abs() > w).to(torch.uint8)
    return dict(uvw=uvw, chan_scale=scale, vis=vis, weight=weight, flag=flag), w


def _config(case, w):
    param = {"kb": KB_BETA, "table": KB_BETA, "gauss": GAUSS_SIGMA}[case["kernel"]][case["S"]]
    return rick.Config(N=case["N"], n_wplanes=case["Nw"], support=case["S"], n_channels=case["C"],
                       fov_rad=math.radians(case["fov_deg"]), w_min=-w, w_max=w, kernel=case["kernel"],
                       kernel_param=param, hermitian_fold=case["fold"], w_support=case["w_support"],
                       w_kernel_param=8.0 if case["w_support"] else 0.0, weighting=case["weighting"],
                       robust=case["robust"], grid_size=case["N"] * case["pad"] if case["pad"] > 1 else 0,
                       grid_budget_bytes=case["budget_mb"] * 1_000_000)


def _network(case, seed):
    """A network part-way through training: small corrections to the taps."""
    k = learned.LearnedKernel(case["Nw"], case["hidden"], case["lattice"], seed % 65536, zero_output=False)
    k.params[-16 * (case["hidden"] + 1):].mul_(0.05)
    return k


def prepare(case, seed):
    data, w = _inputs(case, seed)
    cfg = _config(case, w)
    C, N, Ng, P, rows = case["C"], cfg.N, cfg.Ng, cfg.stored_planes, case["rows"]
    s = dict(case=case, cfg=cfg, data=data, rows=rows)
    new = lambda *n, t=torch.float32: torch.zeros(*n, dtype=t, device="cuda")  # noqa: E731
    if case["op"] == "train":
        s["net"] = _network(case, seed)
        s["learn"] = rick.Learn(cfg, case["lattice"], data["uvw"], data["weight"].reshape(-1))
        s["seed"] = 1_000_000 + 1000 * (seed % 100_000)
        return s
    s["plan"] = plan = rick.Plan(cfg)
    s["wsum"], s["counts"] = new(C, t=torch.float64), new(2, t=torch.int64)
    if case["op"] == "host":
        s["data"] = {k: None if v is None else v.cpu().pin_memory() for k, v in data.items()}
        s["image"] = torch.empty(C, N, N, pin_memory=True)
        s["wsum"], s["counts"] = torch.zeros(C, dtype=torch.float64).pin_memory(), torch.zeros(2, dtype=torch.int64).pin_memory()
        return s
    plan.reserve(rows)
    if case["op"] == "predict":
        # a CLEAN-like model: components inside the central 70 % of the field
        g = np.random.Generator(np.random.Philox(key=[seed, 8]))
        at = torch.from_numpy((N * (0.5 + 0.7 * (g.random((C, 200, 2)) - 0.5))).astype(np.int64)).cuda()
        s["model"] = new(C, N, N)
        s["model"][torch.arange(C, device="cuda")[:, None], at[..., 0], at[..., 1]] = torch.from_numpy(g.exponential(0.3, (C, 200))).float().cuda()
        s["out"] = new(rows, C, t=torch.complex64)
        return s
    if case["op"] in ("planes", "lgrid"):
        s["grids"] = new(C, P, Ng, Ng, t=torch.complex64)
    if case["op"] == "lgrid":
        s["net"] = _network(case, seed)
        return s
    s["image"] = new(C, N, N)
    if case["op"] == "graph":
        d = data
        s["graph"] = plan.capture_graph(d["uvw"], d["chan_scale"], d["vis"], d["weight"], d["flag"], rows, None,
                                        s["wsum"], s["image"], s["counts"])
    return s


def run(s):
    d, plan, cfg, op = s["data"], s.get("plan"), s["cfg"], s["case"]["op"]
    args = (d["uvw"], d["chan_scale"], d["vis"], d["weight"], d["flag"], s["rows"])
    C, P = cfg.n_channels, cfg.stored_planes
    if op == "image":
        s["image"].zero_()
        plan.dirty_image(*args, s["image"], None, s["wsum"], s["counts"])
    elif op == "graph":
        s["graph"].launch()
    elif op == "host":
        plan.dirty_image_host(*args[:5], s["image"], s["wsum"], s["counts"])
    elif op == "planes":
        s["image"].zero_()
        plan.grid(*args, 0, P, s["grids"], s["wsum"], s["counts"])
        plan.fft_wplanes(s["grids"], C * P)
        plan.phase_correct_reduce(s["grids"], 0, C, 0, P, s["wsum"], s["image"])
        return dict(image=s["image"], planes=s["grids"], wsum=s["wsum"], counts=s["counts"])
    elif op == "predict":
        plan.predict(d["uvw"], d["chan_scale"], d["weight"], d["flag"], s["rows"], s["model"], s["out"], s["counts"])
        return dict(vis=s["out"], counts=s["counts"])
    elif op == "lgrid":
        k = s["net"]
        plan.set_kernel_table(k.bake(), k.L)
        plan.grid(*args, 0, P, s["grids"], s["wsum"], s["counts"])
        return dict(table=k.table, planes=s["grids"], wsum=s["wsum"], counts=s["counts"])
    else:
        k = s["net"]
        k.train(s["learn"], 1, 1e-5, s["case"]["batch"], field_seed0=s["seed"], inner=0.4)
        return dict(params=k.params, grad=k.grad, table_grad=k.table_grad, loss=k.loss)
    return dict(image=s["image"], wsum=s["wsum"], counts=s["counts"])


def work(case):
    C, N, Ng, S, rows = case["C"], case["N"], case["N"] * case["pad"], case["S"], case["rows"]
    total = case["Nw"] + case["w_support"]
    planes = (total + 1) // 2 if case["fold"] else total
    sw = max(1, case["w_support"])
    vis = rows * C
    flops = 4.0 * S * S * sw * vis
    image = 4 * C * N * N
    dft = 5.0 * N * Ng * math.log2(Ng) * C * planes   # one transform per image row and plane
    data = 24 * rows + 8 * C + (12 + (case["layout"] != "disk")) * vis
    if case["op"] == "train":
        table = 64 * case["Nw"] * (case["lattice"] + 1) ** 2
        return dict(bytes=28 * rows + 2 * table, flops=case["batch"] * rows * 64.0 * 2 * 150)
    if case["op"] == "lgrid":
        return dict(bytes=data + 8 * C * planes * Ng * Ng + 64 * case["Nw"] * (case["lattice"] + 1) ** 2, flops=flops)
    if case["op"] == "planes":
        return dict(bytes=data + 8 * C * planes * Ng * Ng + image, flops=flops + 2 * dft)
    if case["op"] == "predict":
        return dict(bytes=24 * rows + 8 * C + 5 * vis + image + 8 * vis, flops=flops + dft)
    return dict(bytes=data + image, flops=flops + dft)


# ---- the same in 64 bits ------------------------------------------------------------


def _kernel(case, s):
    """The gridding kernel at distances s (float64 tensor, cells)."""
    S = case["S"]
    if case["kernel"] == "gauss":
        g = torch.exp(-0.5 * (s / GAUSS_SIGMA[S]) ** 2)
    else:
        b = KB_BETA[S]
        g = torch.i0(b * (1.0 - (2.0 * s / S) ** 2).clamp_min(0.0).sqrt()) / float(np.i0(b))
    return torch.where(s.abs() <= 0.5 * S, g, torch.zeros_like(g))


def _taper(case):
    S, N, Ng = case["S"], case["N"], case["N"] * case["pad"]
    x, wt = np.polynomial.legendre.leggauss(24)
    s = torch.from_numpy((np.arange(S)[:, None] - 0.5 * S + 0.5 + 0.5 * x).ravel()).cuda()
    g = _kernel(case, s) * torch.from_numpy(np.tile(0.5 * wt, S)).cuda()
    p = torch.arange(N, device="cuda", dtype=torch.float64) - N // 2
    return (torch.cos(2.0 * math.pi / Ng * p[:, None] * s) * g).sum(1)


def _place(case, cfg, d, c, w):
    """Channel c's visibilities on the mesh: indices, first cells, fractions, planes, plane weights [n][Sw]."""
    S, Ng, Nw, sw = case["S"], cfg.Ng, case["Nw"], case["w_support"]
    ok = (d["weight"][:, c] != 0) & ((d["flag"][:, c] == 0) if d["flag"] is not None else True)
    uvw = d["uvw"] * d["chan_scale"][c]
    xy = uvw[:, :2] * (cfg.fov_rad * Ng / cfg.N) + 0.5 * Ng
    sx = xy - 0.5 * S
    fl = sx.floor()
    ok &= ((fl >= -1) & (fl + S <= Ng - 1)).all(1)
    at = ok.nonzero()[:, 0]
    first, frac, uvw = fl[at].long() + 1, (sx - fl)[at], uvw[at]
    if Nw == 1 and not sw:
        return at, first, frac, torch.zeros_like(first[:, :1]), torch.ones_like(frac[:, :1])
    t = (uvw[:, 2] + w) * (Nw / (2.0 * w))
    if not sw:
        return at, first, frac, t.floor().clamp(0, Nw - 1).long()[:, None], torch.ones_like(frac[:, :1])
    z = (t - 0.5).clamp(-0.5, Nw - 0.5) - 0.5 * sw
    a = torch.arange(sw, device="cuda")
    dist = a + 1 - 0.5 * sw - (z - z.floor())[:, None]
    g = torch.i0(8.0 * (1.0 - (2.0 * dist / sw) ** 2).clamp_min(0.0).sqrt()) / float(np.i0(8.0))
    return at, first, frac, (z.floor().long() + 1 + sw // 2)[:, None] + a, g


def _weights(case, cfg, d, c, at):
    W = d["weight"][at, c].double()
    if case["weighting"] == "natural":
        return W
    N = cfg.N
    xy = d["uvw"][at][:, :2] * d["chan_scale"][c] * cfg.fov_rad + 0.5 * N
    i, j = (xy + 0.5).floor().long().remainder(N).unbind(1)
    D = torch.zeros(N * N, dtype=torch.float64, device="cuda")
    D.index_add_(0, j * N + i, W).index_add_(0, (-j).remainder(N) * N + (-i).remainder(N), W)
    if case["weighting"] == "uniform":
        return W / D[j * N + i]
    f2 = (5.0 * 10.0 ** -case["robust"]) ** 2 * D.sum() / (D * D).sum()
    return W / (1.0 + f2 * D[j * N + i])


def _cells(case, first, frac, Ng):
    """Flat cells [n][S*S] of the footprints and the separable taps, checkerboard included."""
    a = torch.arange(case["S"], device="cuda")
    g = _kernel(case, a + 1 - 0.5 * case["S"] - frac[:, :, None])
    g = g * (1 - 2 * ((first[:, :, None] + a) & 1))
    cell = (first[:, 1, None, None] + a[:, None]) * Ng + first[:, 0, None, None] + a
    return cell.reshape(len(first), -1), (g[:, 1, :, None] * g[:, 0, None, :]).reshape(len(first), -1)


def _field(case, cfg):
    """n and n - 1 of every pixel."""
    x = (torch.arange(cfg.N, device="cuda", dtype=torch.float64) - cfg.N // 2) * (cfg.fov_rad / cfg.N)
    r2 = x[:, None] ** 2 + x ** 2
    n = (1.0 - r2).sqrt()
    return n, -r2 / (1.0 + n)


def _screen(case, w, k, delta):
    Nw, sw = case["Nw"], case["w_support"]
    wk = -w + (k - sw // 2 + 0.5) * (2.0 * w / Nw) if Nw > 1 else 0.0
    t = wk * delta
    t = 2.0 * math.pi * (t - t.round())
    return torch.complex(t.cos(), t.sin())


def _scale(case, cfg, w, delta):
    """1 / (C(p) C(q) C_w) of every pixel."""
    C = _taper(case)
    out = 1.0 / (C[:, None] * C)
    if case["w_support"]:
        nu = math.pi * case["w_support"] * delta * (2.0 * w / case["Nw"])
        r = (64.0 - nu * nu).sqrt()
        out = out * r * float(np.i0(8.0)) / (case["w_support"] * torch.sinh(r))
    return out


def _network64(case, params):
    """The table of corrections [Nw][L+1][L+1][16] from parameters (float64, may require grad)."""
    H, L, Nw = case["hidden"], case["lattice"], case["Nw"]
    W1, b1, W2, b2, W3, b3 = params.split([3 * H, H, H * H, H, 16 * H, 16])
    x = torch.arange(L + 1, device="cuda", dtype=torch.float64) / L
    k = torch.arange(Nw, device="cuda", dtype=torch.float64)
    k = (2.0 * k - (Nw - 1)) / (Nw - 1)
    at = torch.stack(torch.meshgrid(k, x, x, indexing="ij")[::-1], -1).reshape(-1, 3)
    act = lambda v: torch.nn.functional.gelu(v, approximate="tanh")  # noqa: E731
    z = act(at @ W1.view(H, 3).T + b1)
    return act(z @ W2.view(H, H).T + b2) @ W3.view(16, H).T + b3


def _lattice(case, frac, k):
    """Rows of the table around each fraction [n][4] and their bilinear weights."""
    L = case["lattice"]
    at = (frac * L).long().clamp_max(L - 1)
    x, y = (frac * L - at).unbind(1)
    row = (k * (L + 1) + at[:, 1]) * (L + 1) + at[:, 0]
    return (torch.stack([row, row + 1, row + L + 1, row + L + 2], 1),
            torch.stack([(1 - x) * (1 - y), x * (1 - y), (1 - x) * y, x * y], 1))


def _exact_train(case, seed):
    d, w = _inputs(case, seed)
    cfg, net = _config(case, w), _network(case, seed)
    N, fov = cfg.N, cfg.fov_rad
    at, first, frac, k, _ = _place(case, cfg, d, 0, w)
    k, W, uvw = k[:, 0], d["weight"][at, 0].double(), d["uvw"][at]
    params = net.params.double().requires_grad_()
    table = _network64(case, params)
    flat = table.detach()
    grad, loss = torch.zeros_like(flat), None
    taper = _taper(case)
    for b in range(case["batch"]):
        fs = 1_000_000 + 1000 * (seed % 100_000) + b
        src = learned.training_field(fs, N, inner=0.4)
        probes = torch.from_numpy(learned.field_probes(fs, N, src).astype(np.int64)).cuda()
        src = torch.from_numpy(src).cuda()
        # the library takes source rows as 32-bit numbers
        src = src.float().double()
        lm = (src[:, :2] - N // 2) * (fov / N)
        n = (1.0 - (lm * lm).sum(1)).sqrt()
        V = torch.zeros(len(at), dtype=torch.complex128, device="cuda")
        for s in range(len(src)):
            t = uvw[:, 0] * lm[s, 0] + uvw[:, 1] * lm[s, 1] + uvw[:, 2] * (n[s] - 1.0)
            t = -2.0 * math.pi * (t - t.round())
            V += src[s, 2] / n[s] * torch.complex(t.cos(), t.sin())
        WV = W * V
        pc = (probes - N // 2).double()
        plm = pc * (fov / N)
        pn = (1.0 - (plm * plm).sum(1)).sqrt()
        scale = pn / (taper[probes[:, 0]] * taper[probes[:, 1]])
        ph = torch.stack([_screen(case, w, q, pn - 1.0) for q in range(case["Nw"])])
        turns = torch.arange(N, device="cuda", dtype=torch.float64) * (2.0 * math.pi / N)
        unit = torch.complex(turns.cos(), turns.sin())
        a = torch.arange(4, device="cuda")

        def terms(j0, j1):
            """W V exp(..) of the tap cells at the probes: [n][probes] and the two axes [n][probes][4]."""
            f = first[j0:j1]
            E = [unit[((f[:, x, None, None] + a - N // 2) * (probes[:, x, None] - N // 2)).remainder(N)] for x in (0, 1)]
            return scale * WV[j0:j1, None] * ph[k[j0:j1]], E[0], E[1]

        def taps(j0, j1):
            rows, bl = _lattice(case, frac[j0:j1], k[j0:j1])
            g = _kernel(case, a + 1 - 2.0 - frac[j0:j1, :, None])
            return (g[:, 1, :, None] * g[:, 0, None, :]) + (flat[rows] * bl[..., None]).sum(1).view(-1, 4, 4)

        step = 1 << 16
        I, D = torch.zeros_like(pn), torch.zeros_like(pn)
        for j0 in range(0, len(at), step):
            j1 = min(len(at), j0 + step)
            c, Ex, Ey = terms(j0, j1)
            inner = torch.einsum("nba,npa->npb", taps(j0, j1).to(Ex.dtype), Ex)
            I += (c * (inner * Ey).sum(2)).real.sum(0)
            t = uvw[j0:j1, :1] * plm[:, 0] + uvw[j0:j1, 1:2] * plm[:, 1] + uvw[j0:j1, 2:] * (pn - 1.0)
            t = 2.0 * math.pi * (t - t.round())
            D += (pn * WV[j0:j1, None] * torch.complex(t.cos(), t.sin())).real.sum(0)
        I, D = I / W.sum(), D / W.sum()
        loss = ((I - D) ** 2).sum() / (D ** 2).sum()
        ge = 2.0 * (I - D) / (D ** 2).sum() / W.sum() / case["batch"]
        for j0 in range(0, len(at), step):
            j1 = min(len(at), j0 + step)
            c, Ex, Ey = terms(j0, j1)
            gt = torch.einsum("npb,npa->nba", (ge * c)[..., None] * Ey, Ex).real.reshape(-1, 16)
            rows, bl = _lattice(case, frac[j0:j1], k[j0:j1])
            for q in range(4):
                grad.index_add_(0, rows[:, q], bl[:, q, None] * gt)
    table.backward(grad)
    g = params.grad
    # the first Adam step of one update (its rate is the schedule's first)
    new = net.params.double() - 1e-5 * g / (g.abs() + 1e-8)
    return dict(params=new, grad=g, table_grad=grad, loss=loss.reshape(1))


def exact(case, seed):
    if case["op"] == "train":
        return _exact_train(case, seed)
    d, w = _inputs(case, seed)
    cfg = _config(case, w)
    C, N, Ng, Nt = case["C"], cfg.N, cfg.Ng, cfg.planes_total
    off = (Ng - N) // 2
    if case["op"] == "lgrid":
        table = _network64(case, _network(case, seed).params.double())
        at, first, frac, k, _ = _place(case, cfg, d, 0, w)
        W = d["weight"][at, 0].double()
        cell, g = _cells(case, first, frac, Ng)
        sign = 1 - 2 * ((cell // Ng + cell % Ng) & 1)
        rows, bl = _lattice(case, frac, k[:, 0])
        g = g + sign * (table[rows] * bl[..., None]).sum(1)
        G = torch.zeros(Nt * Ng * Ng, 2, dtype=torch.float64, device="cuda")
        V = torch.view_as_real(d["vis"][at, 0].to(torch.complex128)) * W[:, None]
        for q in range(16):
            G.index_add_(0, k[:, 0] * (Ng * Ng) + cell[:, q], V * g[:, q, None])
        planes = torch.view_as_complex(G).view(1, Nt, Ng, Ng)
        return dict(table=table, planes=planes, wsum=W.sum().reshape(1), counts=None)
    n, delta = _field(case, cfg)
    scale = _scale(case, cfg, w, delta)
    p = torch.arange(N, device="cuda") + off
    board = (1.0 - 2.0 * ((p[:, None] + p) & 1).double())
    if case["op"] == "predict":
        model = prepare(case, seed)["model"]
        out = torch.zeros(case["rows"], C, dtype=torch.complex128, device="cuda")
        for c in range(C):
            at, first, frac, k, gw = _place(case, cfg, d, c, w)
            J = model[c].double() * board * scale / n
            for q in torch.unique(k).tolist():
                M = torch.zeros(Ng, Ng, dtype=torch.complex128, device="cuda")
                M[off:off + N, off:off + N] = J * _screen(case, w, q, delta).conj()
                F = torch.fft.fft2(M).reshape(-1)
                r, s = (k == q).nonzero(as_tuple=True)
                cell, g = _cells(case, first[r], frac[r], Ng)
                out[at[r], c] += gw[r, s] * (F[cell] * g).sum(1)
        return dict(vis=out, counts=None)
    image = torch.zeros(C, N, N, dtype=torch.float64, device="cuda")
    wsum = torch.zeros(C, dtype=torch.float64, device="cuda")
    planes = torch.zeros(C, Nt, Ng, Ng, dtype=torch.complex128, device="cuda") if case["op"] == "planes" and not case["fold"] else None
    for c in range(C):
        at, first, frac, k, gw = _place(case, cfg, d, c, w)
        W = _weights(case, cfg, d, c, at)
        wsum[c] = W.sum()
        V = torch.view_as_real(d["vis"][at, c].to(torch.complex128)) * W[:, None]
        for q in torch.unique(k).tolist():
            r, s = (k == q).nonzero(as_tuple=True)
            G = torch.zeros(Ng * Ng, 2, dtype=torch.float64, device="cuda")
            for b in range(0, len(r), 1 << 18):
                rb, sb = r[b:b + (1 << 18)], s[b:b + (1 << 18)]
                cell, g = _cells(case, first[rb], frac[rb], Ng)
                G.index_add_(0, cell.reshape(-1), ((gw[rb, sb, None] * g)[..., None] * V[rb, None]).reshape(-1, 2))
            F = torch.fft.ifft2(torch.view_as_complex(G).view(Ng, Ng), norm="forward")
            del G
            if planes is not None:
                planes[c, q] = F
            F = F[off:off + N, off:off + N]
            e = _screen(case, w, q, delta)
            image[c] += F.real * e.real - F.imag * e.imag
            del F, e
        image[c] *= board * n * scale / wsum[c]
    out = dict(image=image, wsum=wsum, counts=None)
    if case["op"] == "planes":
        out["planes"] = planes
    return out
