"""The work that a user of this library has it do, as cases that can be timed
and checked: training steps from a few hundred Gaussians on small images to
the benchmark workload, projections, validation passes, the CTF step on its
own, a training iteration with its optimiser, the density query, the Fourier
shell correlation of two half maps, and nearest neighbours.

Inputs follow the recipe of the repository's synthetic workloads (clustered
centres, log-uniform scales, Haar-random views, 300 kV CTFs, noise images at
SNR 0.1), drawn on the GPU from the seed.  ``exact`` is the mathematics of
each path in float64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_25075_gb300 import binding
from paper_2509_25075_gb300 import train

NPAR = 11
APIX = float(np.float32(1.2))  # the library takes the pixel size as float32
SIDES = (16, 32, 48, 64, 96, 128, 144, 192, 256, 288, 384, 432, 512, 576, 768)  # 2^a 3^b, multiples of 16
NARROW = (0.5, 3.0)  # smallest and largest scale, pixels
WIDE = (0.3, 12.0)   # heavy-tailed scales: many needles, few clusters
TRAIN_LR = (0.05, 0.01, 0.002, 0.02)


def _case(kind, name=None, **kw):
    c = dict(kind=kind, d=64, M=2000, B=32, wide=False, tau=True, norm=0, zsort=1, norot=False, iso=False,
             array=False, tune=False, k=1)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call of the hot path: a CPU-sized problem (workload A1)
        # trained on the GPU, or the first levels of a coarse-to-fine run;
        # launches and latency count
        _case("step", "step_small", d=64, M=2000, B=32),
        # a mid-sized fit, large batch of small images (workload A2), its
        # rasteriser configurations picked by the autotuner as the benchmark
        # does
        _case("step", "step_mid", d=128, M=20000, B=256, tune=True),
        # heavy-tailed, elongated Gaussians in few clusters (the recipe of
        # workload A4) at the training loop's default batch of 64: tile
        # imbalance and the general binning path
        _case("step", "step_wide", d=128, M=50000, B=64, wide=True),
        # the benchmark workload A5: large images, half a million Gaussians
        _case("step", "step_large", d=384, M=500000, B=16, tune=True),
        # library defaults (tau 0: every pair counts) on a ragged problem,
        # projection only, line-integral amplitudes: rendering a few views
        _case("project", "project_every_pair", d=64, M=1999, B=9, tau=False, norm=1),
        # validation: predictions and loss of held-out images, no gradient
        # (workload A3)
        _case("predict", "predict", d=256, M=100000, B=64),
        # the CTF step alone with measured transfer arrays, odd side and
        # batch, every output wanted: a caller with a renderer of its own
        _case("ctf", "ctf_array", d=144, M=1, B=50, array=True),
        # one iteration of the training loop through Trainer.step: batch
        # gather, step, optimiser
        _case("train", "train_iteration", d=128, M=20000, B=64),
        # the density map of a fitted model on its voxel grid, for viewing or
        # for the FSC (the grid of workload A3)
        _case("query", "query_map", d=256, M=100000, B=64),
        # gold-standard FSC of two half maps
        _case("fsc", "fsc_half_maps", d=256, M=1, B=1),
        # nearest-neighbour scales of the isotropic ablation, every step
        _case("nearest", "nearest", d=384, M=500000, B=1),
        # the optimiser alone at the benchmark's size
        _case("adam", "adam", d=384, M=500000, B=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["project"] * 2 + ["predict"] * 2 + ["ctf"] * 2 + ["train"] * 2 +
                      ["query", "fsc", "nearest", "adam"])
    c = _case(kind)
    c["zsort"] = 0 if rng.random() < 0.15 else 1
    c["norm"] = 1 if rng.random() < 0.25 else 0
    c["norot"] = rng.random() < 0.1
    c["iso"] = rng.random() < 0.1
    if kind in ("step", "project", "predict", "train"):
        c["wide"] = rng.random() < 0.25 and kind != "train"
        c["d"] = rng.choice([s for s in SIDES if 32 <= s <= (192 if c["wide"] else 384)])
        c["M"] = _log_int(rng, 300, 50000 if c["wide"] else 500000)
        most = (3.2e6 if c["wide"] else 8e6) / c["M"]
        c["B"] = _log_int(rng, 2, max(2, min(256, most, 4.2e6 / c["d"] ** 2)))
        c["array"] = rng.random() < 0.3 and kind in ("step", "predict")
        c["tune"] = kind == "step" and rng.random() < 0.3
        if kind == "project" and rng.random() < 0.5:
            # every pair: a tile list entry for each (view, Gaussian, tile)
            c.update(tau=False, wide=False, d=rng.choice([32, 48, 64, 96]), M=_log_int(rng, 300, 4000),
                     B=_log_int(rng, 1, 16))
        most = work(_case("step", d=384, M=500000, B=16))["flops"]
        while work(dict(c, kind="step"))["flops"] > most:  # no dearer than the largest listed case
            c["B" if c["B"] > 2 else "M"] //= 2
    elif kind == "ctf":
        c["d"] = rng.choice(SIDES)
        c["B"] = _log_int(rng, max(2, 130000 // c["d"] ** 2), max(3, 8e6 / c["d"] ** 2))
        c.update(M=1, array=rng.random() < 0.5)
    elif kind == "query":
        c["d"] = rng.choice([64, 96, 128, 144, 192, 256])
        c.update(M=_log_int(rng, 2000, 100000), B=rng.choice([16, 32, 50, 64]))
    elif kind == "fsc":
        c.update(d=rng.choice([64, 96, 128, 144, 192, 256, 288]), M=1, B=1)
    elif kind == "nearest":
        c.update(M=_log_int(rng, 1000, 500000), k=rng.choice([1, 1, 1, 3, 8]), B=1)
    else:
        c.update(M=_log_int(rng, 1000, 500000), B=1)
    return c


# ------------------------------------------------------------ inputs ----


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _scales(case):
    return WIDE if case["wide"] else NARROW


def _tau(case):
    """1e-4 of the largest peak that the recipe allows (0: every pair)."""
    if not case["tau"]:
        return 0.0
    lo, hi = _scales(case)
    if case["norm"] == 0:
        peak = 1.5 / (2 * math.pi * (lo * APIX) ** 2)
    else:
        peak = 1.5 * math.sqrt(2 * math.pi) * hi * APIX
    return float(np.float32(1e-4 * peak))


def _tau_query(case):
    lo, _ = _scales(case)
    peak = 1.5 if case["norm"] else 1.5 / ((2 * math.pi) ** 1.5 * (lo * APIX) ** 3)
    return float(np.float32(1e-4 * peak))


def _unit(q):
    return q / q.norm(dim=-1, keepdim=True)


def _rotation(q):
    """[..., 4] unit quaternions (w x y z) -> [..., 3, 3]."""
    w, x, y, z = q.unbind(-1)
    rows = [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
            2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
            2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]
    return torch.stack(rows, -1).reshape(*q.shape[:-1], 3, 3)


def _gaussians(case, g):
    M, box = case["M"], case["d"] * APIX
    nc = 8 if case["wide"] else 64
    rnd = dict(device="cuda", dtype=torch.float64, generator=g)
    dirs = _unit(torch.randn(nc, 3, **rnd))
    centres = dirs * (0.3 * box * torch.rand(nc, 1, **rnd) ** (1 / 3))
    member = torch.randint(nc, (M,), device="cuda", generator=g)
    p = centres[member] + 0.04 * box * torch.randn(M, 3, **rnd)
    lo, hi = _scales(case)
    s = torch.exp(math.log(lo) + math.log(hi / lo) * torch.rand(M, 3, **rnd)) * APIX
    q = torch.randn(M, 4, **rnd)
    rho = 0.5 + torch.rand(M, 1, **rnd)
    return torch.cat([p, s, q, rho], 1).float().contiguous()


def _views(B, g):
    R = _rotation(_unit(torch.randn(B, 4, device="cuda", dtype=torch.float64, generator=g)))
    t = 2 * APIX * torch.randn(B, 2, device="cuda", dtype=torch.float64, generator=g)
    return R.float().contiguous(), t.float().contiguous()


def _ctf(case, B, g):
    """(ctf_params [B][8], None) or (None, ctf [B][d][d/2+1])."""
    if case["array"]:
        return None, 2 * torch.rand(B, case["d"], case["d"] // 2 + 1, device="cuda", generator=g) - 1
    u = torch.rand(B, 3, device="cuda", dtype=torch.float64, generator=g)
    df, ast = 1.0e4 + 1.5e4 * u[:, 0], 500 * u[:, 1]
    c = torch.zeros(B, 8, device="cuda", dtype=torch.float64)
    c[:, 0], c[:, 1], c[:, 2] = df + 0.5 * ast, df - 0.5 * ast, math.pi * u[:, 2]
    c[:, 3], c[:, 4], c[:, 5] = 300.0, 2.7, 0.1
    return c.float().contiguous(), None


def _images(case, B, g):
    disc = math.pi * (0.3 * case["d"] * APIX) ** 2
    sigma = case["M"] / disc / math.sqrt(0.1)
    return sigma * torch.randn(B, case["d"], case["d"], device="cuda", generator=g)


def _maps(case, g):
    """Two half maps: a common low-passed density plus independent noise."""
    d = case["d"]
    f = torch.fft.fftfreq(d, device="cuda")
    k2 = f[:, None, None] ** 2 + f[None, :, None] ** 2 + f[None, None, :d // 2 + 1].abs() ** 2
    spec = torch.fft.rfftn(torch.randn(d, d, d, device="cuda", generator=g)) * torch.exp(-k2 / (2 * 0.06 ** 2))
    signal = torch.fft.irfftn(spec, s=(d, d, d))
    signal = signal / signal.std()
    return [(signal + 0.7 * torch.randn(d, d, d, device="cuda", generator=g)).contiguous() for _ in range(2)]


def _adam_inputs(case, g):
    M = case["M"]
    params = _gaussians(case, g)
    raw = params.clone()
    raw[:, 3:6] = raw[:, 3:6].log()
    raw[:, 10] = raw[:, 10].log()
    grad = 1e-3 * torch.randn(M, NPAR, device="cuda", generator=g)
    m = 3e-4 * torch.randn(M, NPAR, device="cuda", generator=g)
    v = 1e-6 * (0.5 + torch.rand(M, NPAR, device="cuda", generator=g))
    return raw, m, v, grad


def _train_inputs(case, seed):
    """Parameters, a data set of four batches, optimiser moments of a run
    that is under way, and the state of the batch generator."""
    g = _gen(seed)
    params = _gaussians(case, g)
    N = 4 * case["B"]
    R, t = _views(N, g)
    prm, _ = _ctf(case, N, g)
    data = {"images": _images(case, N, g), "R": R, "t": t, "ctf_params": prm}
    # the loss scales with the squared signal, its gradient with signal / d^2
    # per pixel and image; the moments only need its order of magnitude
    G = float(data["images"].std()) / case["d"] ** 2
    m = 0.3 * G * torch.randn(case["M"], NPAR, device="cuda", generator=g)
    v = G * G * (0.5 + torch.rand(case["M"], NPAR, device="cuda", generator=g))
    return params, data, m, v, np.random.default_rng(int(seed))


def _inputs(case, seed):
    """What the call reads, by name (also what exact() starts from)."""
    kind, g = case["kind"], _gen(seed)
    if kind == "ctf":
        shape = (case["B"], case["d"], case["d"])
        prm, arr = _ctf(case, case["B"], g)
        signal = torch.randn(shape, device="cuda", generator=g)
        return {"proj": signal, "images": 3 * torch.randn(shape, device="cuda", generator=g), "ctf_params": prm,
                "ctf": arr}
    if kind == "fsc":
        return {"maps": _maps(case, g)}
    if kind == "adam":
        return dict(zip(("raw", "m", "v", "grad"), _adam_inputs(case, g)))
    out = {"params": _gaussians(case, g)}
    if kind in ("step", "project", "predict"):
        out["R"], out["t"] = _views(case["B"], g)
    if kind in ("step", "predict"):
        out["ctf_params"], out["ctf"] = _ctf(case, case["B"], g)
        out["images"] = _images(case, case["B"], g)
    return out


def _context(case):
    tau = _tau(case)
    per = 16
    if case["wide"]:
        per = 32
    if not case["tau"]:  # every tile of every view
        per = max(16, (case["d"] // 16) ** 2)
    return binding.Context(case["d"], APIX, case["B"], case["M"], tau=tau, norm_mode=case["norm"],
                           zsort=case["zsort"], no_rotation=int(case["norot"]), isotropic=int(case["iso"]),
                           max_pairs=per * case["B"] * case["M"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        params, data, m, v, rng = _train_inputs(case, seed)
        tr = train.Trainer(
            train.ModelConfig(d=case["d"], apix=APIX, M=case["M"], tau=_tau(case), norm_mode=case["norm"],
                              no_rotation=int(case["norot"]), isotropic=int(case["iso"]), zsort=case["zsort"]),
            train.TrainConfig(batch=case["B"], lr=TRAIN_LR, seed=int(seed), iso_nn=False),
            params.cpu().numpy(), {k: x.cpu().numpy() for k, x in data.items()})
        st = tr.state_dict()  # resume a run that has been under way for 1000 steps
        st.update(m=m.cpu(), v=v.cpu(), step=1000)
        tr.load_state_dict(st)
        return {"case": case, "trainer": tr}
    s = _inputs(case, seed)
    s["case"] = case
    B, d, M = case["B"], case["d"], case["M"]
    new = dict(device="cuda")
    if kind == "ctf":
        s["ctx"] = binding.Context(d, APIX, B, 1)
        s["pred"], s["dproj"] = torch.empty(B, d, d, **new), torch.empty(B, d, d, **new)
        s["loss_img"] = torch.empty(B, dtype=torch.float64, **new)
    elif kind == "adam":
        s["ctx"] = binding.Context(d, APIX, 1, M)
        s["params"] = torch.empty_like(s["raw"])
        s["step"] = 1000
    elif kind in ("fsc", "nearest"):
        s["ctx"] = binding.Context(d, APIX, 1, M)
    else:
        s["ctx"] = _context(case)
    if kind == "nearest":
        s["dist"], s["idx"] = torch.empty(M, case["k"], **new), torch.empty(M, case["k"], dtype=torch.int32, **new)
    if kind == "query":
        s["vol"] = torch.empty(d, d, d, **new)
    if kind == "project":
        s["proj"] = torch.empty(B, d, d, **new)
    if kind == "predict":
        s["pred"] = torch.empty(B, d, d, **new)
    if kind in ("ctf", "step", "predict"):
        s["loss"] = torch.empty(1, dtype=torch.float64, **new)
    if kind == "step":
        s["grad"] = torch.empty(M, NPAR, **new)
        if case["tune"]:
            s["ctx"].gem_autotune(s["params"], s["R"], s["t"])
    return s


# -------------------------------------------------------------- runs ----


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "train":
        tr = s["trainer"]
        loss = tr.step()
        return {"loss": loss, "params": tr.params, "raw": tr.raw, "m": tr.m, "v": tr.v}
    ctx = s["ctx"]
    if kind == "step":
        ctx.gem_forward(s["params"], s["R"], s["t"], s["images"], s["loss"], ctf=s["ctf"],
                        ctf_params=s["ctf_params"])
        ctx.gem_backward(s["grad"])
        return {"loss": s["loss"], "grad": s["grad"]}
    if kind == "project":
        ctx.gem_project(s["params"], s["R"], s["t"], s["proj"])
        return {"proj": s["proj"]}
    if kind == "predict":
        ctx.gem_forward(s["params"], s["R"], s["t"], s["images"], s["loss"], ctf=s["ctf"],
                        ctf_params=s["ctf_params"], pred=s["pred"])
        return {"loss": s["loss"], "pred": s["pred"]}
    if kind == "ctf":
        ctx.gem_ctf_loss(s["proj"], s["images"], ctf=s["ctf"], ctf_params=s["ctf_params"], pred=s["pred"],
                         dproj=s["dproj"], loss_img=s["loss_img"], loss=s["loss"])
        return {"pred": s["pred"], "dproj": s["dproj"], "loss_img": s["loss_img"], "loss": s["loss"]}
    if kind == "query":
        ctx.gem_query(s["params"], tau=_tau_query(case), vol=s["vol"])
        return {"vol": s["vol"]}
    if kind == "fsc":
        fsc, sums, res = ctx.gem_fsc(*s["maps"])
        return {"fsc": fsc, "sums": sums, "resolution": res}
    if kind == "nearest":
        ctx.gem_nn_distance(s["params"], case["k"], dist=s["dist"], idx=s["idx"])
        return {"dist": s["dist"], "idx": s["idx"]}
    s["step"] += 1
    ctx.gem_adam_step(s["raw"], s["m"], s["v"], s["grad"], s["params"], TRAIN_LR, s["step"])
    return {"raw": s["raw"], "m": s["m"], "v": s["v"], "params": s["params"]}


# -------------------------------------------------------------- work ----


def _kept_pixels(case, query=False):
    """Mean number of pixels (voxels) where one Gaussian of the recipe is
    above the threshold, from a fixed sample (the image border ignored)."""
    n = 4096
    rng = np.random.default_rng(7)
    lo, hi = _scales(case)
    s = np.exp(rng.uniform(math.log(lo), math.log(hi), (n, 3)))
    if case["iso"]:
        s[:] = s[:, :1]
    q = rng.normal(size=(n, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    W = _rotation(torch.from_numpy(q)).numpy()
    rho = rng.uniform(0.5, 1.5, n)
    if query:
        det = np.prod(s, axis=1)  # sqrt of the determinant, pixel^3
        amp = rho if case["norm"] else rho / ((2 * math.pi) ** 1.5 * det * APIX ** 3)
        head = np.maximum(2 * np.log(amp / _tau_query(case)), 0.0)
        return float(np.mean(4 / 3 * math.pi * head ** 1.5 * det))
    if not case["tau"]:
        return float(case["d"] ** 2)
    S = np.einsum("nik,nk,njk->nij", W[:, :2], s ** 2, W[:, :2])
    det = np.sqrt(np.linalg.det(S))
    if case["norm"] == 0:
        amp = rho / (2 * math.pi * det * APIX ** 2)
    else:
        amp = rho * math.sqrt(2 * math.pi) * np.prod(s, axis=1) / det * APIX
    head = np.maximum(2 * np.log(amp / _tau(case)), 0.0)
    return float(np.mean(math.pi * head * det))


def work(case):
    kind, d, M, B = case["kind"], case["d"], case["M"], case["B"]
    img, par = 4 * B * d * d, 4 * M * NPAR
    ctf = 4 * B * (d * (d // 2 + 1) if case["array"] else 8)
    fft2 = 5 * B * d * d * 2 * math.log2(d)  # one complex 2D transform of every image
    if kind == "adam":
        return {"bytes": 8 * par, "flops": 20 * M * NPAR}
    if kind == "nearest":
        return {"bytes": 12 * M + 8 * M * case["k"], "flops": 8 * 27 * 2 * M}
    if kind == "fsc":
        return {"bytes": 8 * d ** 3, "flops": 5 * d ** 3 * 3 * math.log2(d) + 14 * d ** 3}
    if kind == "query":
        return {"bytes": par + 4 * d ** 3, "flops": 10 * M * _kept_pixels(case, query=True)}
    if kind == "ctf":
        return {"bytes": 4 * img + ctf, "flops": 2 * fft2 + 60 * B * d * d}
    kept = M * B * _kept_pixels(case)
    views = 44 * B
    if kind == "project":
        return {"bytes": par + views + img, "flops": 10 * kept}
    if kind == "predict":
        return {"bytes": par + views + ctf + 2 * img, "flops": 10 * kept + 2 * fft2 + 60 * B * d * d}
    # forward and backward of every kept pair, both transforms
    step = {"bytes": 2 * par + views + ctf + img, "flops": 40 * kept + 2 * fft2 + 60 * B * d * d}
    if kind == "train":
        return {"bytes": step["bytes"] + 7 * par, "flops": step["flops"] + 20 * M * NPAR}
    return step


# ------------------------------------------------------------- exact ----


def _project_64(case, th, R, t):
    """[n][11] float64 Gaussians, views [v] -> (px, py, cxx, cxy, cyy, ln A),
    each [v][n], in pixel units."""
    s = th[:, 3:4].expand(-1, 3) if case["iso"] else th[:, 3:6]
    one = torch.tensor([1.0, 0.0, 0.0, 0.0], dtype=torch.float64, device=th.device).expand(th.shape[0], 4)
    Rq = _rotation(one if case["norot"] else _unit(th[:, 6:10]))
    L = Rq * s[:, None, :]  # Sigma = L L^T
    V = torch.einsum("vak,nkc->vnac", R[:, :2], L)  # the viewed factor, two rows
    p = torch.einsum("vak,nk->vna", R[:, :2], th[:, :3]) + t[:, None, :]
    px, py = p[..., 0] / APIX + case["d"] / 2, p[..., 1] / APIX + case["d"] / 2
    a = torch.linalg.cross(V[..., 0, :], V[..., 1, :])
    det = (a * a).sum(-1)  # of the projected covariance, Angstrom^4
    sxx, sxy, syy = (V[..., 0, :] ** 2).sum(-1), (V[..., 0, :] * V[..., 1, :]).sum(-1), (V[..., 1, :] ** 2).sum(-1)
    f = APIX ** 2 / det
    ln = torch.log(th[:, 10]) - 0.5 * torch.log(det)
    if case["norm"] == 0:
        ln = ln - math.log(2 * math.pi)
    else:
        ln = ln + 0.5 * math.log(2 * math.pi) + torch.log(s.abs()).sum(-1)
    return px, py, syy * f, -sxy * f, sxx * f, ln


def _boxes(case, q):
    """The extent box of every (view, Gaussian) above the threshold, grouped
    by size: (indices into the flattened q, x0, y0, box width, box height)."""
    px, py, cxx, cxy, cyy, ln = [x.detach().reshape(-1) for x in q]
    d, tau = case["d"], _tau(case)
    n = px.numel()
    if tau == 0.0:
        zero = torch.zeros(n, dtype=torch.int64, device=px.device)
        yield torch.arange(n, device=px.device), zero, zero, d, d
        return
    head = 2 * (ln - math.log(tau))
    det = cxx * cyy - cxy * cxy
    rx, ry = (head.clamp(min=0) * cyy / det).sqrt(), (head.clamp(min=0) * cxx / det).sqrt()
    x0, x1 = (px - rx).ceil().clamp(min=0), (px + rx).floor().clamp(max=d - 1)
    y0, y1 = (py - ry).ceil().clamp(min=0), (py + ry).floor().clamp(max=d - 1)
    side = torch.maximum(x1 - x0, y1 - y0) + 1
    live = (head > 0) & (x1 >= x0) & (y1 >= y0)
    lo = 0
    for hi in (4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 768):
        ix = (live & (side > lo) & (side <= hi)).nonzero().view(-1)
        lo = hi
        if ix.numel():
            yield ix, x0[ix].long(), y0[ix].long(), min(hi, d), min(hi, d)


def _pairs(case, q):
    """Chunks of the kept pairs' boxes: (index, dx, dy, value, flat pixel,
    kept) with one row per (view, Gaussian)."""
    px, py, cxx, cxy, cyy, ln = [x.detach().reshape(-1) for x in q]
    d, tau, n = case["d"], _tau(case), q[0].shape[1]
    for ix, x0, y0, w, h in _boxes(case, q):
        step = max(1, (1 << 25) // (w * h))
        for c in range(0, ix.numel(), step):
            i = ix[c:c + step]
            u = (x0[c:c + step, None] + torch.arange(w, device=i.device))[:, None, :]
            v = (y0[c:c + step, None] + torch.arange(h, device=i.device))[:, :, None]
            dx, dy = u - px[i, None, None], v - py[i, None, None]
            val = torch.exp(ln[i, None, None] - 0.5 * (cxx[i, None, None] * dx * dx + cyy[i, None, None] * dy * dy) -
                            cxy[i, None, None] * dx * dy)
            kept = (val > tau) & (u < d) & (v < d)
            pix = ((i // n)[:, None, None] * d + v.clamp(max=d - 1)) * d + u.clamp(max=d - 1)
            yield i, dx, dy, val, pix, kept


def _view_chunks(case):
    step = max(1, (1 << 21) // case["M"])
    return [(b, min(case["B"], b + step)) for b in range(0, case["B"], step)]


def _images_64(case, th, R, t):
    d = case["d"]
    out = torch.zeros(case["B"], d, d, dtype=torch.float64, device=th.device)
    with torch.no_grad():
        for b0, b1 in _view_chunks(case):
            flat = out[b0:b1].view(-1)
            for _, _, _, val, pix, kept in _pairs(case, _project_64(case, th, R[b0:b1], t[b0:b1])):
                flat.index_add_(0, pix[kept], val[kept])
    return out


def _gradient_64(case, th, R, t, dproj):
    """dL/dparams from dL/dproj over the kept pairs."""
    grad = torch.zeros_like(th)
    for b0, b1 in _view_chunks(case):
        x = th.clone().requires_grad_(True)
        q = _project_64(case, x, R[b0:b1], t[b0:b1])
        cxx, cxy, cyy = [a.detach().reshape(-1) for a in q[2:5]]
        up = torch.zeros(6, q[0].numel(), dtype=torch.float64, device=th.device)
        g = dproj[b0:b1].reshape(-1)
        for i, dx, dy, val, pix, kept in _pairs(case, q):
            w = torch.where(kept, g[pix] * val, torch.zeros_like(val))
            wx, wy = w * dx, w * dy
            sx, sy = wx.sum((1, 2)), wy.sum((1, 2))
            up[0, i], up[1, i] = cxx[i] * sx + cxy[i] * sy, cxy[i] * sx + cyy[i] * sy
            up[2, i], up[3, i] = -0.5 * (wx * dx).sum((1, 2)), -(wx * dy).sum((1, 2))
            up[4, i], up[5, i] = -0.5 * (wy * dy).sum((1, 2)), w.sum((1, 2))
        (gx,) = torch.autograd.grad(list(q), [x], [u.view_as(q[0]) for u in up])
        grad += gx
    return grad


def _transfer_64(case, prm, arr):
    """The transfer function on the full DFT grid, made even."""
    d = case["d"]
    if arr is not None:
        a = arr.double()
        H = torch.empty(a.shape[0], d, d, dtype=torch.float64, device=a.device)
        H[:, :, :d // 2 + 1] = a
        neg = (-torch.arange(d, device=a.device)) % d
        H[:, :, d // 2 + 1:] = a[:, neg][:, :, neg[d // 2 + 1:]]
    else:
        p = prm.double()[:, :, None, None]
        k = torch.fft.fftfreq(d, d=APIX, device=prm.device, dtype=torch.float64)
        kx, ky = k[None, None, :], k[None, :, None]
        k2 = kx ** 2 + ky ** 2
        volt, cs = p[:, 3] * 1e3, p[:, 4] * 1e7
        lam = 12.2643247 / torch.sqrt(volt * (1 + 0.978466e-6 * volt))
        df = 0.5 * (p[:, 0] + p[:, 1]) + 0.5 * (p[:, 0] - p[:, 1]) * torch.cos(2 * (torch.atan2(ky, kx) - p[:, 2]))
        chi = math.pi * lam * df * k2 - 0.5 * math.pi * cs * lam ** 3 * k2 ** 2 + p[:, 6]
        H = -(torch.sqrt(1 - p[:, 5] ** 2) * torch.sin(chi) + p[:, 5] * torch.cos(chi)) * torch.exp(-p[:, 7] * k2 / 4)
    neg = (-torch.arange(d, device=H.device)) % d
    return 0.5 * (H + H[:, neg][:, :, neg])


def _loss_64(case, proj, images, prm, arr):
    """(pred, dproj, loss_img [B], loss [1])."""
    H = _transfer_64(case, prm, arr)
    pred = torch.fft.ifft2(H * torch.fft.fft2(proj)).real
    r = pred - images.double()
    loss_img = (r * r).mean((1, 2))
    scale = 2.0 / (r.shape[0] * case["d"] ** 2)
    dproj = torch.fft.ifft2(H * torch.fft.fft2(scale * r)).real
    return pred, dproj, loss_img, loss_img.mean().view(1)


def _adam_64(raw, m, v, grad, step):
    raw, m, v, g = (x.double() for x in (raw, m, v, grad))
    lr = torch.tensor([TRAIN_LR[0]] * 3 + [TRAIN_LR[1]] * 3 + [TRAIN_LR[2]] * 4 + [TRAIN_LR[3]], dtype=torch.float64,
                      device=raw.device)
    log = torch.tensor([0] * 3 + [1] * 3 + [0] * 4 + [1], dtype=torch.bool, device=raw.device)
    b1, b2 = (float(np.float32(x)) for x in (0.9, 0.999))
    g = torch.where(log, g * raw.exp(), g)
    m = b1 * m + (1 - b1) * g
    v = b2 * v + (1 - b2) * g * g
    raw = raw - lr * (m / (1 - b1 ** step)) / (torch.sqrt(v / (1 - b2 ** step)) + 1e-8)
    return raw, m, v, torch.where(log, raw.exp(), raw)


def _query_64(case, th):
    """The density on the voxel grid: every Gaussian over its extent box."""
    d, tau = case["d"], _tau_query(case)
    s = th[:, 3:4].expand(-1, 3) if case["iso"] else th[:, 3:6]
    Rq = torch.eye(3, dtype=torch.float64, device=th.device).expand(th.shape[0], 3, 3) if case["norot"] else \
        _rotation(_unit(th[:, 6:10]))
    ln = torch.log(th[:, 10])
    if case["norm"] == 0:
        ln = ln - 1.5 * math.log(2 * math.pi) - torch.log(s.abs()).sum(-1)
    P = torch.einsum("nik,nk,njk->nij", Rq, s ** -2, Rq) * APIX ** 2
    S = torch.einsum("nik,nk,nik->ni", Rq, s ** 2, Rq) / APIX ** 2
    c = th[:, :3] / APIX + d / 2
    head = 2 * (ln - math.log(tau))
    r = (head.clamp(min=0)[:, None] * S).sqrt()
    x0, x1 = (c - r).ceil().clamp(min=0), (c + r).floor().clamp(max=d - 1)
    side = (x1 - x0 + 1).amax(1)
    live = (head > 0) & (x1 >= x0).all(1)
    vol = torch.zeros(d ** 3, dtype=torch.float64, device=th.device)
    lo = 0
    for hi in (4, 6, 8, 10, 12, 16, 20, 24, 32, 48, 64, 96, 128):
        ix = (live & (side > lo) & (side <= hi)).nonzero().view(-1)
        lo = hi
        w = torch.arange(min(hi, d), device=th.device)
        step = max(1, (1 << 24) // w.numel() ** 3)
        for k in range(0, ix.numel(), step):
            i = ix[k:k + step]
            v = [x0[i, a].long()[:, None] + w for a in range(3)]  # x, y, z
            D = [v[a] - c[i, a, None] for a in range(3)]
            X, Y, Z = D[0][:, None, None, :], D[1][:, None, :, None], D[2][:, :, None, None]
            p = P[i][:, :, :, None, None, None]
            val = torch.exp(ln[i, None, None, None] - 0.5 * (p[:, 0, 0] * X * X + p[:, 1, 1] * Y * Y + p[:, 2, 2] * Z * Z) -
                            p[:, 0, 1] * X * Y - p[:, 0, 2] * X * Z - p[:, 1, 2] * Y * Z)
            vx, vy, vz = v[0][:, None, None, :], v[1][:, None, :, None], v[2][:, :, None, None]
            kept = (val > tau) & (vx < d) & (vy < d) & (vz < d)
            pix = (vz * d + vy) * d + vx
            vol.index_add_(0, pix[kept], val[kept])
    return vol.view(d, d, d)


def _fsc_64(case, maps, threshold=float(np.float32(0.143))):
    d = case["d"]
    F1, F2 = (torch.fft.fftn(m.double()) for m in maps)
    k = torch.fft.fftfreq(d, d=1.0 / d, device="cuda", dtype=torch.float64).round()
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2
    shell = torch.floor(k2.sqrt() + 0.5).long().view(-1)
    n = d // 2 + 1
    at = shell < n
    sums = torch.stack([torch.bincount(shell[at], x.reshape(-1)[at], n) for x in
                        ((F1 * F2.conj()).real, F1.abs() ** 2, F2.abs() ** 2)])
    fsc = sums[0] / (sums[1] * sums[2]).sqrt()
    f, kstar = fsc.cpu().numpy(), float(n - 1)
    for i in range(1, n):
        if f[i] < threshold:
            kstar = i - 1 + (f[i - 1] - threshold) / (f[i - 1] - f[i])
            break
    return fsc, sums, torch.tensor([d * APIX / kstar], dtype=torch.float64)


def _nearest_64(case, th):
    p, M, k = th[:, :3], case["M"], case["k"]
    out = torch.empty(M, k, dtype=torch.float64, device=th.device)
    step = max(1, (1 << 28) // M)
    for c in range(0, M, step):
        n = min(step, M - c)
        d2 = torch.zeros(n, M, dtype=torch.float64, device=th.device)
        for a in range(3):
            x = p[c:c + n, a, None] - p[None, :, a]
            d2 += x.mul_(x)
        i = torch.arange(n, device=th.device)
        d2[i, c + i] = math.inf
        out[c:c + n] = d2.amin(1, keepdim=True) if k == 1 else d2.topk(k, dim=1, largest=False).values
    return out.sqrt()


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        params, data, m, v, rng = _train_inputs(case, seed)
        ix = torch.as_tensor(np.sort(rng.choice(4 * case["B"], size=case["B"], replace=False)), device="cuda")
        raw = torch.as_tensor(train_raw(params.cpu().numpy())).cuda()
        th = raw.double()
        th = torch.cat([th[:, :3], th[:, 3:6].exp(), th[:, 6:10], th[:, 10:].exp()], 1)
        R, t = data["R"][ix].double(), data["t"][ix].double()
        _, dproj, _, loss = _loss_64(case, _images_64(case, th, R, t), data["images"][ix], data["ctf_params"][ix], None)
        grad = _gradient_64(case, th, R, t, dproj)
        raw, m, v, p = _adam_64(raw, m, v, grad, 1001)
        return {"loss": loss, "params": p, "raw": raw, "m": m, "v": v}
    s = _inputs(case, seed)
    if kind == "adam":
        raw, m, v, p = _adam_64(s["raw"], s["m"], s["v"], s["grad"], 1001)
        return {"raw": raw, "m": m, "v": v, "params": p}
    if kind == "fsc":
        return dict(zip(("fsc", "sums", "resolution"), _fsc_64(case, s["maps"])))
    if kind == "ctf":
        pred, dproj, loss_img, loss = _loss_64(case, s["proj"].double(), s["images"], s["ctf_params"], s["ctf"])
        return {"pred": pred, "dproj": dproj, "loss_img": loss_img, "loss": loss}
    th = s["params"].double()
    if kind == "nearest":
        if case["k"] > 1 and case["M"] > 150000:  # a minute of selection
            return None
        return {"dist": _nearest_64(case, th), "idx": None}
    if kind == "query":
        return {"vol": _query_64(case, th)}
    R, t = s["R"].double(), s["t"].double()
    proj = _images_64(case, th, R, t)
    if kind == "project":
        return {"proj": proj}
    pred, dproj, _, loss = _loss_64(case, proj, s["images"], s["ctf_params"], s["ctf"])
    if kind == "predict":
        return {"loss": loss, "pred": pred}
    return {"loss": loss, "grad": _gradient_64(case, th, R, t, dproj)}


def train_raw(params):
    """float32 (p, log s, q, log rho), as a training run starts from them."""
    raw = np.array(params, dtype=np.float32)
    raw[:, 3:6] = np.log(raw[:, 3:6])
    raw[:, 10] = np.log(raw[:, 10])
    return raw
