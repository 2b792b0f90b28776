"""What a user of this framework has it do, as cases that can be timed and checked.

Wave cases model shots, gradients and Born data on a padded 2D or 3D grid through
``wave_forward``, ``wave_gradient``, ``wave_born``, ``forward_model`` (autograd) and
``wave_gradient_batch``; FNO cases run one Fourier layer of the BF16 inference path
and one training step of the preconditioner network.  ``exact`` solves the same
problems in float64 with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2304_05592_gb300 import autograd, fno, wave

DEV = "cuda"
STORES = {"checkpoint": wave.STORE_CHECKPOINT, "bf16": wave.STORE_BF16, "fp32": wave.STORE_FP32}


def listed():
    return [
        # the size of the smoke test and of most unit tests: latency and launches
        dict(name="fwd2d_smoke", kind="forward2d", nx=67, nz=45, nb=12, h=10.0, nt=160, nshot=2, nrec=23, f0=12.0,
             snap=False),
        # one shot over a 2 km two-layer style section, as a line search evaluates it
        dict(name="fwd2d_one_shot", kind="forward2d", nx=201, nz=201, nb=40, h=10.0, nt=1000, nshot=1, nrec=201,
             f0=15.0, snap=True),
        # stochastic FWI: the gradient of four random shots at the library's default checkpoint budget
        dict(name="grad2d_four_shots", kind="gradient2d", nx=512, nz=256, nb=40, h=6.25, nt=2000, nshot=4, nrec=512,
             f0=20.0, snap=True, store="checkpoint", nsnap=64, velocity=False),
        # the flagship: the checkpointed gradient of a 32-shot survey with the benchmark's checkpoint budget
        dict(name="grad2d_survey", kind="gradient2d", nx=512, nz=256, nb=40, h=6.25, nt=4000, nshot=32, nrec=512,
             f0=20.0, snap=True, store="checkpoint", nsnap=1536, velocity=False),
        # preconditioner training data: the 8-shot velocity gradient with the BF16 store
        dict(name="grad2d_pairs_bf16", kind="gradient2d", nx=512, nz=256, nb=40, h=10.0, nt=2000, nshot=8, nrec=512,
             f0=15.0, snap=True, store="bf16", nsnap=1, velocity=True),
        # differentiable modelling in a user's own loss: ragged grid, points off the grid, both pullbacks
        dict(name="autograd2d_ragged", kind="autograd2d", nx=301, nz=173, nb=37, h=7.5, nt=900, nshot=3, nrec=97,
             f0=14.0, snap=False),
        # one linearised modelling of a least-squares migration iteration over the survey
        dict(name="born2d_survey", kind="born2d", nx=512, nz=256, nb=40, h=6.25, nt=1000, nshot=32, nrec=512, f0=20.0,
             snap=True),
        # 3D modelling of one shot into a full surface grid of receivers
        dict(name="fwd3d_shot", kind="forward3d", nx=400, ny=400, nz=300, nb=40, h=10.0, nt=240, nshot=1, rx=400,
             ry=400, f0=15.0),
        # a small 3D gradient with checkpoints
        dict(name="grad3d_small", kind="gradient3d", nx=101, ny=83, nz=67, nb=20, h=10.0, nt=300, nshot=2, rx=25, ry=20,
             f0=15.0, store="checkpoint", nsnap=24, velocity=False),
        # independent problems of different sizes, models and record lengths in one call
        dict(name="batch2d_uneven", kind="batch2d", nprob=24, nx_lo=256, nx_hi=768, nz_lo=128, nz_hi=384, nt_lo=1500,
             nt_hi=4000, nb=40, store="bf16", layout=4),
        # one Fourier layer of the preconditioner's BF16 inference
        dict(name="fno_layer_bf16", kind="fno_layer", B=8, Nz=256, Nx=512, width=32, mz=16, mx=16, dtype="bf16"),
        # one optimiser step of the preconditioner's training
        dict(name="fno_train_step", kind="fno_train", B=8, Nz=256, Nx=512, width=32, hidden=64, layers=4, mz=16, mx=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward2d", "forward2d", "gradient2d", "gradient2d", "autograd2d", "born2d", "forward3d",
                       "gradient3d", "batch2d", "fno_layer", "fno_train"])
    if kind in ("forward2d", "gradient2d", "autograd2d", "born2d"):
        c = dict(kind=kind, nx=_log(rng, 60, 640), nz=_log(rng, 45, 360), nb=rng.choice([12, 20, 30, 40]),
                 h=rng.choice([6.25, 7.5, 10.0, 12.5]), nt=_log(rng, 160, 4000),
                 nshot=_log(rng, 1, 4 if kind == "autograd2d" else 32), nrec=_log(rng, 20, 512),
                 f0=rng.uniform(8.0, 20.0), snap=rng.random() < 0.5)
        # no more work than the flagship of its kind
        most = {"forward2d": 32 * 4000, "gradient2d": 32 * 2000, "autograd2d": 4 * 2000, "born2d": 32 * 1000}[kind]
        c["nt"] = max(160, min(c["nt"], most // c["nshot"]))
        if kind == "gradient2d":
            c.update(store=rng.choice(["checkpoint", "checkpoint", "bf16", "fp32"]), nsnap=rng.choice([16, 64, 256]),
                     velocity=rng.random() < 0.5)
            cell = (c["nx"] + 2 * c["nb"] + 31) // 32 * 32 * (c["nz"] + 2 * c["nb"])
            if c["store"] != "checkpoint":  # a full store within 20 GB
                c["nt"] = max(160, min(c["nt"], int(20e9 / (4.0 * cell * c["nshot"]))))
        return c
    if kind in ("forward3d", "gradient3d"):
        big = kind == "forward3d"
        c = dict(kind=kind, nx=_log(rng, 40, 320 if big else 140), ny=_log(rng, 40, 320 if big else 140),
                 nz=_log(rng, 30, 240 if big else 100), nb=rng.choice([8, 20, 40] if big else [8, 20]),
                 h=rng.choice([7.5, 10.0, 12.5]), nt=_log(rng, 80, 300), nshot=1 if big else rng.choice([1, 2, 3]),
                 rx=rng.randint(5, 40), ry=rng.randint(5, 40), f0=rng.uniform(10.0, 18.0))
        if not big:
            c.update(store=rng.choice(["checkpoint", "bf16"]), nsnap=rng.choice([8, 24]), velocity=rng.random() < 0.5)
        return c
    if kind == "batch2d":
        lo, zl = _log(rng, 80, 256), _log(rng, 60, 128)
        return dict(kind=kind, nprob=rng.randint(3, 20), nx_lo=lo, nx_hi=3 * lo, nz_lo=zl, nz_hi=3 * zl,
                    nt_lo=_log(rng, 300, 1500), nt_hi=_log(rng, 1600, 3000), nb=rng.choice([20, 40]),
                    store=rng.choice(["bf16", "bf16", "fp32"]), layout=rng.randint(5, 10000))
    Nz, Nx = _log(rng, 48, 256), _log(rng, 64, 512)
    c = dict(kind=kind, B=rng.randint(1, 8), Nz=Nz, Nx=Nx, width=rng.choice([16, 32, 32]), mz=rng.choice([8, 12, 16]),
             mx=rng.choice([8, 12, 16]))
    if kind == "fno_layer":
        c["dtype"] = rng.choice(["bf16", "bf16", "fp32"])
    else:
        c.update(hidden=rng.choice([32, 64]), layers=rng.choice([2, 3, 4]))
    return c


# --- inputs ------------------------------------------------------------------------------------


def _smooth(shape, sigma, gen):
    """White noise smoothed by a Gaussian of sigma cells, unit standard deviation (float64, host)."""
    w = torch.randn(shape, generator=gen, dtype=torch.float64)
    f = torch.fft.rfftn(w)
    for ax, n in enumerate(shape):
        k = torch.fft.rfftfreq(n) if ax == len(shape) - 1 else torch.fft.fftfreq(n)
        g = torch.exp(-2.0 * (math.pi * sigma * k.double()) ** 2)
        f = f * g.reshape([-1 if a == ax else 1 for a in range(len(shape))])
    s = torch.fft.irfftn(f, s=shape)
    return s / s.std()


def _model(shape, gen, vlo=1500.0, vhi=3500.0):
    """Layers of increasing velocity over a linear trend with 3 % smooth heterogeneity, m/s."""
    nz = shape[0]
    z = torch.arange(nz, dtype=torch.float64) / max(nz - 1, 1)
    cuts = torch.sort(torch.rand(4, generator=gen, dtype=torch.float64) * 0.8 + 0.1).values
    layer = torch.searchsorted(cuts, z).double() / 4
    v = vlo + (vhi - vlo) * (0.5 * z + 0.5 * layer)
    v = v.reshape([nz] + [1] * (len(shape) - 1)) * (1.0 + 0.03 * _smooth(shape, 6.0, gen))
    return v.clamp(1400.0, 4500.0).float()


def _limit(ndim):
    return 2.0 / math.sqrt(ndim * 2048.0 / 315.0)


def _f32(x):
    return float(np.float32(x))


def _ricker(f0, dt, nt):
    a = (math.pi * f0 * (np.arange(nt) * dt - 1.0 / f0)) ** 2
    return ((1.0 - 2.0 * a) * np.exp(-a)).astype(np.float32)


def _points2d(c, gen, h):
    """One source per shot near the surface and a line of receivers, on grid points (snap) or between them."""
    nx, nz, ns, nr = c["nx"], c["nz"], c["nshot"], c["nrec"]
    Lx = (nx - 1) * h
    r = torch.rand((3, max(ns, nr)), generator=gen, dtype=torch.float64).numpy()
    sx = (np.arange(ns) + 0.2 + 0.6 * r[0, :ns]) / ns * Lx
    rx = np.linspace(0.0, Lx, nr)
    sz, rz = np.full(ns, 2 * h), np.full(nr, 2 * h)
    if not c["snap"]:
        sz, rz = sz + h * (0.2 + 0.5 * r[1, :ns]), rz + h * (0.1 + 0.8 * r[2, :nr])
    else:
        sx, rx = np.round(sx / h) * h, np.round(rx / h) * h
    src = np.stack([sx, sz], -1)[:, None, :].astype(np.float32)
    rec = np.repeat(np.stack([rx, rz], -1)[None], ns, 0).astype(np.float32)
    return src, np.minimum(rec, np.float32(Lx))


def _points3d(c, h):
    nx, ny, ns = c["nx"], c["ny"], c["nshot"]
    sx = (np.arange(ns) + 1) / (ns + 1) * (nx - 1) * h
    src = np.stack([sx, np.full(ns, 0.45 * (ny - 1) * h), np.full(ns, h)], -1)[:, None, :].astype(np.float32)
    gx = np.round(np.linspace(0, nx - 1, min(c["rx"], nx))) * h
    gy = np.round(np.linspace(0, ny - 1, min(c["ry"], ny))) * h
    X, Y = np.meshgrid(gx, gy, indexing="xy")
    rec = np.stack([X.ravel(), Y.ravel(), np.full(X.size, h)], -1)[None].astype(np.float32)
    return src, np.repeat(rec, ns, 0)


def _records(src, rec, nt, dt, f0, gen, scale):
    """Observed records: three events with hyperbolic moveout from each source and 5 % noise."""
    ns, nr = src.shape[0], rec.shape[1]
    off = np.linalg.norm(rec[:, :, :-1] - src[:, :, :-1], axis=-1)  # [ns][nr]
    off = torch.from_numpy(off.astype(np.float64)).to(DEV)
    t = torch.arange(nt, dtype=torch.float64, device=DEV)[None, :, None] * dt
    d = torch.zeros((ns, nt, nr), dtype=torch.float32, device=DEV)
    r = torch.rand((3, 2), generator=gen, dtype=torch.float64).tolist()
    for e in range(3):
        t0, v = (0.0, 1600.0) if e == 0 else (r[e][0] * nt * dt * 0.8, 1800.0 + 1000.0 * r[e][1])
        for s in range(ns):
            arr = torch.sqrt(t0 * t0 + (off[s] / v) ** 2)[None, None, :] + 1.0 / f0
            a = (math.pi * f0 * (t - arr)) ** 2
            d[s] += ((0.6 ** e) * (1.0 - 2.0 * a) * torch.exp(-a))[0].float()
    g = torch.Generator(device=DEV).manual_seed(int(gen.initial_seed()) + 7)
    d += 0.05 * torch.randn(d.shape, generator=g, dtype=torch.float32, device=DEV)
    return d.mul_(scale).contiguous()


def _wave_inputs(c, seed):
    """Grid numbers, model, points, wavelet and observed records of a wave case."""
    gen = torch.Generator().manual_seed(seed)
    three = c["kind"].endswith("3d")
    h = _f32(c["h"])
    shape = (c["nz"], c["ny"], c["nx"]) if three else (c["nz"], c["nx"])
    vel = _model(shape, gen)
    src, rec = _points3d(c, h) if three else _points2d(c, gen, h)
    vmax = float(vel.max())
    dt = _f32(0.5 * _limit(3 if three else 2) * h / 4500.0)  # one time step for every model of the run
    q = np.repeat(_ricker(c["f0"], dt, c["nt"])[None, :, None], c["nshot"], 0)
    q *= (1.0 + 0.1 * torch.rand((c["nshot"], 1, 1), generator=gen).numpy()).astype(np.float32)
    x = dict(vel=vel.to(DEV), src=src, rec=rec, q=torch.from_numpy(q).to(DEV), h=h, dt=dt, vref=_f32(vmax), nb=c["nb"],
             nt=c["nt"])
    if c["kind"].startswith(("gradient", "autograd")):
        x["d"] = _records(src, rec, c["nt"], dt, c["f0"], gen, 0.05)
    if c["kind"].startswith("born"):
        x["dm"] = (1e-8 * _smooth(shape, 3.0, gen)).float().to(DEV)
    return x


def _grid(x):
    three = x["vel"].dim() == 3
    s = x["vel"].shape
    return wave.Grid(3 if three else 2, s[-1], s[0], x["h"], x["dt"], x["nt"], x["nb"], s[1] if three else 1, x["vref"])


def _batch_inputs(c, seed):
    """The problems of an uneven batch: sizes from the case alone, models and records from the seed."""
    sizes = np.random.default_rng(c["layout"])
    out = []
    for i in range(c["nprob"]):
        gen = torch.Generator().manual_seed(seed * 1000 + i)
        h = float(sizes.choice([6.25, 7.5, 10.0, 12.5]))
        nx, nz = int(sizes.integers(c["nx_lo"], c["nx_hi"] + 1)), int(sizes.integers(c["nz_lo"], c["nz_hi"] + 1))
        nt, f0 = int(sizes.integers(c["nt_lo"], c["nt_hi"] + 1)), float(sizes.uniform(8.0, 15.0))
        p = dict(kind="gradient2d", nx=nx, nz=nz, nb=c["nb"], h=h, nt=nt, nshot=1, nrec=nx, f0=f0, snap=True)
        vel = _model((nz, nx), gen)
        src, rec = _points2d(p, gen, h)
        dt = _f32(0.4 * _limit(2) * h / 4500.0)
        q = torch.from_numpy(_ricker(f0, dt, nt)[None, :, None]).to(DEV)
        out.append(dict(vel=vel.to(DEV), src=src, rec=rec, q=q, h=h, dt=dt, vref=_f32(float(vel.max())), nb=c["nb"], nt=nt,
                        d=_records(src, rec, nt, dt, f0, gen, 0.05)))
    return out


def _layer_inputs(c, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    W, KZ, mx = c["width"], 2 * c["mz"], c["mx"]
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    n = dict(generator=g, device=DEV)
    k = 1.0 / math.sqrt(W)
    return dict(v=(0.5 * torch.randn((c["B"], W, c["Nz"], c["Nx"]), **n)).to(dt),
                W=(2 * torch.rand((W, W), **n) - 1) * k, b=(2 * torch.rand((W,), **n) - 1) * k,
                R=torch.rand((W, W, KZ, mx, 2), **n) / W)


def _train_inputs(c, seed):
    """A batch of normalised gradients with coordinate channels, targets with a plume-like patch, and the weights."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    B, Nz, Nx = c["B"], c["Nz"], c["Nx"]
    x = torch.randn((B, 3, Nz, Nx), generator=g, device=DEV)
    x[:, 1] = torch.linspace(0, 1, Nz, device=DEV)[:, None]
    x[:, 2] = torch.linspace(0, 1, Nx, device=DEV)[None, :]
    y = -torch.rand((B, 1, Nz, Nx), generator=g, device=DEV)
    y[:, :, : Nz // 2] = 0.0
    W, H, KZ = c["width"], c["hidden"], 2 * c["mz"]
    shapes = [("P", (W, 3)), ("p", (W,))]
    for l in range(c["layers"]):
        shapes += [("W%d" % l, (W, W)), ("b%d" % l, (W,)), ("R%d" % l, (W, W, KZ, c["mx"], 2))]
    shapes += [("Q1", (H, W)), ("q1", (H,)), ("Q2", (1, H)), ("q2", (1,))]
    par = {}
    for name, s in shapes:
        u = torch.rand(s, generator=g, device=DEV)
        fan = s[1] if len(s) == 2 else {"p": 3, "q2": H}.get(name, W)
        par[name] = u / (W * W) if name.startswith("R") else (2 * u - 1) / math.sqrt(fan)
    return x, y, par


def prepare(case, seed):
    k = case["kind"]
    if k == "batch2d":
        return dict(case=case, problems=[wave.BatchProblem(_grid(x), x["vel"], x["src"][0], x["q"][0], x["rec"][0], x["d"][0])
                                         for x in _batch_inputs(case, seed)])
    if k == "fno_layer":
        x = _layer_inputs(case, seed)
        tx, tz = fno.fno_tables(case["Nz"], case["Nx"], case["mz"], case["mx"], DEV)
        return dict(case=case, tx=tx, tz=tz, **x)
    if k == "fno_train":
        x, y, par = _train_inputs(case, seed)
        cfg = fno.FNOConfig(3, case["width"], case["hidden"], case["layers"], case["mz"], case["mx"])
        net = fno.FNO2d(cfg, case["Nz"], case["Nx"], DEV, seed=0)
        for name, v in par.items():
            net.view(name).copy_(v)
        return dict(case=case, net=net, x=x, y=y)
    x = _wave_inputs(case, seed)
    x["grid"] = _grid(x)
    if k == "autograd2d":
        x["vel"].requires_grad_(True)
        x["q"].requires_grad_(True)
    return dict(case=case, **x)


def run(s):
    c = s["case"]
    k = c["kind"]
    if k.startswith("forward"):
        return wave.wave_forward(s["grid"], s["vel"], s["src"], s["q"], s["rec"])
    if k.startswith("gradient"):
        wrt = wave.WRT_VELOCITY if c["velocity"] else wave.WRT_SLOWNESS2
        phi, g, dsyn = wave.wave_gradient(s["grid"], s["vel"], s["src"], s["q"], s["rec"], s["d"],
                                          store=STORES[c["store"]], nsnap=c["nsnap"], want_dsyn=True, wrt=wrt)
        return {"misfit": np.float32(phi), "grad": g, "dsyn": dsyn}
    if k == "autograd2d":
        d = autograd.forward_model(s["vel"], s["q"], s["grid"], s["src"], s["rec"])
        gv, gq = torch.autograd.grad(d, (s["vel"], s["q"]), s["d"])
        return {"data": d, "g_vel": gv, "g_wavelet": gq}
    if k == "born2d":
        return wave.wave_born(s["grid"], s["vel"], s["src"], s["q"], s["rec"], s["dm"])
    if k == "batch2d":
        phi, grads = wave.wave_gradient_batch(s["problems"], store=STORES[c["store"]])
        return {"misfits": np.asarray(phi, np.float32), "grads": list(grads)}
    if k == "fno_layer":
        B, W, Nz, mz, mx = c["B"], c["width"], c["Nz"], c["mz"], c["mx"]
        t1 = fno.fno_dft_x(s["v"], mx, s["tx"][0])
        X = fno.fno_dft_z(t1, B * W, Nz, mz, mx, s["tz"])
        t2 = fno.fno_mix_idft_z(X, s["R"], B, W, W, Nz, mz, mx, s["tz"])
        return fno.fno_combine(s["v"], s["W"], W, bias=s["b"], T=t2, table=s["tx"][1], mx=mx, act=fno.ACT_GELU,
                               out_dtype=s["v"].dtype)
    net = s["net"]
    loss = net.train_step(s["x"], s["y"], 1e-3)
    return {"loss": loss.float(), "grads": net.grads, "params": net.params}


# --- the work of a pass -------------------------------------------------------------------------


def _numel(*shape):
    return float(np.prod(shape))


def _wave_work(nd, phys, npad, nt, ns, nrec, sweeps, extra):
    """Inputs and outputs once; the stencil's operations for every padded point, shot and step."""
    per = 31.0 if nd == 2 else 43.0  # 8th-order Laplacian and the damped update
    return dict(bytes=4.0 * (phys * (2 if extra else 1) + ns * nt + ns * nt * nrec * (2 if extra else 1)),
                flops=per * sweeps * npad * (nt - 1) * ns)


def work(case):
    c, k = case, case["kind"]
    if k == "batch2d":
        sizes, b, f = np.random.default_rng(c["layout"]), 0.0, 0.0
        for _ in range(c["nprob"]):
            sizes.choice([6.25, 7.5, 10.0, 12.5])
            nx, nz = int(sizes.integers(c["nx_lo"], c["nx_hi"] + 1)), int(sizes.integers(c["nz_lo"], c["nz_hi"] + 1))
            nt, _f = int(sizes.integers(c["nt_lo"], c["nt_hi"] + 1)), sizes.uniform(8.0, 15.0)
            w = _wave_work(2, nx * nz, (nx + 2 * c["nb"]) * (nz + 2 * c["nb"]), nt, 1, nx, 2.1, True)
            b, f = b + w["bytes"], f + w["flops"]
        return dict(bytes=b, flops=f)
    if k in ("fno_layer", "fno_train"):
        B, Nz, Nx, W, KZ, mx = c["B"], c["Nz"], c["Nx"], c["width"], 2 * c["mz"], c["mx"]
        pix = float(B * Nz * Nx)
        # the channel mix and both truncated transforms of one layer
        layer = pix * W * (2.0 * W + 8.0 * mx) + 16.0 * B * W * Nz * mx * KZ + 8.0 * B * W * W * KZ * mx
        R = _numel(W, W, KZ, mx, 2)
        if k == "fno_layer":
            e = 2 if c["dtype"] == "bf16" else 4
            return dict(bytes=2 * pix * W * e + 4 * R, flops=layer)
        n = c["layers"] * (R + W * W) + c["hidden"] * W
        fwd = c["layers"] * layer + pix * 2.0 * c["hidden"] * (W + 1)
        return dict(bytes=4 * (4 * pix) + 4 * 7 * n, flops=3 * fwd)
    nb2, nd = 2 * c["nb"], 3 if k.endswith("3d") else 2
    phys = c["nx"] * c["nz"] * (c["ny"] if nd == 3 else 1)
    npad = (c["nx"] + nb2) * (c["nz"] + nb2) * ((c["ny"] + nb2) if nd == 3 else 1)
    nrec = c["nrec"] if nd == 2 else min(c["rx"], c["nx"]) * min(c["ry"], c["ny"])
    sweeps = 1.0 if k.startswith("forward") else 2.2 if k.startswith("born") else 3.1 if k == "autograd2d" else 2.1
    return _wave_work(nd, phys, npad, c["nt"], c["nshot"], nrec, sweeps, not k.startswith("forward"))


# --- the same in float64, plain torch ----------------------------------------------------------------


class _Solver:
    """The leapfrog scheme in float64: fields [nshot][...padded] with a frame of four zero cells."""

    C = [-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0]

    def __init__(self, x):
        v = x["vel"].detach().double()
        self.nd, nb, h, dt, vref = v.dim(), x["nb"], x["h"], x["dt"], x["vref"]
        self.phys, self.nb, self.h, self.dt, self.nt, self.ns = v.shape, nb, h, dt, x["nt"], x["src"].shape[0]
        self.pad = tuple(n + 2 * nb for n in v.shape)
        self.src_of = [torch.arange(n + 2 * nb, device=DEV).sub(nb).clamp(0, n - 1) for n in v.shape]
        self.v = self.extend(v)
        depth = torch.zeros(self.pad, dtype=torch.float64, device=DEV)
        for a, n in enumerate(v.shape):
            i = torch.arange(n + 2 * nb, device=DEV)
            d = torch.maximum(nb - i, i - (nb + n - 1)).clamp(min=0).double()
            depth = torch.maximum(depth, d.reshape([-1 if b == a else 1 for b in range(self.nd)]))
        self.kap = (self.v * dt / h) ** 2
        if nb and vref > 0:
            gamma0 = 3.0 * vref * math.log(1000.0) / (2.0 * nb * h)
            eps = gamma0 * (depth / nb) ** 2 / vref ** 2 * dt * self.v ** 2 / 2.0
        else:
            eps = torch.zeros_like(depth)
        self.eps, self.inv = eps, 1.0 / (1.0 + eps)
        self.src, self.rec = self.taps(x["src"]), self.taps(x["rec"])

    def extend(self, a):
        for ax, i in enumerate(self.src_of):
            a = a.index_select(ax, i)
        return a

    def taps(self, xyz):
        """(flat padded index [ns][npts][2^nd], weight) of linear interpolation; axes of xyz are x, (y,) z."""
        p = torch.from_numpy(xyz).double().to(DEV) / self.h + self.nb
        pad = self.pad[::-1] if self.nd == 2 else (self.pad[2], self.pad[1], self.pad[0])
        lo = torch.stack([p[..., a].floor().long().clamp(max=pad[a] - 2) for a in range(self.nd)], -1)
        fr = p - lo
        idx, w = [], []
        for corner in range(1 << self.nd):
            bit = [(corner >> a) & 1 for a in range(self.nd)]
            c = [lo[..., a] + bit[a] for a in range(self.nd)]
            flat = c[-1]
            if self.nd == 3:
                flat = flat * pad[1] + c[1]
            idx.append(flat * pad[0] + c[0])
            ww = 1.0
            for a in range(self.nd):
                ww = ww * (fr[..., a] if bit[a] else 1.0 - fr[..., a])
            w.append(ww)
        return torch.stack(idx, -1), torch.stack(w, -1)

    def field(self):
        return torch.zeros((self.ns,) + tuple(n + 8 for n in self.pad), dtype=torch.float64, device=DEV)

    def core(self, u):
        return u[(slice(None),) + (slice(4, -4),) * self.nd]

    def step(self, u, um, source=None):
        """The next level from u and um (framed fields), written over um; returns um."""
        lap = self.core(u) * (self.nd * self.C[0])
        for k in range(1, 5):
            for a in range(self.nd):
                n = self.pad[a]
                at = [slice(None)] + [slice(4, -4)] * self.nd
                lo, hi = list(at), list(at)
                lo[a + 1], hi[a + 1] = slice(4 - k, 4 - k + n), slice(4 + k, 4 + k + n)
                lap.add_(u[tuple(lo)], alpha=self.C[k]).add_(u[tuple(hi)], alpha=self.C[k])
        lap.mul_(self.kap).add_(self.core(u), alpha=2.0)
        old = self.core(um)
        lap.addcmul_(self.eps - 1.0, old)
        if source is not None:
            lap.sub_(source)
        old.copy_(lap.mul_(self.inv))
        return um

    def spread(self, u, taps, fac, amp):
        """Adds fac w amp [ns][npts] at the taps."""
        idx, w = taps
        flat = idx.reshape(self.ns, -1)
        val = (w * fac.reshape(-1)[flat].reshape(w.shape) * amp[..., None]).reshape(self.ns, -1)
        inc = torch.zeros((self.ns, fac.numel()), dtype=torch.float64, device=DEV).scatter_add_(1, flat, val)
        self.core(u).add_(inc.reshape((self.ns,) + self.pad))

    def sample(self, u, taps):
        idx, w = taps
        flat = self.core(u).reshape(self.ns, -1).gather(1, idx.reshape(self.ns, -1))
        return (flat.reshape(w.shape) * w).sum(-1)

    def inject(self, u, q):
        self.spread(u, self.src, self.kap * self.h ** (2 - self.nd) * self.inv, q)

    def forward(self, q, data=None, first=0, last=None, state=None, levels=None):
        """Runs steps first..last-1 from state (u^first, u^{first-1}); fills data rows; stores levels[n - first]."""
        u, um = state if state is not None else (self.field(), self.field())
        for n in range(first, self.nt - 1 if last is None else last):
            self.step(u, um)
            u, um = um, u
            self.inject(u, q[:, n])
            if data is not None:
                data[:, n + 1] = self.sample(u, self.rec)
            if levels is not None:
                levels[n + 1 - first] = self.core(u)
        return u, um

    def pull(self, q, r, gradient, source):
        """J' r summed over shots (squared slowness) and F' r, for residuals r [ns][nt][nrec]."""
        K = self.nt - 1
        seg = max(1, int(math.sqrt(K)))
        states, cur = [], (self.field(), self.field())
        for a in range(0, K, seg) if gradient else []:
            states.append((cur[0].clone(), cur[1].clone()))
            cur = self.forward(q, None, a, min(K, a + seg), cur)
        del cur
        fac = self.kap * (self.h / self.dt) ** 2 * self.inv
        lam, lam2 = self.field(), self.field()  # mu^{k+1}, mu^{k+2}
        g = torch.zeros((self.ns,) + self.pad, dtype=torch.float64, device=DEV)
        out = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
        for a in reversed(range(0, K, seg)):
            b = min(K, a + seg)
            if gradient:
                levels = torch.empty((b - a + 1, self.ns) + self.pad, dtype=torch.float64, device=DEV)
                self.forward(q, None, a, b, states.pop(), levels)
            for k in range(b, a, -1):
                acc = self.core(lam2) - 2.0 * self.core(lam)
                self.step(lam, lam2)
                lam, lam2 = lam2, lam
                self.spread(lam, self.rec, fac, r[:, k])
                if gradient:
                    g.addcmul_(levels[k - a], acc.add_(self.core(lam)), value=-1.0)
                if source:
                    out[:, k - 1] = self.sample(lam, self.src) * (self.dt ** 2 / self.h ** self.nd)
        g = g.sum(0)
        for ax, i in enumerate(self.src_of):
            shape = list(g.shape)
            shape[ax] = self.phys[ax]
            g = torch.zeros(shape, dtype=torch.float64, device=DEV).index_add_(ax, i, g)
        return g, out

    def born(self, q, dm):
        data = torch.zeros((self.ns, self.nt, self.rec[0].shape[1]), dtype=torch.float64, device=DEV)
        dmv = self.extend(dm.double()) * self.v ** 2
        u, um, p, pm = self.field(), self.field(), self.field(), self.field()
        for n in range(self.nt - 1):
            src = self.core(um) - 2.0 * self.core(u)
            self.step(u, um)
            u, um = um, u
            self.inject(u, q[:, n])
            src.add_(self.core(u)).mul_(dmv)
            self.step(p, pm, src)
            p, pm = pm, p
            data[:, n + 1] = self.sample(p, self.rec)
        return data


def _gelu(x):
    return 0.5 * x * (1.0 + torch.erf(x / math.sqrt(2.0)))


def _layer64(v, W, b, R, mz, act):
    Nz, Nx = v.shape[-2:]
    mx = R.shape[-1]
    f = torch.fft.rfft2(v)
    X = torch.cat([f[..., :mz, :mx], f[..., Nz - mz:, :mx]], -2)
    Y = torch.einsum("bikx,iokx->bokx", X, R)
    S = torch.zeros(v.shape[:-3] + (W.shape[0], Nz, Nx // 2 + 1), dtype=torch.complex128, device=v.device)
    S[..., :mz, :mx], S[..., Nz - mz:, :mx] = Y[..., :mz, :], Y[..., mz:, :]
    # the truncated real inverse: w_0 = 1, w_kx = 2, real part over kept modes only
    x = torch.arange(Nx, device=v.device, dtype=torch.float64)
    ph = 2.0 * math.pi * torch.arange(mx, device=v.device, dtype=torch.float64)[:, None] * x[None] / Nx
    w = torch.where(torch.arange(mx, device=v.device) == 0, 1.0, 2.0).double()[:, None] / Nx
    z = torch.fft.ifft(S[..., :mx], dim=-2)
    y = z.real @ (w * torch.cos(ph)) - z.imag @ (w * torch.sin(ph))
    u = torch.einsum("oi,bihw->bohw", W, v) + b[None, :, None, None] + y
    return _gelu(u) if act else u


def _train64(c, seed):
    x, y, par = _train_inputs(c, seed)
    p = {k: v.double().requires_grad_(True) for k, v in par.items()}
    pw = lambda M, b, v: torch.einsum("oi,bihw->bohw", M, v) + b[None, :, None, None]  # noqa: E731
    v = pw(p["P"], p["p"], x.double())
    for l in range(c["layers"]):
        v = _layer64(v, p["W%d" % l], p["b%d" % l], torch.view_as_complex(p["R%d" % l]), c["mz"], l < c["layers"] - 1)
    out = pw(p["Q2"], p["q2"], _gelu(pw(p["Q1"], p["q1"], v)))
    loss = ((out - y.double()) ** 2).mean()
    grads = torch.autograd.grad(loss, list(p.values()))
    flat, flat_p = [], []
    for (name, w), g in zip(p.items(), grads):
        n = w.numel()
        zeros = torch.zeros((n + 3) // 4 * 4 - n, dtype=torch.float64, device=DEV)
        new = w.detach() - 1e-3 * g / (g.abs() + 1e-8)  # Adam's first step
        flat += [g.reshape(-1), zeros]
        flat_p += [new.reshape(-1), zeros]
    return {"loss": loss.detach(), "grads": torch.cat(flat), "params": torch.cat(flat_p)}


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "fno_layer":
        x = _layer_inputs(c, seed)
        return _layer64(x["v"].double(), x["W"].double(), x["b"].double(), torch.view_as_complex(x["R"].double()), c["mz"], True)
    if k == "fno_train":
        return _train64(c, seed)
    if k == "batch2d":
        mis, grads = [], []
        for i, x in enumerate(_batch_inputs(c, seed)):
            if i >= 4:  # the first four problems: all of them take minutes in 64 bits
                grads.append(None)
                continue
            s = _Solver(x)
            d = torch.zeros(x["d"].shape, dtype=torch.float64, device=DEV)
            s.forward(x["q"].double(), d)
            grads.append(s.pull(x["q"].double(), d - x["d"].double(), True, False)[0])
        return {"misfits": None, "grads": grads}
    x = _wave_inputs(c, seed)
    s = _Solver(x)
    q = x["q"].detach().double()
    if k == "born2d":
        return s.born(q, x["dm"])
    d = torch.zeros((s.ns, s.nt, x["rec"].shape[1]), dtype=torch.float64, device=DEV)
    s.forward(q, d)
    if k.startswith("forward"):
        return d
    if k == "autograd2d":
        r = x["d"].double()
        g, out = s.pull(q, r, True, True)
        return {"data": d, "g_vel": g * (-2.0 / x["vel"].detach().double() ** 3), "g_wavelet": out}
    r = d - x["d"].double()
    g, _ = s.pull(q, r, True, False)
    if c["velocity"]:
        g = g * (-2.0 / x["vel"].double() ** 3)
    return {"misfit": 0.5 * (r * r).sum(), "grad": g, "dsyn": d}
