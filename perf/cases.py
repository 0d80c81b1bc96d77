"""The work that users of the library have it do, as cases to time and compare.

Four kinds of call, over the sizes of the repository's own workloads (rings of 64 to 1024
transducers, grids of 96 to 512 nodes a side, the three precisions of the contractions):

  update   one Hessian-free update of a model from data: the whole call, ray tracing included,
           with the paper's options (frequency sets, absorption, integration on the non-smoothed
           map, ray linking) where the case says so
  batch    the sweeps of several uneven slices as one CUDA graph
  tables   one step of the update on given ray tables: the Born forward, the predicted data, an
           adjoint, or the update from the tables
  noalloc  the Born forward that allocates nothing, on the caller's tables

Inputs come from the seed alone: a phantom and its blurred initial model (phantoms), data with the
travel times of straight rays through the true phantom and 40 dB of noise, and, for the steps on
given tables, smooth tables close to those of a weakly varying medium, caustics included.

`exact` gives the steps on given tables in 64 bits. A whole update has no such value here: it would
be a second ray tracer.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2211_00316_gb300 import phantoms, rbx

PRECISION = {"fp32": rbx.RBX_FP32, "bf16": rbx.RBX_BF16, "bf16x3": rbx.RBX_BF16X3}
C0 = phantoms.C_WATER


# ------------------------------------------------------------------------------- the cases
def _case(kind, name=None, **k):
    c = {"kind": kind, **k}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the small two-disc problem: one update, where latency and launches count
        _case("update", "update_ring64_grid96_fp32", n=64, nx=96, ny=96, dx=1e-3, radius=45e-3, f=3e5, df=1e5,
              precision="fp32", nf=1, lossy=False, raw=False, link=0, phantom="discs"),
        # the plain FP32 form on the 256-transducer breast slice
        _case("update", "update_ring256_grid288_fp32", n=256, nx=288, ny=288, dx=0.8e-3, radius=110e-3, f=5e5, df=1e5,
              precision="fp32", nf=1, lossy=False, raw=False, link=0, phantom="breast"),
        # the headline workload: one update of the 1024-transducer, 512 x 512 slice
        _case("update", "update_ring1024_grid512_bf16", n=1024, nx=512, ny=512, dx=0.45e-3, radius=110e-3, f=5.05e5,
              df=5.8e4, precision="bf16", nf=1, lossy=False, raw=False, link=0, phantom="breast"),
        # the paper's own configuration on a medium slice: two frequencies per update, lossy medium,
        # integration on the non-smoothed map, linked rays
        _case("update", "set_ring512_grid256_lossy_linked_bf16", n=512, nx=256, ny=256, dx=0.59e-3, radius=70e-3, f=4e5,
              df=1e5, precision="bf16", nf=2, lossy=True, raw=True, link=8, phantom="breast"),
        # the batched form: uneven slices, their sweeps in one graph
        _case("batch", "batch_4_slices_bf16", slices=4, first=5, nf=2, f=1e5, df=1e5, precision="bf16"),
        # data generation: the predicted data of a 512-transducer slice in FP32
        _case("tables", "predict_ring512_grid288_fp32", call="predict", n=512, nx=288, ny=288, dx=0.76e-3, radius=104e-3,
              f=6e5, precision="fp32"),
        # the Born forward at the headline size
        _case("tables", "forward_ring1024_grid512_bf16", call="forward", n=1024, nx=512, ny=512, dx=0.45e-3,
              radius=110e-3, f=5e5, precision="bf16"),
        # the preconditioned back-projection of a large slice
        _case("tables", "adjoint_ring1024_grid384_bf16", call="preconditioned", n=1024, nx=384, ny=384, dx=0.61e-3,
              radius=112e-3, f=7e5, precision="bf16"),
        # the plain adjoint F* R (a functional gradient) of a 768-transducer slice
        _case("tables", "gradient_ring768_grid192_fp32", call="plain", n=768, nx=192, ny=192, dx=0.76e-3, radius=67e-3,
              f=8e5, precision="fp32"),
        # an update from tables already traced, split BF16
        _case("tables", "from_tables_ring768_grid320_bf16x3", call="update", n=768, nx=320, ny=320, dx=0.77e-3,
              radius=118e-3, f=3e5, precision="bf16x3"),
        # a ragged small problem: odd sizes, a grid that is not square, the update alone
        _case("tables", "from_tables_ring50_grid83x77_fp32", call="update", n=50, nx=83, ny=77, dx=1e-3, radius=36e-3,
              f=2.5e5, precision="fp32"),
        # the forward of callers that may not allocate (inside a graph capture, in a service)
        _case("noalloc", "noalloc_ring256_grid288_fp32", n=256, nx=288, ny=288, dx=0.8e-3, radius=110e-3, f=5e5),
    ]


def _nodes(c):
    return math.pi * (0.9 * c["radius"] / c["dx"]) ** 2


def _ms(c):
    """Roughly what a pass costs (ms), to keep drawn cases below the largest listed one."""
    if c["kind"] == "batch":
        geoms = [phantoms.batched_slice(c["first"] + s).geom for s in range(c["slices"])]
        return c["nf"] * sum(_ms({"kind": "update", "n": g.n_xducers, "radius": g.ring_radius, "dx": g.dx, "link": 0,
                                  "precision": c["precision"]}) for g in geoms)
    n, x = c["n"], _nodes(c)
    mac = n * n * x
    fp32 = mac * 8 / 35e9
    if c["kind"] == "noalloc":
        return 0.05 + fp32 * 2.2
    t = 0.0
    if c["kind"] == "update":
        steps = c["radius"] / c["dx"]
        t += 0.4 + 0.008 * steps + n * n * steps * 8e-8 * (3.0 if c["link"] else 1.0)
    per = {"predict": 0.5, "forward": 0.5, "preconditioned": 2.0, "plain": 1.0, "update": 2.5}[c.get("call", "update")]
    rate = 1.0 if c["precision"] == "fp32" or c.get("call") == "plain" else (0.12 if c["precision"] == "bf16x3" else 0.04)
    return t + c.get("nf", 1) * fp32 * per * rate


def _ring(rng, most_n=1024):
    """A ring and a grid that holds it, as the uneven slices draw them but over every size."""
    while True:
        n = int(round(math.exp(rng.uniform(math.log(48), math.log(most_n)))))
        nx = int(round(math.exp(rng.uniform(math.log(80), math.log(512)))))
        ny = nx if rng.random() < 0.6 else max(80, nx + rng.randrange(-24, 25))
        dx = rng.uniform(0.45e-3, 1.0e-3)
        radius = (min(nx, ny) - 1) * dx / 2 - 5e-3
        if radius > 12e-3:
            return {"n": n, "nx": nx, "ny": ny, "dx": dx, "radius": radius}


def draw(rng):
    while True:
        kind = rng.choice(["update", "update", "tables", "tables", "tables", "batch", "noalloc"])
        f = math.exp(rng.uniform(math.log(1e5), math.log(1.2e6)))
        if kind == "batch":
            c = _case("batch", slices=rng.randrange(1, 6), first=rng.randrange(3, 10), nf=rng.randrange(1, 3), f=1e5,
                      df=rng.uniform(5e4, 1.5e5), precision=rng.choice(["bf16", "bf16", "fp32"]))
        elif kind == "update":
            c = _case("update", **_ring(rng), f=f, df=rng.uniform(4e4, 1.2e5), precision=rng.choice(list(PRECISION)),
                      nf=rng.choice([1, 1, 2]), lossy=rng.random() < 0.25, raw=rng.random() < 0.25,
                      link=rng.choice([0, 0, 0, 8]), phantom="breast")
        elif kind == "tables":
            c = _case("tables", call=rng.choice(["predict", "forward", "preconditioned", "plain", "update"]), **_ring(rng),
                      f=f, precision=rng.choice(list(PRECISION)))
        else:
            c = _case("noalloc", **_ring(rng), f=f)
        if _ms(c) < 18.0:
            return c


# ------------------------------------------------------------------------------- inputs
def _geometry(c):
    df = c.get("df", 1e5)
    return phantoms.Geometry(nx=c["nx"], ny=c["ny"], dx=c["dx"], n_xducers=c["n"], ring_radius=c["radius"],
                             tau=phantoms.step_length(df))


def _generator(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _models(c, g, seed):
    """The true sound-speed map and the initial model of a job (ny x nx, numpy)."""
    if c.get("phantom") == "discs":
        r = np.random.default_rng(seed)
        s = c["radius"] / 45e-3
        centres = ((-15.0 * s + r.uniform(-4, 4), -5.0 * s + r.uniform(-4, 4)),
                   (14.0 * s + r.uniform(-4, 4), 10.0 * s + r.uniform(-4, 4)))
        true = phantoms.two_disc_phantom(g, centres, 8.0 * s, (r.uniform(0.02, 0.03), r.uniform(-0.03, -0.02)))
    else:
        true = phantoms.breast_phantom(g, seed)
    return true, phantoms.blur(true, g.dx)


def _data(g, true, freqs, seed):
    """Measured data of the true map, [nf][N][N] complex64: straight-ray travel times, 2-D
    spreading, 40 dB of noise, zero diagonal."""
    n = g.n_xducers
    dev, kw = "cuda", {"dtype": torch.float64, "device": "cuda"}
    th = 2 * math.pi * torch.arange(n, **kw) / n
    xy = g.ring_radius * torch.stack([th.cos(), th.sin()], -1)
    slow = torch.tensor(1.0 / true, dtype=torch.float32, device=dev)[None, None]
    half = torch.tensor([-g.x0, -g.y0], **kw)
    u = ((torch.arange(g.nx, **kw) + 0.5) / g.nx)[:, None]
    mean = torch.empty((n, n), **kw)
    rows = max(1, 2 ** 25 // (n * g.nx))
    for a in range(0, n, rows):
        p = xy[a:a + rows, None, None, :] * (1 - u) + xy[None, :, None, :] * u
        at = (p / half).reshape(1, -1, g.nx, 2).float()
        s = torch.nn.functional.grid_sample(slow, at, mode="bilinear", padding_mode="border", align_corners=True)
        mean[a:a + rows] = s.reshape(-1, n, g.nx).double().mean(-1)
    dist = torch.cdist(xy, xy)
    dist.fill_diagonal_(1.0)
    off = ~torch.eye(n, dtype=torch.bool, device=dev)
    out = torch.empty((len(freqs), n, n), dtype=torch.complex64, device=dev)
    gen = _generator(seed, 1)
    for k, f in enumerate(freqs):
        w = 2 * math.pi * f
        amp = (8 * math.pi * w * dist / g.c0) ** -0.5
        d = torch.polar(amp, w * mean * dist + math.pi / 4) * off
        sigma = 10 ** (-40 / 20) * float(amp[off].max()) / math.sqrt(2)
        noise = torch.randn((n, n, 2), generator=gen, **kw) * sigma
        out[k] = d + torch.view_as_complex(noise) * off
    return out


def _mask(c):
    x = -(c["nx"] - 1) * c["dx"] / 2.0 + c["dx"] * np.arange(c["nx"])
    y = -(c["ny"] - 1) * c["dx"] / 2.0 + c["dx"] * np.arange(c["ny"])
    X, Y = np.meshgrid(x, y)
    return torch.tensor(X, device="cuda"), torch.tensor(Y, device="cuda"), \
        torch.tensor(X * X + Y * Y <= (0.9 * c["radius"]) ** 2, device="cuda")


def _tables(c, seed):
    """Ray tables of a weakly varying medium: T, a, gamma, K [N][X] and exits [N][N-1][4]."""
    kw = {"dtype": torch.float64, "device": "cuda"}
    n, R = c["n"], c["radius"]
    X, Y, m = _mask(c)
    X, Y = X[m], Y[m]
    r = np.random.default_rng(seed)
    ph = [float(v) for v in r.uniform(0, 2 * math.pi, 6)]
    eps = float(r.uniform(0.005, 0.015))
    k = 2 * math.pi / R

    def slow(x, y, b):
        return (1 + eps * torch.sin(k * x + ph[0] + b) * torch.cos(k * y + ph[1])) / C0

    th = 2 * math.pi * torch.arange(n, **kw) / n
    nx = X.numel()
    T, a, gam = (torch.empty((n, nx), dtype=torch.float32, device="cuda") for _ in range(3))
    K = torch.empty((n, nx), dtype=torch.uint8, device="cuda")
    for e in range(n):
        b = th[e]
        dx, dy = X - R * torch.cos(b), Y - R * torch.sin(b)
        s = torch.sqrt(dx * dx + dy * dy)
        T[e] = (s * slow(X, Y, b)).float()
        a[e] = (s ** -0.5 * (1 + 10 * eps * torch.sin(k * (X - Y) + ph[2] + b))).float()
        g = torch.atan2(dy, dx) + 2 * eps * torch.sin(k * (X + Y) + ph[3] + b)
        gam[e] = torch.remainder(g + math.pi, 2 * math.pi).sub(math.pi).float()
        K[e] = ((s > 1.2 * R) & (torch.sin(3 * (torch.atan2(Y, X) - b) + ph[4]) > 0.6)).to(torch.uint8)
    j = torch.arange(1, n, **kw)
    step = 2 * math.pi / n
    rel = step * (j + 0.3 * torch.sin(2 * step * j + ph[5]))[None, :] + 0 * th[:, None]
    chord = 2 * R * torch.sin(rel / 2)
    ang = th[:, None] + rel
    ex, ey = R * torch.cos(ang), R * torch.sin(ang)
    far = (chord > 1.5 * R) & (torch.sin(2 * rel + ph[4]) > 0.5)
    exits = torch.stack([torch.atan2(ey, ex), chord * slow(ex, ey, th[:, None]), chord ** -0.5, far.double()], -1)
    return T, a, gam, K, exits.float().contiguous()


def _map(c, seed, salt, scale):
    """A smooth zero-mean map on the grid."""
    X, Y, _ = _mask(c)
    r = np.random.default_rng(1000003 * int(seed) + salt)
    out = torch.zeros_like(X)
    for _ in range(6):
        kx, ky = r.normal(0, 4 / c["radius"], 2)
        out += r.uniform(0.3, 1.0) * torch.sin(kx * X + ky * Y + r.uniform(0, 2 * math.pi))
    return (scale * out).float().contiguous()


def _table_inputs(c, seed):
    """What a step on given tables takes besides them: (model, dm, R or data)."""
    n = c["n"]
    X, Y, m = _mask(c)
    model = (C0 + _map(c, seed, 2, 12.0) * (X * X + Y * Y < (0.8 * c["radius"]) ** 2)).float().contiguous()
    dm = _map(c, seed, 3, 4e-9) * m
    pair = torch.randn((n, n, 2), generator=_generator(seed, 4), device="cuda") * \
        float((8 * math.pi * 2 * math.pi * c["f"] * c["radius"] / C0) ** -0.5)
    R = torch.view_as_complex(pair).contiguous()
    R.fill_diagonal_(0)
    return model, dm.float().contiguous(), R


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        jobs, models, data, freqs = [], [], [], []
        fr = [c["f"] + c["df"] * k for k in range(c["nf"])]
        for s in range(c["slices"]):
            w = phantoms.batched_slice(c["first"] + s)
            g = w.geom
            g.tau = phantoms.step_length(c["df"])
            true = phantoms.breast_phantom(g, 64 * seed + s)
            job = rbx.Job()
            job.set_geometry(g, precision=PRECISION[c["precision"]])
            jobs.append(job)
            models.append(torch.tensor(phantoms.blur(true, g.dx), dtype=torch.float32, device="cuda"))
            data.append(_data(g, true, fr, 64 * seed + s))
            freqs.append(np.array(fr))
        return {"c": c, "jobs": jobs, "models": models, "data": data, "freqs": freqs}
    if c["kind"] == "noalloc":
        T, a, _, K, _ = _tables(c, seed)
        _, _, m = _mask(c)
        v = ((2 * math.pi * c["f"]) ** 2 * c["dx"] ** 2 * _map(c, seed, 3, 4e-9)[m].double()).float().contiguous()
        return {"c": c, "T": T, "a": a, "K": K, "v": v}
    g = _geometry(c)
    job = rbx.Job()
    job.set_geometry(g, precision=PRECISION[c["precision"]])
    if c["kind"] == "tables":
        model, dm, R = _table_inputs(c, seed)
        job.set_model(model)
        job.set_tables(*_tables(c, seed))
        job.sync()
        return {"c": c, "job": job, "model": model, "dm": dm, "R": R}
    true, init = _models(c, g, seed)
    if c["lossy"]:
        job.set_absorption(torch.tensor(phantoms.absorption_map(true), dtype=torch.float32, device="cuda"))
    job.set_integration(c["raw"])
    job.set_linking(c["link"])
    freqs = [c["f"] + c["df"] * k for k in range(c["nf"])]
    return {"c": c, "job": job, "model": torch.tensor(init, dtype=torch.float32, device="cuda"), "freqs": freqs,
            "data": _data(g, true, freqs, seed)}


# ------------------------------------------------------------------------------- one pass
def _updated(job, st):
    return {"model": job.get_model(), "resid_norm2": st["resid_norm2"], "n_uncovered": st["n_uncovered"]}


def run(state):
    s, c = state, state["c"]
    if c["kind"] == "batch":
        for job, m in zip(s["jobs"], s["models"]):
            job.set_model(m)
        last, _ = rbx.batch_run(s["jobs"], s["freqs"], s["data"])
        return [_updated(job, st) for job, st in zip(s["jobs"], last)]
    if c["kind"] == "noalloc":
        n, nodes = s["T"].shape
        out = torch.empty((n, n), dtype=torch.complex64, device="cuda")
        err = ctypes.create_string_buffer(256)
        st = rbx.load().rbx_forward_noalloc(s["T"].data_ptr(), s["a"].data_ptr(), s["K"].data_ptr(), s["v"].data_ptr(),
                                            n, nodes, c["f"], C0, out.data_ptr(),
                                            torch.cuda.current_stream().cuda_stream or None, err, 256)
        if st != 0:
            raise rbx.RbxError(st, err.value.decode())
        return out
    job, f = s["job"], c["f"]
    if c["kind"] == "update":
        job.set_model(s["model"])
        if c["nf"] > 1:
            return _updated(job, job.update_set(s["freqs"], c["df"], s["data"]))
        return _updated(job, job.update_frequency(f, c["df"], s["data"]))
    if c["call"] == "predict":
        return job.predict(f)
    if c["call"] == "forward":
        return job.forward(f, s["dm"])
    if c["call"] in ("preconditioned", "plain"):
        return job.adjoint(f, s["R"], c["call"] == "preconditioned")
    job.set_model(s["model"])
    return _updated(job, job.update_from_tables(f, 1e5, s["R"]))


# ------------------------------------------------------------------------------- floors
def work(case):
    c = case
    if c["kind"] == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for s in range(c["slices"]):
            g = phantoms.batched_slice(c["first"] + s).geom
            w = work({"kind": "update", "n": g.n_xducers, "nx": g.nx, "ny": g.ny, "dx": g.dx, "radius": g.ring_radius,
                      "nf": 1, "raw": False})
            for k in total:
                total[k] += c["nf"] * w[k]
        return total
    n, x = c["n"], _nodes(c)
    grid, pairs = 4.0 * c["nx"] * c["ny"], 8.0 * n * n
    half, full = 4.0 * n * (n + 1) * x, 8.0 * n * n * x     # one symmetric, one general contraction
    if c["kind"] == "noalloc":
        return {"bytes": 9.0 * n * x + 4 * x + pairs, "flops": half}
    if c["kind"] == "update":
        # about 200 operations per step of a ray and its paraxial partner, mean chord 4 R / pi
        rays = 200.0 * n * (n - 1) * (4 / math.pi) * c["radius"] / (0.5 * c["dx"])
        return {"bytes": 2 * grid + c["nf"] * pairs, "flops": rays + c["nf"] * ((0 if c["raw"] else half) + 2 * full)}
    table = 16.0 * n * x
    flops = {"predict": half, "forward": half, "preconditioned": 2 * full, "plain": full, "update": half + 2 * full}
    moved = {"predict": grid + pairs, "forward": grid + pairs, "preconditioned": pairs + 8 * x, "plain": pairs + 8 * x,
             "update": 2 * grid + pairs}
    return {"bytes": table + moved[c["call"]], "flops": flops[c["call"]]}


# ------------------------------------------------------------------------------- in 64 bits
def _green(T, a, K, f):
    w = 2 * math.pi * f
    cyc = f * T.double() - 0.25 * K.double() + 0.125
    return torch.polar((8 * math.pi * w / C0) ** -0.5 * a.double(), 2 * math.pi * torch.remainder(cyc, 1.0))


def _direct(exits, f):
    """Direct Green's function: T and a interpolated in exit angle to each receiver."""
    n = exits.shape[0]
    ex = exits.double()
    step = 2 * math.pi / n
    e = torch.arange(n, device="cuda")
    th = torch.remainder(ex[..., 0] - step * e[:, None], 2 * math.pi).contiguous()
    at = (step * torch.arange(1, n, dtype=torch.float64, device="cuda")).expand(n, n - 1).contiguous()
    hi = torch.searchsorted(th, at)
    near = (hi == 0) | (hi == n - 1)
    hi = hi.clamp(1, n - 2)
    lo = hi - 1
    ta, tb = th.gather(1, lo), th.gather(1, hi)
    fr = (at - ta) / (tb - ta)
    fr = torch.where(near, (fr > 0.5).double(), fr)

    def mid(q):
        return torch.lerp(ex[..., q].gather(1, lo), ex[..., q].gather(1, hi), fr)

    K = torch.where(fr < 0.5, ex[..., 3].gather(1, lo), ex[..., 3].gather(1, hi))
    g = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
    to = torch.remainder(e[:, None] + torch.arange(1, n, device="cuda"), n)
    return g.scatter_(1, to, _green(mid(1), mid(2), K, f))


def _window(f, dx):
    w = 13.0 if f < 0.4e6 else 11.0 if f < 0.7e6 else 9.0 if f < 1.0e6 else 7.0
    return 2 * max(0, math.floor((w * (1e-3 / dx) - 1) / 2 + 0.5)) + 1


def _rough(model, f, dx):
    """m - m_s: squared slowness less that of the smoothed slowness."""
    w = _window(f, dx)
    n = 1.0 / model.double()
    p = torch.nn.functional.pad(n[None, None], (w // 2,) * 4, mode="replicate")
    return n * n - torch.nn.functional.avg_pool2d(p, w, stride=1)[0, 0] ** 2


def _born(G, v):
    return (G * v) @ G.T


def exact(case, seed):
    c = case
    if c["kind"] in ("update", "batch"):
        return None
    f, w, dA = c["f"], 2 * math.pi * c["f"], c["dx"] ** 2
    T, a, gam, K, exits = _tables(c, seed)
    _, _, m = _mask(c)
    G = _green(T, a, K, f)
    if c["kind"] == "noalloc":
        v = (w ** 2 * dA * _map(c, seed, 3, 4e-9)[m].double()).float()
        return _born(G, v.double())
    model, dm, R = _table_inputs(c, seed)
    if c["call"] == "forward":
        return _born(G, w * w * dA * dm.double()[m])
    if c["call"] in ("predict", "update"):
        g = _born(G, w * w * dA * _rough(model, f, c["dx"])[m]) + _direct(exits, f)
        g.fill_diagonal_(0)
        if c["call"] == "predict":
            return g
        R = g - R.to(torch.complex128)
        norm2 = float(R.abs().square().sum())
    R = R.to(torch.complex128)
    R = 0.5 * (R + R.T)
    if c["call"] == "plain":
        G = G.conj().resolve_conj()
        return w * w * dA * ((R @ G) * G).sum(0)
    d = gam.double().roll(-1, 0) - gam.double().roll(1, 0)
    d = 0.5 * (torch.remainder(d + math.pi, 2 * math.pi) - math.pi).abs()
    U = d / G
    del G
    kap = torch.polar(torch.ones_like(d), gam.double())
    grad = ((R @ U) * U).sum(0)
    U *= kap
    grad -= ((R @ (U * kap.conj().square())) * U).sum(0)
    grad *= 2
    if c["call"] == "preconditioned":
        return grad
    m0 = 1.0 / model.double()[m].square()
    step = -(2 * math.pi * 1e5 / (2 * math.pi) ** 3) * (m0 / w) * grad.real
    out = torch.full(model.shape, C0, dtype=torch.float64, device="cuda")
    out[m] = (m0 + phantoms.step_length(1e5) * step).rsqrt()
    return {"model": out, "resid_norm2": norm2, "n_uncovered": None}
