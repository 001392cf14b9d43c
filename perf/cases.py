"""Performance cases: what programs built on this library have it compute, from a
delay-and-sum image of a 64 x 64 frame to a 128^3 volume.

``listed()`` names fixed cases, ``draw(rng)`` gives further ones of the same
ranges.  ``prepare`` makes what a program holds before the call (the plan, the
measured traces, start images), ``run`` is one call through the public entry
points, ``exact`` the same result in plain FP64 torch, and ``work`` the bytes and
operations that one call cannot do without.

Every case is a dict of plain values.  Geometry: ``dim``, ``nx``/``ny``/``nz``
pixels of ``h`` metres, ``layout`` (ring, linear or planar array of ``sensors``),
``K`` samples at ``fs``.  ``kind`` selects the call.
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

C0 = 1500.0  # m/s
FS = 40e6    # Hz
CHUNK_PAIRS = 1 << 24  # (sensor, pixel) pairs per FP64 block of the exact operators


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _case(kind, name=None, **kw):
    c = {"kind": kind, "dim": 2, "nx": 256, "ny": 256, "nz": 1, "h": 1e-4, "layout": "ring",
         "sensors": 256, "K": 2048, "fs": FS, "t0_samples": 0.0, "y16": False}
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # live preview while scanning: one filtered back-projection of a small
        # linear-array frame, where latency and launches are all there is
        _case("backproject", "bp_64_linear64", nx=64, ny=64, layout="linear", sensors=64, K=512),
        # simulation of the traces of one frame; also the A of any solver that the
        # program writes itself
        _case("forward", "forward_256_ring256"),
        # delay-and-sum of a frame of odd size, fewer sensors, 1-based time axis
        _case("adjoint", "adjoint_301x187_ring173", nx=301, ny=187, sensors=173, K=1501,
              t0_samples=1.0),
        # the normal operator's two halves on a volume: A x and A^T r (the largest case)
        _case("volume", "volume_128_planar1024", dim=3, nx=128, ny=128, nz=128, h=2e-4,
              layout="planar", sensors=1024, K=1024),
        # reconstruction of one frame, stopped before noise is fitted
        _case("cgls", "cgls5_256_ring256", iters=5),
        # the full objective (data, L1 and TV terms) on one frame
        _case("fista", "fista20_256_ring256", iters=20),
        # a time series of frames of uneven size, FP16 traces, in one batch
        _case("batch", "batch16_ragged_landweber10", frames=16, mix=4, iters=10, y16=True,
              method="landweber"),
        # a training batch: loss and its gradients in the images and in the speed of sound
        _case("fit", "fit8_256_ring128", frames=8, sensors=128, speeds=1),
        # calibration of the speed of sound: loss and gradients of one frame at
        # successive candidate speeds
        _case("fit", "calibrate3_256_ring128", frames=1, sensors=128, speeds=3),
        # an unrolled reconstruction network, forward and backward
        _case("unroll", "unroll4_200_ring128_4", nx=200, ny=200, sensors=128, K=1600, frames=4,
              iters=4),
        # the frequency-domain model: spectra of a frame and the gradient of the data term
        _case("freq", "freq256_256_ring256", freqs=256, df=78125.0),
        # the dense-matrix mode at the size of the published experiment, both products
        _case("dense", "dense_6144x16384_f64", nx=128, ny=128, sensors=48, K=128, fs=10e6,
              wide=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["backproject", "forward", "adjoint", "volume", "cgls", "fista", "batch",
                       "fit", "unroll", "freq", "dense"])
    nx = _log_int(rng, 48, 480)
    ny = max(32, int(nx * rng.uniform(0.6, 1.2)))
    sensors = _log_int(rng, 48, 480)
    layout = rng.choice(["ring", "ring", "linear"])
    # enough samples for the farthest pixel, or fewer (the traces are cut off)
    K = int((2.2 * max(nx, ny) * 1e-4 + 4e-3) * FS / C0 * rng.uniform(0.7, 1.1))
    geo = dict(nx=nx, ny=ny, sensors=sensors, layout=layout, K=K,
               t0_samples=rng.choice([0.0, 0.0, 1.0, 12.5]))
    if kind in ("backproject", "forward", "adjoint"):
        return _case(kind, **geo)
    if kind == "volume":
        n = _log_int(rng, 40, 120)
        s = _log_int(rng, 8, 30)
        return _case("volume", dim=3, nx=n, ny=max(24, int(n * rng.uniform(0.7, 1.1))),
                     nz=max(24, int(n * rng.uniform(0.6, 1.0))), h=2e-4, layout="planar",
                     sensors=s * s, K=rng.randint(400, 1024))
    if kind == "cgls":
        return _case("cgls", iters=rng.randint(3, 5), **dict(geo, y16=rng.random() < 0.3))
    if kind == "fista":
        return _case("fista", iters=rng.randint(8, 30), **geo)
    if kind == "batch":
        method = rng.choice(["landweber", "cgls"])
        return _case("batch", frames=rng.randint(4, 20), mix=rng.randrange(1 << 20),
                     iters=rng.randint(3, 10) if method == "landweber" else rng.randint(3, 5),
                     y16=rng.random() < 0.7, method=method)
    if kind == "fit":
        speeds = rng.choice([1, 1, 2])
        geo.update(nx=min(nx, 300), ny=min(ny, 300), sensors=min(sensors, 256), layout="ring",
                   t0_samples=0.0)
        return _case("fit", frames=rng.randint(1, 8), speeds=speeds, **geo)
    if kind == "unroll":
        geo.update(nx=min(nx, 220), ny=min(ny, 220), sensors=min(sensors, 200), layout="ring",
                   t0_samples=0.0)
        return _case("unroll", frames=rng.randint(1, 5), iters=rng.randint(2, 5), **geo)
    if kind == "freq":
        geo.update(nx=min(nx, 320), ny=min(ny, 320), sensors=min(sensors, 300))
        q = _log_int(rng, 24, 300)
        return _case("freq", freqs=q, df=20e6 / q, **geo)
    nx, s, k = rng.choice([64, 96, 100, 128]), rng.randint(24, 64), rng.randint(80, 160)
    return _case("dense", nx=nx, ny=rng.choice([nx, nx - 3]), sensors=s, K=k, fs=10e6,
                 wide=rng.random() < 0.6)


# ---------------------------------------------------------------------------
# geometry and inputs
# ---------------------------------------------------------------------------
def _geometry(case):
    shape = (case["nx"], case["ny"], case["nz"])
    h, n = case["h"], case["sensors"]
    spacing = (h, h, h)
    origin = tuple(-(m - 1) / 2.0 * h for m in shape)
    if case["layout"] == "ring":
        # outside the frame's corners by 2 mm
        r = 0.5 * h * math.hypot(shape[0], shape[1]) + 2e-3
        th = 2.0 * np.pi * np.arange(n) / n
        sens = np.stack([r * np.cos(th), r * np.sin(th)], axis=1)
    elif case["layout"] == "linear":
        # spans the frame's width, 2 mm above it
        pitch = 1.5 * shape[0] * h / n
        xs = (np.arange(n) - (n - 1) / 2.0) * pitch
        sens = np.stack([xs, np.full(n, 0.5 * shape[1] * h + 2e-3)], axis=1)
    else:
        # square planar array over the volume's top face, 5 mm above it
        m = int(round(math.sqrt(n)))
        xs = (np.arange(m) - (m - 1) / 2.0) * (shape[0] * h / m)
        gy, gx = np.meshgrid(xs, xs, indexing="ij")
        sens = np.stack([gx.ravel(), gy.ravel(), np.full(m * m, 0.5 * shape[2] * h + 5e-3)], axis=1)
    return SimpleNamespace(dim=case["dim"], shape=shape, spacing=spacing, origin=origin,
                           sensors=sens, c=C0, fs=case["fs"], K=case["K"],
                           t0=case["t0_samples"] / case["fs"], S=sens.shape[0],
                           N=shape[0] * shape[1] * shape[2])


def _frame_cases(case):
    """The frames of a batch: grids of 128 to 384 pixels a side (or one of odd size),
    128 to 400 sensors, 1024 to 3000 samples."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["frames"]):
        n = rng.choice([128, 192, 256, 384, 250])
        out.append(_case("frame", nx=n, ny=n, sensors=rng.randint(128, 400),
                         K=rng.randint(1024, 3000), y16=case["y16"]))
    return out


def _pixels(geo, device):
    ax = [torch.arange(m, dtype=torch.float64, device=device) * h + o
          for m, h, o in zip(geo.shape, geo.spacing, geo.origin)]
    gz, gy, gx = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    pts = [gx.reshape(-1), gy.reshape(-1), gz.reshape(-1)]
    return torch.stack(pts[:geo.dim], dim=1)


def _vessels(geo, gen, device, n=14):
    """Vessels: straight tubes of random place, width and amplitude; most of the
    image is zero."""
    pts = _pixels(geo, device)
    ext = torch.tensor([m * h for m, h in zip(geo.shape, geo.spacing)][:geo.dim],
                       dtype=torch.float64, device=device)
    u = torch.rand((n, 2, geo.dim), generator=gen, device=device, dtype=torch.float64)
    ends = (u - 0.5) * ext
    width = (0.6 + 2.4 * torch.rand(n, generator=gen, device=device, dtype=torch.float64)) * geo.spacing[0]
    amp = 0.5 + 0.5 * torch.rand(n, generator=gen, device=device, dtype=torch.float64)
    img = torch.zeros(pts.shape[0], dtype=torch.float64, device=device)
    for i in range(n):
        a, b = ends[i, 0], ends[i, 1]
        v = b - a
        t = ((pts - a) @ v / (v @ v).clamp_min(1e-30)).clamp(0.0, 1.0)
        dist = (pts - a - t[:, None] * v).norm(dim=1)
        img = torch.where(dist <= width[i], torch.maximum(img, amp[i]), img)
    return img.to(torch.float32)


def _iterate(geo, gen, device):
    """An image as it stands inside a solver: vessels over a dense, noisy background."""
    return (_vessels(geo, gen, device)
            + 0.05 * torch.randn(geo.N, generator=gen, device=device)).contiguous()


def _residual(geo, gen, device, frames=None):
    """Traces as a solver back-projects them: noise over a few samples' bandwidth."""
    shape = (geo.S, geo.K + 2) if frames is None else (frames, geo.S, geo.K + 2)
    w = torch.randn(shape, generator=gen, device=device)
    return (0.25 * w[..., :-2] + 0.5 * w[..., 1:-1] + 0.25 * w[..., 2:]).contiguous()


def _measured(geo, x, gen, c=None, half=False):
    """y = A x plus 1% noise (and FP16 storage), A in FP64."""
    p = _A(geo, x.double(), c)
    p = p + 0.01 * p.abs().max() * torch.randn(p.shape, generator=gen, device=p.device,
                                               dtype=torch.float64)
    return p.to(torch.float16 if half else torch.float32).contiguous()


def _step_bound(geo, device):
    """An upper bound of the largest eigenvalue of A^T A: ||A||_1 ||A||_inf."""
    rows = _A(geo, torch.ones(geo.N, dtype=torch.float64, device=device)).max()
    cols = _At(geo, torch.ones((geo.S, geo.K), dtype=torch.float64, device=device)).max()
    return float(rows * cols)


def _plan(geo, y16=False):
    from paper_2404_10928_gb300.api import Plan
    return Plan(geo.sensors, geo.shape, geo.spacing, geo.origin, geo.c, geo.fs, geo.K, t0=geo.t0,
                y_dtype="f16" if y16 else "f32", dim=geo.dim)


def _inputs(case, seed):
    """The case's inputs (no plan): what prepare() and exact() share."""
    device = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=device)
    gen.manual_seed(int(seed) * 7919 + 17)
    kind = case["kind"]
    s = SimpleNamespace(kind=kind, case=case)
    if kind == "batch":
        s.geos = [_geometry(f) for f in _frame_cases(case)]
        s.ys = [_measured(g, _vessels(g, gen, device), gen, half=case["y16"]) for g in s.geos]
        s.omegas = [1.0 / _step_bound(g, device) for g in s.geos]
        return s
    geo = s.geo = _geometry(case)
    if kind in ("backproject", "adjoint"):
        s.p = _residual(geo, gen, device)
    elif kind == "forward":
        s.x = _iterate(geo, gen, device)
    elif kind == "volume":
        s.x = _iterate(geo, gen, device)
        s.p = _residual(geo, gen, device)
    elif kind == "cgls":
        s.y = _measured(geo, _vessels(geo, gen, device), gen, half=case["y16"])
    elif kind == "fista":
        s.y = _measured(geo, _vessels(geo, gen, device), gen)
        lam = _step_bound(geo, device)
        s.eps = 1e-2
        s.l1 = 1e-3 * float(_At(geo, s.y.double()).abs().max())
        s.tv = 0.01 * lam * s.eps
        s.tau = 1.0 / (2.0 * lam + 8.0 * s.tv / s.eps)
    elif kind == "fit":
        xs = [_vessels(geo, gen, device) for _ in range(case["frames"])]
        s.y = torch.stack([_measured(geo, x, gen, c=1540.0) for x in xs])
        s.x = torch.stack(xs) + 0.05 * torch.randn((len(xs), geo.N), generator=gen, device=device)
        s.speeds = [1500.0, 1520.0, 1540.0][:case["speeds"]]
        s.tv, s.eps = 1e-3, 1e-2
    elif kind == "unroll":
        # soft tissue: a positive background everywhere, vessels on top
        xs = [0.4 + 0.5 * _vessels(geo, gen, device) for _ in range(case["frames"])]
        s.target = torch.stack(xs)
        s.y = torch.stack([_measured(geo, x, gen) for x in xs])
        s.x0 = 0.5 + 0.02 * torch.randn((len(xs), geo.N), generator=gen, device=device)
        s.omega = 0.5 / _step_bound(geo, device)
    elif kind == "freq":
        s.x = _iterate(geo, gen, device)
        re, im = (torch.randn((geo.S, case["freqs"]), generator=gen, device=device) for _ in range(2))
        s.spec = torch.complex(re, im) * 1e6
    elif kind == "dense":
        dt = torch.float64 if case["wide"] else torch.float32
        s.v = _iterate(geo, gen, device).to(dt)
        s.r = _residual(geo, gen, device).reshape(-1).to(dt)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = s.kind
    if kind == "batch":
        from paper_2404_10928_gb300.api import Batch
        s.plans = [_plan(g, case["y16"]) for g in s.geos]
        s.batch = Batch(s.plans)
        s.xs = [torch.zeros(g.N, device=y.device) for g, y in zip(s.geos, s.ys)]
        return s
    s.plan = _plan(s.geo, case["y16"])
    if kind in ("cgls", "fista"):
        s.out = torch.zeros(s.geo.N, device=s.y.device)  # the frame's image buffer
    elif kind == "unroll":
        from paper_2404_10928_gb300.autograd import UnrolledLandweber
        s.net = UnrolledLandweber(s.plan, case["iters"], s.omega)
    elif kind == "dense":
        s.m = s.plan.dense_assemble(s.v.dtype)
    return s


def run(s):
    kind, case = s.kind, s.case
    if kind == "backproject":
        return s.plan.backproject(s.p, "ubp")
    if kind == "forward":
        return s.plan.forward(s.x)
    if kind == "adjoint":
        return s.plan.adjoint(s.p)
    if kind == "volume":
        return {"p": s.plan.forward(s.x), "g": s.plan.adjoint(s.p)}
    if kind == "cgls":
        s.out.zero_()
        return s.plan.reconstruct(s.y, "cgls", case["iters"], out=s.out)
    if kind == "fista":
        s.out.zero_()
        return s.plan.reconstruct(s.y, "fista", case["iters"], out=s.out, omega=s.tau, l1=s.l1,
                                  tv=s.tv, tv_eps=s.eps)
    if kind == "batch":
        torch._foreach_zero_(s.xs)
        s.batch.reconstruct(s.ys, s.xs, case["method"], case["iters"],
                            omegas=s.omegas if case["method"] == "landweber" else None)
        return s.xs
    if kind == "fit":
        from paper_2404_10928_gb300.autograd import data_tv_loss
        out = []
        for c0 in s.speeds:
            x = s.x.detach().requires_grad_(True)
            c = torch.tensor(c0, device=s.x.device, requires_grad=True)
            loss = data_tv_loss(s.plan, x, c, s.y, s.tv, s.eps)
            loss.backward()
            out.append({"loss": loss.detach().float(), "x": x.grad, "c": c.grad})
        return out
    if kind == "unroll":
        x0 = s.x0.detach().requires_grad_(True)
        c = torch.tensor(C0, device=s.x0.device, requires_grad=True)
        xn = s.net(x0, s.y, c)
        loss = torch.nn.functional.mse_loss(xn, s.target)
        loss.backward()
        return {"xn": xn.detach(), "loss": loss.detach(), "x": x0.grad, "c": c.grad}
    if kind == "freq":
        q, df = case["freqs"], case["df"]
        return {"p": s.plan.freq_forward(s.x, q, df, df), "g": s.plan.freq_adjoint(s.spec, q, df, df)}
    if kind == "dense":
        return {"p": s.plan.dense_matvec(s.m, s.v), "g": s.plan.dense_matvec(s.m, s.r, transpose=True)}
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: each input read and each output written once.  Flops: 18 per (pixel,
    sensor) pair and application of A, A^T or the derivative in c (nine fused
    multiply-adds: squared distance, arrival, weight, interpolation), 4 per
    (pixel, sensor, frequency) term, 2 per matrix entry."""
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        apps = 2 * case["iters"] + (1 if case["method"] == "landweber" else 2)
        for g in map(_geometry, _frame_cases(case)):
            b += g.S * g.K * (2 if case["y16"] else 4) + 4 * g.N
            f += 18.0 * apps * g.S * g.N
        return {"bytes": b, "flops": f}
    g = _geometry(case)
    pairs, tr, img = float(g.S) * g.N, 4.0 * g.S * g.K, 4.0 * g.N
    if kind in ("backproject", "forward", "adjoint"):
        return {"bytes": tr + img, "flops": 18.0 * pairs}
    if kind == "volume":
        return {"bytes": 2 * (tr + img), "flops": 36.0 * pairs}
    if kind == "cgls":
        return {"bytes": tr * (0.5 if case["y16"] else 1.0) + img,
                "flops": 18.0 * pairs * (2 * case["iters"] + 2)}
    if kind == "fista":
        return {"bytes": tr + img, "flops": 18.0 * pairs * (2 * case["iters"] + 1)}
    if kind == "fit":  # A, A^T and the derivative in c
        n = case["frames"] * case["speeds"]
        return {"bytes": n * (tr + 2 * img), "flops": n * 54.0 * pairs}
    if kind == "unroll":  # per step A and A^T; backward A, A^T, A and two derivatives in c
        n = case["frames"]
        return {"bytes": n * (tr + 4 * img), "flops": n * case["iters"] * 7 * 18.0 * pairs}
    if kind == "freq":
        return {"bytes": 2 * (8.0 * g.S * case["freqs"] + img),
                "flops": 2 * 4.0 * pairs * case["freqs"]}
    e = 8.0 if case["wide"] else 4.0
    return {"bytes": 2 * e * g.S * g.K * g.N, "flops": 4.0 * g.S * g.K * g.N}


# ---------------------------------------------------------------------------
# the same results in FP64
# ---------------------------------------------------------------------------
def _blocks(geo, c, device):
    """Blocks of sensors: (slice, 1/d, tap index, fraction), each [sensors][N]."""
    pts = _pixels(geo, device)
    sens = torch.tensor(geo.sensors, dtype=torch.float64, device=device)
    step = max(1, CHUNK_PAIRS // geo.N)
    c = geo.c if c is None else c
    for a in range(0, geo.S, step):
        sl = slice(a, min(geo.S, a + step))
        d2 = torch.zeros((sl.stop - a, geo.N), dtype=torch.float64, device=device)
        for j in range(geo.dim):
            d2 += (pts[None, :, j] - sens[sl, None, j]) ** 2
        d = d2.sqrt_()
        u = d * (geo.fs / c) - geo.t0 * geo.fs
        k0 = torch.floor(u)
        yield sl, 1.0 / d, k0.to(torch.int64), u - k0


def _A(geo, x, c=None):
    p = torch.zeros((geo.S, geo.K + 2), dtype=torch.float64, device=x.device)
    for sl, w, k0, f in _blocks(geo, c, x.device):
        w = w * x[None, :]
        # columns 0 and K + 1 take the taps outside the trace
        p[sl].scatter_add_(1, (k0 + 1).clamp(0, geo.K + 1), w * (1.0 - f))
        p[sl].scatter_add_(1, (k0 + 2).clamp(0, geo.K + 1), w * f)
    return p[:, 1:-1].contiguous()


def _taps(p, k0, geo, sl):
    pp = torch.nn.functional.pad(p[sl], (1, 1))
    lo = pp.gather(1, (k0 + 1).clamp(0, geo.K + 1))
    return lo, pp.gather(1, (k0 + 2).clamp(0, geo.K + 1))


def _At(geo, p, c=None):
    g = torch.zeros(geo.N, dtype=torch.float64, device=p.device)
    for sl, w, k0, f in _blocks(geo, c, p.device):
        lo, hi = _taps(p, k0, geo, sl)
        g += (w * ((1.0 - f) * lo + f * hi)).sum(0)
    return g


def _dc(geo, x, p, c):
    total = 0.0
    for sl, _, k0, _ in _blocks(geo, c, p.device):
        lo, hi = _taps(p, k0, geo, sl)
        total = total + ((hi - lo) * x[None, :]).sum()
    return -total * geo.fs / (c * c)


def _tv_grad(geo, x, eps):
    img = x.reshape(geo.shape[2], geo.shape[1], geo.shape[0])
    d = [torch.zeros_like(img) for _ in range(2)]
    d[0][:, :, :-1] = img[:, :, 1:] - img[:, :, :-1]
    d[1][:, :-1] = img[:, 1:] - img[:, :-1]
    m = (d[0] ** 2 + d[1] ** 2 + eps * eps).sqrt()
    a, b = d[0] / m, d[1] / m
    g = -(a + b)
    g[:, :, 1:] += a[:, :, :-1]
    g[:, 1:] += b[:, :-1]
    return g.reshape(-1), m.sum()


def _exact_cgls(geo, y, iters):
    x = torch.zeros(geo.N, dtype=torch.float64, device=y.device)
    r = y.double()
    s = _At(geo, r)
    p, gamma = s, s @ s
    for _ in range(iters):
        q = _A(geo, p)
        alpha = gamma / (q * q).sum()
        x, r = x + alpha * p, r - alpha * q
        s = _At(geo, r)
        new = s @ s
        p, gamma = s + (new / gamma) * p, new
    return x.clamp_min(0.0)


def _exact_landweber(geo, y, iters, omega):
    x = torch.zeros(geo.N, dtype=torch.float64, device=y.device)
    for _ in range(iters):
        x = (x + omega * _At(geo, y.double() - _A(geo, x))).clamp_min(0.0)
    return x


def _exact_fista(geo, s, iters):
    x = torch.zeros(geo.N, dtype=torch.float64, device=s.y.device)
    z, t = x, 1.0
    for _ in range(iters):
        grad = -2.0 * _At(geo, s.y.double() - _A(geo, z)) + s.tv * _tv_grad(geo, z, s.eps)[0]
        new = (z - s.tau * grad - s.tau * s.l1).clamp_min(0.0)
        tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        z, x, t = new + ((t - 1.0) / tn) * (new - x), new, tn
    return x


def _exact_fit(geo, s, c):
    loss, gx, gc = 0.0, [], 0.0
    for x, y in zip(s.x.double(), s.y.double()):
        r = y - _A(geo, x, c)
        tg, tv = _tv_grad(geo, x, s.eps)
        loss = loss + (r * r).sum() + s.tv * tv
        gx.append(-2.0 * _At(geo, r, c) + s.tv * tg)
        gc = gc - 2.0 * _dc(geo, x, r, c)
    return {"loss": loss, "x": torch.stack(gx), "c": gc}


def _exact_unroll(geo, s, iters):
    n, om = s.x0.numel(), s.omega
    loss, xn, gx, gc = 0.0, [], [], 0.0
    for x0, y, target in zip(s.x0.double(), s.y.double(), s.target.double()):
        xs, zs, rs = [x0], [], []
        for _ in range(iters):
            r = y - _A(geo, xs[-1])
            z = xs[-1] + om * _At(geo, r)
            rs.append(r)
            zs.append(z)
            xs.append(z.clamp_min(0.0))
        loss = loss + ((xs[-1] - target) ** 2).sum() / n
        lam = 2.0 * (xs[-1] - target) / n
        for k in reversed(range(iters)):
            gz = lam * (zs[k] > 0)
            q = _A(geo, gz)
            gc = gc + om * (_dc(geo, gz, rs[k], geo.c) - _dc(geo, xs[k], q, geo.c))
            lam = gz - om * _At(geo, q)
        xn.append(xs[-1])
        gx.append(lam)
    return {"xn": torch.stack(xn), "loss": loss, "x": torch.stack(gx), "c": gc}


def _exact_freq(geo, s, q, df):
    p = torch.zeros((geo.S, q), dtype=torch.complex128, device=s.x.device)
    g = torch.zeros(geo.N, dtype=torch.float64, device=s.x.device)
    pts = _pixels(geo, s.x.device)
    sens = torch.tensor(geo.sensors, dtype=torch.float64, device=s.x.device)
    f = df * (1.0 + torch.arange(q, dtype=torch.float64, device=s.x.device))
    x, spec = s.x.double(), s.spec.to(torch.complex128)
    step = max(1, CHUNK_PAIRS // geo.N)
    for m in range(geo.S):
        d = (pts - sens[m]).norm(dim=1)
        for a in range(0, q, step):
            sl = slice(a, min(q, a + step))
            ph = torch.polar(torch.ones((), dtype=torch.float64, device=d.device),
                             (2.0 * math.pi / geo.c) * f[sl, None] * d[None, :])  # exp(+i k d)
            ck = 2.0 * math.pi * f[sl]
            w = (x / d).to(torch.complex128)
            p[m, sl] = 1j * ck * (ph.conj() @ w)
            g += ((ck * spec[m, sl]) @ ph).imag / d
    return {"p": p.to(torch.complex128), "g": g}


def exact(case, seed):
    s = _inputs(case, seed)
    kind = s.kind
    if kind == "batch":
        if case["method"] == "cgls":
            return [_exact_cgls(g, y, case["iters"]) for g, y in zip(s.geos, s.ys)]
        return [_exact_landweber(g, y, case["iters"], om)
                for g, y, om in zip(s.geos, s.ys, s.omegas)]
    geo = s.geo
    if kind == "backproject":
        p = s.p.double()
        pad = torch.nn.functional.pad(p, (1, 1))
        k = torch.arange(geo.K, dtype=torch.float64, device=p.device)
        b = 2.0 * p - (geo.t0 * geo.fs + k) * (pad[:, 2:] - pad[:, :-2])
        return _At(geo, b)
    if kind == "forward":
        return _A(geo, s.x.double())
    if kind == "adjoint":
        return _At(geo, s.p.double())
    if kind == "volume":
        return {"p": _A(geo, s.x.double()), "g": _At(geo, s.p.double())}
    if kind == "cgls":
        return _exact_cgls(geo, s.y, case["iters"])
    if kind == "fista":
        return _exact_fista(geo, s, case["iters"])
    if kind == "fit":
        return [_exact_fit(geo, s, c) for c in s.speeds]
    if kind == "unroll":
        return _exact_unroll(geo, s, case["iters"])
    if kind == "freq":
        return _exact_freq(geo, s, case["freqs"], case["df"])
    # dense: M's entries as the plan holds them (FP64, or rounded once to FP32)
    p = torch.zeros((geo.S, geo.K), dtype=torch.float64, device=s.v.device)
    g = torch.zeros(geo.N, dtype=torch.float64, device=s.v.device)
    v, r = s.v.double(), s.r.double().reshape(geo.S, geo.K)
    k = torch.arange(geo.K, device=s.v.device)
    for sl, w, k0, f in _blocks(geo, None, s.v.device):
        for i in range(sl.stop - sl.start):
            lo = (k[:, None] == k0[i][None, :]) * (w[i] * (1.0 - f[i]))[None, :]
            m = lo + (k[:, None] == k0[i][None, :] + 1) * (w[i] * f[i])[None, :]
            m = m.to(s.v.dtype).double()
            p[sl.start + i] = m @ v
            g += m.T @ r[sl.start + i]
    return {"p": p.reshape(-1), "g": g}
