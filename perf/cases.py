"""The work that is timed: calls a program makes through this package's public entry points.

Rays traced one set at a time, single images, batched views in the three precisions, a panel of the paper's
figures, the ray equations themselves, and the surrogate network's two calls (inference and one gradient).
A surrogate render is the network's forward pass plus the integrator on the remaining rays; both are here.
"""
import math

import numpy as np
import torch

from paper_1209_6038_gb300 import cloak as ck
from paper_1209_6038_gb300 import inputs

INTEGRATORS = {"rk4": ck.RK4, "dp45": ck.DP45}
PRECISIONS = {"fp64": ck.FP64, "mixed": ck.MIXED, "mixed_ff": ck.MIXED_FF}
SCHEDULES = {"plain": ck.SCHED_PLAIN, "wavefront": ck.SCHED_WAVEFRONT}
DIMS = (7, 256, 256, 256, 256, 5)  # the surrogate network's layers
R1, R2, H = inputs.GEOMETRY["R1"], inputs.GEOMETRY["R2"], inputs.GEOMETRY["H"]
# (variant, polarization): radial / azimuthal cloak, ordinary / extraordinary light
MEDIA = ((0, 0), (0, 1), (1, 0), (1, 1))


def listed():
    return [
        # a handful of rays with the handle's defaults (fixed-step RK4): the smallest call, all latency
        dict(name="trace_few", kind="trace", rays=61, variant=0, pol=1, integ="rk4", h_or_tol=1e-3),
        # a ray set under error control, as in a convergence study: near-axis, grazing and cap rays among them
        dict(name="trace_set", kind="trace", rays=30011, variant=1, pol=0, integ="dp45", h_or_tol=1e-9),
        # the small workload: one preview image with the handle's defaults
        dict(name="image_preview", kind="image", variant=0, pol=1, width=128, height=96, spp=1, integ="rk4",
             h_or_tol=1e-3, schedule="plain", elevation=0.0),
        # one final image
        dict(name="image_1080p", kind="image", variant=0, pol=1, width=1920, height=1080, spp=4, integ="dp45",
             h_or_tol=1e-9, schedule="wavefront", elevation=20.0),
        # per-sample records (exit, time of flight, weight) of an odd-sized image, for analysis
        dict(name="records", kind="records", variant=1, pol=1, width=481, height=271, spp=3, integ="dp45",
             h_or_tol=1e-9, schedule="wavefront", elevation=20.0),
        # the full workload: twelve views in one batched FP64 render
        dict(name="batch_full", kind="batch", views=12, orbit=False, width=1920, height=1080, spp=4,
             precision="fp64"),
        # views of an orbit at mixed resolutions, mixed precision with the FP64 band
        dict(name="batch_orbit_mixed", kind="batch", views=12, orbit=True, width=1920, height=1080, spp=1,
             precision="mixed"),
        # the full workload in mixed precision with the double-float band, the fastest accurate render
        dict(name="batch_full_mixed_ff", kind="batch", views=12, orbit=False, width=1920, height=1080, spp=4,
             precision="mixed_ff"),
        # the paper's unpolarised panel with first-order reflections
        dict(name="panel_reflections", kind="panel", panel=ck.PANEL_UNPOLARIZED, variant=0, width=640, height=480,
             spp=2, reflections=True, elevation=20.0),
        # the ray equations on a large set of states
        dict(name="rhs", kind="rhs", states=1 << 20, variant=0, pol=1),
        # the network on a render's queue of rays, not a multiple of a tile
        dict(name="network_forward", kind="forward", rows=1_000_003, fp16=False),
        # one gradient of the training batch
        dict(name="network_gradient", kind="gradient", rows=19456, stage=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["trace", "trace", "image", "image", "records", "batch", "batch", "panel", "rhs", "forward",
                       "gradient"])
    variant, pol = rng.choice(MEDIA)
    if kind == "trace":
        integ = rng.choice(["rk4", "dp45"])
        return dict(kind=kind, rays=_log(rng, 1, 300_000), variant=variant, pol=pol, integ=integ,
                    h_or_tol=1e-3 if integ == "rk4" else rng.choice([1e-7, 1e-9, 1e-11]))
    if kind in ("image", "records"):
        width = _log(rng, 64, 1920)
        height = max(1, int(width * rng.uniform(0.5, 1.0)))
        integ = rng.choice(["rk4", "dp45", "dp45"])
        return dict(kind=kind, variant=variant, pol=pol, width=width, height=height, spp=rng.choice([1, 1, 2, 4]),
                    integ=integ, h_or_tol=2e-3 if integ == "rk4" else rng.choice([1e-7, 1e-9]),
                    schedule="wavefront" if width > 256 else rng.choice(["plain", "wavefront"]),
                    elevation=rng.uniform(0.0, 60.0))
    if kind == "batch":
        width = _log(rng, 96, 1920)
        return dict(kind=kind, views=rng.choice([1, 2, 4, 7, 12]), orbit=rng.random() < 0.5, width=width,
                    height=max(1, int(width * rng.uniform(0.5, 0.6))), spp=rng.choice([1, 2, 4]),
                    precision=rng.choice(["fp64", "fp64", "mixed", "mixed_ff"]))
    if kind == "panel":
        width = _log(rng, 96, 1280)
        return dict(kind=kind, panel=rng.choice([ck.PANEL_UNPOLARIZED, ck.PANEL_POLARIZER_RIGHT, ck.PANEL_TOF]),
                    variant=variant, width=width, height=max(1, int(width * rng.uniform(0.5, 1.0))),
                    spp=rng.choice([1, 2, 4]), reflections=rng.random() < 0.5, elevation=rng.uniform(0.0, 60.0))
    if kind == "rhs":
        return dict(kind=kind, states=_log(rng, 100, 4_000_000), variant=variant, pol=pol)
    if kind == "forward":
        return dict(kind=kind, rows=_log(rng, 100, 4_000_000), fp16=rng.random() < 0.5)
    return dict(kind=kind, rows=128 * _log(rng, 2, 304), stage=rng.choice([1, 1, 2]))


# ------------------------------------------------------------------ inputs
def _params(seed):
    """Network parameters at unit gain: per layer W (out x in) then b."""
    rng = np.random.default_rng(seed)
    ps = []
    for a, b in zip(DIMS[:-1], DIMS[1:]):
        ps.append(rng.normal(0, 1.0 / math.sqrt(a), (b, a)).ravel())
        ps.append(rng.normal(0, 0.05, b))
    return np.concatenate(ps).astype(np.float32)


def _rows(case, seed):
    """Network inputs and training targets (t0..t3, confidence target, mask, two spare) of a batch."""
    rng = np.random.default_rng([seed, 1])
    n = case["rows"]
    x = rng.uniform(-1, 1, (n, 7)).astype(np.float32)
    t = np.zeros((n, 8), np.float32)
    if case["kind"] == "gradient":
        t[:, :5] = rng.normal(0, 1, (n, 5))
        t[:, 5] = rng.uniform(0, 1, n) < 0.8
    return x, t


def _states(case, seed):
    """States inside the shell: radius in (R1, R2), velocities of order one."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = case["states"]
    u = torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64)
    v = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    r = R1 + (R2 - R1) * (1e-3 + 0.999 * u[:, 0])
    a = 2 * math.pi * u[:, 1]
    pos = torch.stack([r * torch.cos(a), r * torch.sin(a), H * (u[:, 2] - 0.5)], 1)
    return torch.cat([pos, v], 1).contiguous()


def _camera(case, seed):
    azimuth = np.random.default_rng([seed, 2]).uniform(0.0, 360.0)
    return inputs.camera_pose(case["elevation"], azimuth)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind in ("trace", "rhs"):
        c = ck.Cloak(case["variant"], R1, R2, H)
        st["c"] = c
        if kind == "trace":
            c.integrator(INTEGRATORS[case["integ"]], case["h_or_tol"])
            st["rays"] = torch.from_numpy(inputs.ray_set(case["rays"], seed, "mixed", R2, H)).cuda()
        else:
            st["y"] = _states(case, seed)
    elif kind in ("image", "records", "panel"):
        eye, target, up = _camera(case, seed)
        c = ck.Cloak(case["variant"], R1, R2, H)
        c.camera(eye, target, up, 60.0, case["width"], case["height"])
        if kind == "panel":
            c.integrator(ck.DP45, 1e-9).reflections(case["reflections"])
        else:
            c.integrator(INTEGRATORS[case["integ"]], case["h_or_tol"]).schedule(SCHEDULES[case["schedule"]])
        st["c"] = c
    elif kind == "batch":
        c = ck.Cloak(ck.RADIAL, R1, R2, H)
        c.integrator(ck.DP45, 1e-9, PRECISIONS[case["precision"]]).schedule(ck.SCHED_WAVEFRONT)
        rng = np.random.default_rng([seed, 3])
        azimuth = rng.uniform(0.0, 360.0)
        W, Hp = case["width"], case["height"]
        sizes = ((W, Hp), (Hp, Hp), (max(1, W // 2), max(1, Hp // 2)), (max(1, W // 4 + 1), max(1, Hp // 3)))
        views = []
        for i in range(case["views"]):
            v, p = MEDIA[i % 4]
            if case["orbit"]:  # seeded poses, each at its own resolution, rendered for every medium
                if i % 4 == 0:
                    pose = inputs.camera_pose(rng.uniform(0.0, 60.0), rng.uniform(0.0, 360.0))
                    w, h = sizes[(i // 4) % 4]
            else:
                pose = inputs.camera_pose((0.0, 20.0, 45.0)[(i // 4) % 3], azimuth)
                w, h = W, Hp
            out = torch.empty((h, w, 4), dtype=torch.float32, device="cuda")
            views.append((v, p, *pose, 60.0, out))
        st["c"], st["views"] = c, views
    else:
        c = ck.Cloak(ck.RADIAL, R1, R2, H)
        ck.cloak_surrogate_params(c.h, _params(seed))
        x, t = _rows(case, seed)
        st["c"], st["x"] = c, torch.from_numpy(x).cuda()
        if kind == "forward":
            ck.cloak_surrogate_set_precision(c.h, case["fp16"])
            st["y"] = torch.empty((case["rows"], 5), dtype=torch.float32, device="cuda")
        else:
            st["t"] = torch.from_numpy(t).cuda()
    return st


def _fields(recs):
    """A record buffer's floating-point fields (exit point and direction, time of flight, weight) and its
    integers (tile, status, steps, mode), as views."""
    rows = recs.view(-1, ck.RECORD_BYTES)
    return rows.view(torch.float64)[:, :8], rows.view(torch.int32)[:, 16:]


def run(st):
    case, c, seed = st["case"], st["c"], st["seed"]
    kind = case["kind"]
    if kind == "trace":
        return _fields(c.trace_rays(case["pol"], st["rays"]))
    if kind == "image":
        return c.render(case["pol"], case["spp"], seed)
    if kind == "records":
        return _fields(c.render_records(case["pol"], case["spp"], seed))
    if kind == "panel":
        return c.panel(case["panel"], case["spp"], seed)
    if kind == "batch":
        ck.cloak_render_batch(c.h, st["views"], case["spp"], seed)
        return [v[-1] for v in st["views"]]
    if kind == "rhs":
        return c.eval_rhs(case["pol"], st["y"])
    if kind == "forward":
        ck.cloak_surrogate_forward(c.h, st["x"], st["y"])
        return st["y"]
    return ck.cloak_surrogate_step(c.h, st["x"], st["t"], stage=case["stage"], lr=0.0)


# ------------------------------------------------------------------ the work of one pass
# Operations per step attempt from the equations (an FMA counts two): right-hand side 36 (radial e),
# 30 (azimuthal e), 34 (azimuthal o), 0 (radial o); six of them and 362 for the stages, the end point and
# the error estimate of DP5(4), four and 102 for RK4.  Mean step attempts per entering ray and the share of
# camera rays that enter, at distance 5 and 60 degrees: 1.19e9 attempts on 99.5e6 camera rays at tolerance
# 1e-9 (about 12 per camera ray); RK4 covers a mean path of about 1.6 at its fixed step.
_RHS_FLOPS = {(0, 0): 0, (0, 1): 36, (1, 0): 34, (1, 1): 30}


def _ray_flops(integ, h_or_tol, variant, pol, camera):
    rhs = _RHS_FLOPS[(variant, pol)]
    if integ == "rk4":
        return 1.6 / h_or_tol * (4 * rhs + 102) * (0.15 if camera else 0.8)
    return 12.0 * (1e-9 / h_or_tol) ** 0.2 * (6 * rhs + 362) * (1.0 if camera else 5.0)


def work(case):
    kind = case["kind"]
    if kind == "trace":
        n = case["rays"]
        return dict(bytes=n * (48 + 80), flops=n * _ray_flops(case["integ"], case["h_or_tol"], case["variant"],
                                                              case["pol"], False))
    if kind in ("image", "records"):
        px = case["width"] * case["height"]
        n = px * case["spp"]
        return dict(bytes=n * 80 if kind == "records" else px * 16,
                    flops=n * _ray_flops(case["integ"], case["h_or_tol"], case["variant"], case["pol"], True))
    if kind == "panel":
        px = case["width"] * case["height"]
        return dict(bytes=px * 16, flops=sum(px * case["spp"] * _ray_flops("dp45", 1e-9, case["variant"], p, True)
                                             for p in (0, 1)) * (3 if case["reflections"] else 1))
    if kind == "batch":
        W, Hp = case["width"], case["height"]
        sizes = ((W, Hp), (Hp, Hp), (max(1, W // 2), max(1, Hp // 2)), (max(1, W // 4 + 1), max(1, Hp // 3)))
        b = f = 0.0
        for i in range(case["views"]):
            w, h = sizes[(i // 4) % 4] if case["orbit"] else (W, Hp)
            b += w * h * 16
            f += w * h * case["spp"] * _ray_flops("dp45", 1e-9, *MEDIA[i % 4], True)
        return dict(bytes=b, flops=f)
    if kind == "rhs":
        n = case["states"]
        return dict(bytes=n * 96, flops=n * _RHS_FLOPS[(case["variant"], case["pol"])])
    n = case["rows"]
    weights = sum(a * b for a, b in zip(DIMS[:-1], DIMS[1:]))
    if kind == "forward":
        return dict(bytes=n * 48 + 4 * weights, flops=2.0 * n * weights)
    # forward, weight gradients, and the gradients handed back through every layer but the first
    layers = 3 * weights - DIMS[0] * DIMS[1]
    return dict(bytes=n * 60 + 8 * weights, flops=2.0 * n * layers)


# ------------------------------------------------------------------ the same in 64 bits
def _layers(params):
    out, o = [], 0
    p = torch.from_numpy(params).cuda().double()
    for a, b in zip(DIMS[:-1], DIMS[1:]):
        out.append((p[o:o + a * b].view(b, a), p[o + a * b:o + a * b + b]))
        o += a * b + b
    return out


def _network(layers, x):
    for i, (w, b) in enumerate(layers):
        x = x @ w.t() + b
        if i < len(layers) - 1:
            x = torch.nn.functional.gelu(x, approximate="tanh")
    return x


def exact(case, seed):
    """The ray equations and the network in plain torch at 64 bits.  None for traced rays: a ray near the inner
    radius takes tens of thousands of dependent steps, each some hundreds of small tensor operations."""
    kind = case["kind"]
    if kind == "rhs":
        y = _states(case, seed)
        x, v = y[:, :3], y[:, 3:]
        r = torch.hypot(x[:, 0], x[:, 1])
        rh = torch.stack([x[:, 0] / r, x[:, 1] / r], 1)
        vr = v[:, 0] * rh[:, 0] + v[:, 1] * rh[:, 1]
        vt = v[:, 1] * rh[:, 0] - v[:, 0] * rh[:, 1]
        vz = v[:, 2]
        u = r - R1
        g = 2.0 * R1 / (r * u)  # f' / f
        zero = torch.zeros_like(r)
        if (case["variant"], case["pol"]) == (0, 0):
            ar = at = az = zero
        elif case["pol"] == 0:
            ar, at, az = 0.5 * g * (vt * vt + vz * vz - vr * vr), -g * vr * vt, -g * vr * vz
        elif case["variant"] == 0:
            ar, at, az = R1 * (u * vz * vz - r * vt * vt) / r ** 3, -g * vr * vt, -g * vr * vz
        else:
            ar, at, az = -R1 * vt * vt / (r * r), -g * vr * vt, zero
        ax = ar * rh[:, 0] - at * rh[:, 1]
        ay = ar * rh[:, 1] + at * rh[:, 0]
        return torch.cat([v, torch.stack([ax, ay, az], 1)], 1)
    if kind == "forward":
        x, _ = _rows(case, seed)
        layers = _layers(_params(seed))
        return torch.cat([_network(layers, part.cuda().double()) for part in torch.from_numpy(x).split(1 << 18)])
    if kind == "gradient":
        xs, ts = _rows(case, seed)
        layers = [(w.clone().requires_grad_(), b.clone().requires_grad_()) for w, b in _layers(_params(seed))]
        y, t = _network(layers, torch.from_numpy(xs).cuda().double()), torch.from_numpy(ts).cuda().double()
        if case["stage"] == 1:  # masked squared error of the regression outputs, the time of flight at a tenth
            scale = torch.tensor([1.0, 1.0, 1.0, 0.1], dtype=torch.float64, device="cuda")
            loss = (t[:, 5:6] * scale * (y[:, :4] - t[:, :4]) ** 2).sum() / case["rows"]
        else:  # absolute error of the confidence output
            loss = (y[:, 4] - t[:, 4]).abs().sum() / case["rows"]
        loss.backward()
        return torch.cat([p.grad.reshape(-1) for layer in layers for p in layer]).cpu().numpy()
    return None
