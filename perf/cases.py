"""Timed workloads of the tracer through its public entry points.

Each case is one call pattern of a user's program: an image of a hole, the
mixed per-ray stream, the Sec. 3 grid projection, the Sec. 4 ring study, a
batched shadow sweep, the headless view of live photons, the initial
conditions with their conserved quantities, and a serving run.  Sizes, spins,
windows and options follow ``paper_1303_5057_gb300/inputs.py``, ``bench.py``
and the tests.

A ray's outcome does not depend on batching, queue order or launch shape, so
every output is reproducible bit for bit.

``exact`` integrates the same rays in plain torch in 64 bits where their end
points are determined by the inputs: under the Eq. 2 step rule without a floor
under the step, as the ring study runs it.  Under the benchmark step rule some
rays graze a pole and leave their geodesic (their angles grow to 1e3 - 1e6
rad, the digits set by rounding), so those images have no such value, and
neither have integer outputs.
"""
import math
import random

import numpy as np
import torch

from paper_1303_5057_gb300 import batch, gray, inputs, serve

# Photon RK4 steps per ray and flop per step of the method (FMA = 2): four
# right-hand sides, stage states, the RK4 sums, the Eq. 4 monitor, the step
# rule.  Means over images from r_obs = 1000 M.
FLOP_PER_STEP = 559
STEPS = {"bench": 385, "eq2": 515, "equator": 166, "ring": 620}


def listed():
    return [
        # one small render request by itself, unplanned: the latency of a single call
        {"name": "request_32", "kind": "image", "nx": 32, "ny": 32, "a": 0.7, "incl": 50.0,
         "precision": "fp32_kahan_sel64", "rule": "bench", "r_sw": 0.02, "plan": False, "out": "pixels32"},
        # the Schwarzschild check image, in double precision throughout
        {"name": "schwarzschild_64_fp64", "kind": "image", "nx": 64, "ny": 64, "a": 0.0, "incl": 60.0,
         "precision": "fp64", "rule": "bench", "r_sw": 0.0, "plan": False, "out": "pixels64"},
        # Sec. 3 grid projection: rays stopped on the equatorial plane
        {"name": "projection_128", "kind": "projection", "nx": 128, "ny": 128, "a": 0.95, "incl": 60.0,
         "precision": "fp32_kahan_sel64", "r_sw": 0.02},
        # a ragged image in double precision with full records, as an accuracy study takes it
        {"name": "kerr_300x211_fp64", "kind": "image", "nx": 300, "ny": 211, "a": 0.9, "incl": 75.0,
         "precision": "fp64", "rule": "bench", "r_sw": 0.0, "plan": True, "out": "record"},
        # the headline image: planned queue, single precision with the extended-precision zone
        {"name": "kerr_1024", "kind": "image", "nx": 1024, "ny": 1024, "a": 0.99, "incl": 90.0,
         "precision": "fp32_kahan_sel64", "rule": "bench", "r_sw": 0.02, "plan": True, "out": "pixels32"},
        # an odd-sized image under the paper's own Eq. 2 step rule (many steps near the horizon)
        {"name": "eq2_509", "kind": "image", "nx": 509, "ny": 509, "a": 0.94, "incl": 40.0,
         "precision": "fp32_kahan_sel64", "rule": "eq2", "r_sw": 0.02, "plan": True, "out": "pixels32"},
        # a list of single rays, half of them near their own critical curve (no image grid, no plan)
        {"name": "mixed_rays_524288", "kind": "rays", "n": 524288, "precision": "fp32_kahan_sel64", "r_sw": 0.02},
        # many images of uneven size in one launch, reduced to their shadows
        {"name": "sweep_24", "kind": "sweep", "n_images": 24, "side_lo": 64, "side_hi": 512},
        # Sec. 4 ring study: polar grids, Eq. 2 rule, compensated single precision
        {"name": "ring_3x1500x181", "kind": "ring", "n_images": 3, "n_r": 1500, "n_th": 181},
        # the interactive mode, headless: a few steps per frame, live photons drawn as sprites
        {"name": "view_512", "kind": "view", "side": 512, "frames": 48, "frame_steps": 8, "width": 1920,
         "height": 1080, "precision": "fp32_kahan_sel64"},
        # initial conditions of a large image with full records and conserved quantities (no trace)
        {"name": "initial_1000x777", "kind": "initial", "nx": 1000, "ny": 777, "a": 0.9, "incl": 65.0,
         "precision": "fp32_kahan_sel64"},
        # a burst of render requests of mixed size through the continuous-batching server
        {"name": "serve_16", "kind": "serve", "n_requests": 16, "side_max": 512, "capacity": 1 << 21},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["image", "image", "image", "image64", "projection", "rays", "sweep", "ring", "view",
                       "initial", "serve"])
    hole = {"a": round(rng.uniform(0.0, 0.999), 4), "incl": round(rng.uniform(1.0, 90.0), 3)}
    prec = rng.choice(["fp32", "fp32_kahan", "fp32_kahan_sel64", "fp32_kahan_sel64"])
    if kind == "image":
        n = _log_int(rng, 400, 900000)
        nx = max(8, int(math.sqrt(n) * rng.uniform(0.6, 1.6)))
        ny = max(8, n // nx)
        return {"kind": "image", "nx": nx, "ny": ny, **hole, "precision": prec,
                "rule": rng.choice(["bench", "bench", "eq2"]), "r_sw": rng.choice([0.02, 0.02, 0.25]),
                "plan": nx * ny >= 65536 or rng.random() < 0.3, "out": rng.choice(["pixels32", "pixels32", "record"])}
    if kind == "image64":
        nx, ny = _log_int(rng, 16, 250), _log_int(rng, 16, 250)
        return {"kind": "image", "nx": nx, "ny": ny, **hole, "precision": "fp64",
                "rule": rng.choice(["bench", "eq2"]), "r_sw": 0.0, "plan": nx * ny >= 16384,
                "out": rng.choice(["pixels64", "record"])}
    if kind == "projection":
        side = _log_int(rng, 8, 512)
        return {"kind": "projection", "nx": side, "ny": side, "a": hole["a"], "incl": round(rng.uniform(10.0, 80.0), 3),
                "precision": rng.choice(["fp32_kahan_sel64", "fp32_kahan_sel64", "fp32_kahan", "fp64"])
                if side <= 200 else "fp32_kahan_sel64", "r_sw": 0.02}
    if kind == "rays":
        return {"kind": "rays", "n": _log_int(rng, 3000, 520000), "precision": prec, "r_sw": 0.02}
    if kind == "sweep":
        lo = rng.randrange(16, 100)
        return {"kind": "sweep", "n_images": rng.randrange(2, 24), "side_lo": lo, "side_hi": lo + rng.randrange(1, 400)}
    if kind == "ring":
        return {"kind": "ring", "n_images": rng.randrange(1, 4), "n_r": _log_int(rng, 200, 1500),
                "n_th": rng.randrange(19, 182)}
    if kind == "view":
        return {"kind": "view", "side": _log_int(rng, 64, 512), "frames": rng.randrange(4, 48),
                "frame_steps": rng.choice([4, 8, 16]), "width": 1280, "height": rng.choice([720, 721]),
                "precision": prec}
    if kind == "initial":
        return {"kind": "initial", "nx": _log_int(rng, 30, 1000), "ny": _log_int(rng, 30, 777), **hole,
                "precision": rng.choice([prec, "fp64"])}
    return {"kind": "serve", "n_requests": rng.randrange(3, 16), "side_max": rng.choice([64, 128, 256, 512]),
            "capacity": rng.choice([1 << 19, 1 << 21])}


# ------------------------------------------------------------- preparation ---

def _jitter(case, seed):
    """Spin and inclination (radians) of a case's hole for one seed."""
    rng = random.Random(seed)
    a = case["a"] * (1.0 - 0.01 * rng.random())
    incl = case["incl"] + (0.5 if case["incl"] < 45.0 else -0.5) * rng.random()
    return a, math.radians(incl)


def _options(case):
    eq2 = case.get("rule") == "eq2"  # the paper's rule has no floor under the step
    return gray.Options(precision=gray.PRECISIONS[case["precision"]],
                        step_rule=gray.STEP_EQ2 if eq2 else gray.STEP_BENCH, h_min=1e-9 if eq2 else 1e-3,
                        max_steps=20000, r_sw=case.get("r_sw", 0.0),
                        stop_equator=1 if case["kind"] == "projection" else 0)


def _image(case, seed):
    a, incl = _jitter(case, seed)
    w = 15.0 if case["kind"] == "projection" else 10.0
    return inputs.Image(a=a, incl=incl, nx=case["nx"], ny=case["ny"], alpha0=-w, alpha1=w, beta0=-w, beta1=w)


def _ring_images(case, seed):
    rng = random.Random(seed)
    return [inputs.polar_image(rng.uniform(0.0, 0.98), rng.uniform(15.0, 90.0), case["n_r"], case["n_th"])
            for _ in range(case["n_images"])]


SIDES = (32, 64, 128, 256, 512)
OUT = {"pixels32": (gray.RENDER_PIXELS32, 16), "pixels64": (gray.RENDER_PIXELS64, 32),
       "record": (gray.RENDER_RECORD, 8 * gray.RECORD)}


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, kind = case, case["kind"]
    if kind in ("image", "projection"):
        s.image = _image(case, seed)
        s.tracer = gray.Tracer(_options(case), s.image.n)
        s.render, per = OUT[case.get("out", "pixels32")]
        s.out = torch.empty(per * s.image.n, dtype=torch.uint8, device="cuda")
        s.order = torch.empty(s.image.n, dtype=torch.int32, device="cuda") if case.get("plan") else None
    elif kind == "rays":
        n = case["n"]
        s.rays = torch.from_numpy(inputs.mixed_rays(n, offset=(seed % 4096) * n)).cuda()
        s.tracer = gray.Tracer(_options(case), n)
        s.render, per = OUT["pixels32"]
        s.out = torch.empty(per * n, dtype=torch.uint8, device="cuda")
    elif kind == "sweep":
        ims = inputs.shadow_sweep(case["n_images"], case["side_lo"], case["side_hi"], seed_index=3 + seed).images
        s.sweep = batch.ShadowSweep(ims, gray.Options(precision=gray.FP32_KAHAN_SEL64, max_steps=10000, r_sw=0.02))
    elif kind == "ring":
        s.images = _ring_images(case, seed)
        n = sum(im.n for im in s.images)
        s.tracer = gray.Tracer(gray.Options(precision=gray.FP32_KAHAN, step_rule=gray.STEP_EQ2, h_min=1e-9,
                                            max_steps=100000), n)
        s.order = torch.empty(n, dtype=torch.int32, device="cuda")
        s.info = torch.empty(gray.RING_DTYPE.itemsize * len(s.images), dtype=torch.uint8, device="cuda")
        s.boundary = torch.empty(sum(im.ny for im in s.images), dtype=torch.float64, device="cuda")
    elif kind == "view":
        rng = random.Random(seed)
        s.image = inputs.Image(a=rng.uniform(0.99, 0.999), incl=math.radians(rng.uniform(58.0, 62.0)),
                               nx=case["side"], ny=case["side"])
        s.tracer = gray.Tracer(gray.Options(precision=gray.PRECISIONS[case["precision"]], max_steps=10000, r_sw=0.02),
                               s.image.n)
        s.camera = gray.Camera(eye=(30.0, -22.0, 16.0), fov=math.radians(60.0), sprite=1.0, width=case["width"],
                               height=case["height"], status_mask=1 << gray.ACTIVE)
        s.count = torch.empty((case["height"], case["width"]), dtype=torch.int32, device="cuda")
        s.depth = torch.empty((case["height"], case["width"]), dtype=torch.float32, device="cuda")
    elif kind == "initial":
        s.image = _image(case, seed)
        s.tracer = gray.Tracer(gray.Options(precision=gray.PRECISIONS[case["precision"]]), s.image.n)
        s.record = torch.empty(8 * gray.RECORD * s.image.n, dtype=torch.uint8, device="cuda")
        s.invariants = torch.empty(32 * s.image.n, dtype=torch.uint8, device="cuda")
    else:
        sides = [x for x in SIDES if x <= case["side_max"]]
        s.requests = inputs.request_stream(1000.0, case["n_requests"], seed_index=4 + 16 * seed, sides=(32,))
        for k, q in enumerate(s.requests):  # the case's mix of sizes, spins and inclinations of the seed
            q.image.nx = q.image.ny = sides[(7 * k + case["n_requests"]) % len(sides)]
        s.server = serve.Server(gray.Options(precision=gray.FP32_KAHAN_SEL64, max_steps=10000, r_sw=0.02),
                                capacity=case["capacity"])
    return s


# -------------------------------------------------------------------- runs ---

def _pixels(out, kind):
    """The rendered buffer as (floating fields, integer fields), views of it."""
    if kind == gray.RENDER_PIXELS32:
        return {"point": out.view(torch.float32).view(-1, 4)[:, :3], "status": out.view(torch.int32).view(-1, 4)[:, 3]}
    if kind == gray.RENDER_PIXELS64:
        return {"point": out.view(torch.float64).view(-1, 4)[:, :3], "status": out.view(torch.int32).view(-1, 8)[:, 6:]}
    return {"record": out.view(torch.float64).view(-1, gray.RECORD)}


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind in ("image", "projection"):
        if s.order is not None:
            s.tracer.setup_plan([s.image], order=s.order)
        else:
            s.tracer.setup([s.image])
        s.tracer.trace(wait=False, order=s.order)
        return _pixels(s.tracer.render(s.render, out=s.out), s.render)
    if kind == "rays":
        s.tracer.setup_rays(s.rays)
        s.tracer.trace(wait=False)
        return _pixels(s.tracer.render(s.render, out=s.out), s.render)
    if kind == "sweep":
        sh, _ = s.sweep.run()
        return {"counts": np.stack([sh[k] for k in ("n_captured", "n_escaped", "n_other")]),
                "shadow": np.stack([sh[k] for k in ("area", "radius", "alpha_c", "beta_c")])}
    if kind == "ring":
        tr = s.tracer
        tr.setup_plan(s.images, order=s.order)
        tr.trace(wait=False, order=s.order)
        gray.gray_ring(tr.ctx, tr.state, tr.n, s.images, out=s.info, boundary=s.boundary)
        words = s.info.view(-1, gray.RING_DTYPE.itemsize)
        return {"metrics": words[:, :40].contiguous().view(torch.float64), "boundary": s.boundary,
                "counts": words[:, 40:].contiguous().view(torch.int32)}
    if kind == "view":
        tr = s.tracer
        tr.setup([s.image])
        live = []
        for _ in range(case["frames"]):
            _, n_active, _ = tr.trace(step_budget=case["frame_steps"])
            gray.gray_splat(tr.ctx, tr.state, tr.n, s.camera, count=s.count, depth=s.depth)
            live.append(n_active)
        return {"count": s.count, "depth": s.depth, "live": np.array(live)}
    if kind == "initial":
        s.tracer.setup([s.image])
        rec = s.tracer.render(gray.RENDER_RECORD, out=s.record)
        inv = s.tracer.render(gray.RENDER_INVARIANTS, out=s.invariants)
        return {"record": rec.view(torch.float64).view(-1, gray.RECORD), "invariants": inv.view(torch.float64).view(-1, 4)}
    stats = s.server.run(s.requests, realtime=False)
    out = []
    for r in sorted(stats.results, key=lambda r: r.rid):
        out.append({"point": r.pixels.view(np.float32).reshape(-1, 4)[:, :3],
                    "status": r.pixels.view(np.int32).reshape(-1, 4)[:, 3]})
    return out


def work(case):
    """Bytes of a pass: ray lists read and results written (images are a few
    numbers); flops: the method's steps in the case's arithmetic."""
    kind = case["kind"]
    if kind in ("image", "projection"):
        n = case["nx"] * case["ny"]
        steps = STEPS["equator"] if kind == "projection" else STEPS[case["rule"]]
        return {"bytes": n * OUT[case.get("out", "pixels32")][1], "flops": n * steps * FLOP_PER_STEP}
    if kind == "rays":
        return {"bytes": case["n"] * (40 + 16), "flops": case["n"] * STEPS["bench"] * FLOP_PER_STEP}
    if kind == "sweep":
        lo, hi = case["side_lo"], case["side_hi"]
        n = case["n_images"] * (lo * lo + lo * hi + hi * hi) / 3.0
        return {"bytes": 56 * case["n_images"], "flops": n * STEPS["bench"] * FLOP_PER_STEP}
    if kind == "ring":
        n = case["n_images"] * case["n_r"] * case["n_th"]
        return {"bytes": 8 * case["n_images"] * case["n_th"], "flops": n * STEPS["ring"] * FLOP_PER_STEP}
    if kind == "view":
        n = case["side"] ** 2
        steps = min(case["frames"] * case["frame_steps"], STEPS["bench"])
        return {"bytes": case["frames"] * 8 * case["width"] * case["height"], "flops": n * steps * FLOP_PER_STEP}
    if kind == "initial":
        n = case["nx"] * case["ny"]
        return {"bytes": n * (8 * gray.RECORD + 32), "flops": n * 300}
    sides = [x for x in SIDES if x <= case["side_max"]]
    n = case["n_requests"] * sum(x * x for x in sides) / len(sides)
    return {"bytes": 16 * n, "flops": n * STEPS["bench"] * FLOP_PER_STEP}


# ------------------------------------------- the same results in 64 bits ---

def _metric(a, r, th):
    """Kerr metric (M = 1) and its r and theta derivatives: three lists of
    (g_tt, g_tph, g_rr, g_thth, g_phph)."""
    s, c = torch.sin(th), torch.cos(th)
    a2, s2, sc = a * a, s * s, s * c
    S, D = r * r + a2 * c * c, r * r - 2.0 * r + a2
    u = 2.0 * r / S
    ur, uh = (2.0 - 2.0 * r * u) / S, 2.0 * a2 * sc * u / S
    P = r * r + a2 + a2 * s2 * u
    g = [u - 1.0, -a * s2 * u, S / D, S, s2 * P]
    gr = [ur, -a * s2 * ur, 2.0 * r / D - S * (2.0 * r - 2.0) / (D * D), 2.0 * r, s2 * (2.0 * r + a2 * s2 * ur)]
    gh = [uh, -a * (2.0 * sc * u + s2 * uh), -2.0 * a2 * sc / D, -2.0 * a2 * sc,
          2.0 * sc * P + s2 * a2 * (2.0 * sc * u + s2 * uh)]
    return g, gr, gh


def _start(a, incl, r_obs, alpha, beta):
    """(t, r, theta, phi, k) of image-plane positions, rows of 8, E = 1."""
    si, ci = math.sin(incl), math.cos(incl)
    x, z = r_obs * si - beta * ci, r_obs * ci + beta * si
    r, rho = torch.sqrt(r_obs ** 2 + alpha ** 2 + beta ** 2), torch.sqrt(x * x + alpha * alpha)
    th, ph = torch.atan2(rho, z), torch.atan2(alpha, x)
    kr = r_obs / r
    kh = (z * r_obs - r * r * ci) / (rho * r * r)
    kp = -alpha * si / (rho * rho)
    g, _, _ = _metric(a, r, th)
    B, C = 2.0 * g[1] * kp, g[2] * kr * kr + g[3] * kh * kh + g[4] * kp * kp
    kt = (-B - torch.sqrt(B * B - 4.0 * g[0] * C)) / (2.0 * g[0])
    E = -(g[0] * kt + g[1] * kp)
    return torch.stack([torch.zeros_like(r), r, th, ph, kt / E, kr / E, kh / E, kp / E])


def _rhs(a, y):
    """dy/dl of the second-order geodesic equation: k_t and k_phi conserved,
    the r and theta components from the metric's derivatives."""
    kt, kr, kh, kp = y[4], y[5], y[6], y[7]
    g, gr, gh = _metric(a, y[1], y[2])
    d = [p * kr + q * kh for p, q in zip(gr, gh)]
    bt, bp = d[0] * kt + d[1] * kp, d[1] * kt + d[4] * kp
    det = g[0] * g[4] - g[1] * g[1]

    def half(e):
        return 0.5 * (e[0] * kt * kt + 2.0 * e[1] * kt * kp + e[2] * kr * kr + e[3] * kh * kh + e[4] * kp * kp)

    return torch.stack([kt, kr, kh, kp, (g[1] * bp - g[4] * bt) / det, (half(gr) - d[2] * kr) / g[2],
                        (half(gh) - d[3] * kh) / g[3], (g[1] * bt - g[0] * bp) / det])


def _hermite(y0, y1, h, s):
    s2, s3 = s * s, s * s * s
    return ((2 * s3 - 3 * s2 + 1) * y0[:4] + (s3 - 2 * s2 + s) * h * y0[4:] + (3 * s2 - 2 * s3) * y1[:4]
            + (s3 - s2) * h * y1[4:])


def _trace(a, y, r_obs):
    """End points (t, r, theta, phi) and capture flags of rays traced under
    the Eq. 2 rule from the columns of y; a is a number or one value per ray."""
    n = y.shape[1]
    a = a if torch.is_tensor(a) else torch.full((n,), a, dtype=torch.float64, device=y.device)
    r_h = 1.0 + torch.sqrt(1.0 - a * a)
    ids = torch.arange(n, device=y.device)
    ends = []  # stopped rays: (ids, state before, state after, step, stop radius, captured)
    while ids.numel():
        r, kr = y[1], y[5].abs()
        h = (1.0 / 32.0) / (kr / r + y[6].abs() + y[7].abs())
        h = -torch.clamp(torch.minimum(h, (r - r_h) / (2.0 * kr)), min=1e-9)
        k1 = _rhs(a, y)
        k2 = _rhs(a, y + 0.5 * h * k1)
        k3 = _rhs(a, y + 0.5 * h * k2)
        y1 = y + h / 6.0 * (k1 + 2.0 * (k2 + k3) + _rhs(a, y + h * k3))
        g, _, _ = _metric(a, y1[1], y1[2])
        xi = (g[2] * y1[5] ** 2 + g[4] * y1[7] ** 2 + g[3] * y1[6] ** 2 + 2.0 * g[1] * y1[4] * y1[7]) / (
            g[0] * y1[4] ** 2)
        redo = ~((xi + 1.0).abs() <= 1e-3)
        h = torch.where(redo, h / 9.0, h)
        y1 = torch.where(redo, y + h * k1, y1)
        cap, esc = y1[1] <= 1.01 * r_h, (y1[1] >= r_obs) & (h * y1[5] > 0.0)
        stop = cap | esc
        if bool(stop.any()):
            target = torch.where(cap, 1.01 * r_h, r_obs)
            ends.append((ids[stop], y[:, stop], y1[:, stop], h[stop], target[stop], cap[stop]))
        over, under = y1[2] > math.pi, y1[2] < 0.0
        y1[3] = y1[3] + math.pi * over - math.pi * under
        y1[2] = torch.where(over, 2.0 * math.pi - y1[2], y1[2].abs())
        y1[6] = torch.where(over | under, -y1[6], y1[6])
        keep = ~stop
        y, a, r_h, ids = y1[:, keep], a[keep], r_h[keep], ids[keep]
    ids, y0, y1, h, target, cap = (torch.cat(x, dim=-1) for x in zip(*ends))
    lo, hi = torch.zeros_like(h), torch.ones_like(h)
    below = y0[1] < target
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        same = (_hermite(y0, y1, h, mid)[1] < target) == below
        lo, hi = torch.where(same, mid, lo), torch.where(same, hi, mid)
    p = _hermite(y0, y1, h, 0.5 * (lo + hi))
    over, under = p[2] > math.pi, p[2] < 0.0
    p[3] = p[3] + math.pi * over - math.pi * under
    p[2] = torch.where(over, 2.0 * math.pi - p[2], p[2].abs())
    back = torch.argsort(ids)
    return p[:, back], cap[back]


def _grid(im, device):
    i = torch.arange(im.n, device=device)
    row, col = (i // im.nx).double(), (i % im.nx).double()
    if im.grid:
        R = im.alpha0 + (col + 0.5) * (im.alpha1 - im.alpha0) / im.nx
        v = im.beta0 + row * (im.beta1 - im.beta0) / (im.ny - 1)
        return R * torch.cos(v), R * torch.sin(v)
    return (im.alpha0 + (col + 0.5) * (im.alpha1 - im.alpha0) / im.nx,
            im.beta0 + (row + 0.5) * (im.beta1 - im.beta0) / im.ny)


def _ring(im, captured):
    """Boundary radius per angle row and (D, <R>, A, alpha_min, alpha_max)."""
    C = torch.cumsum(captured.view(im.ny, im.nx).long(), dim=1)
    k = torch.arange(im.nx + 1, device=C.device)
    score = torch.cat([torch.zeros_like(C[:, :1]), 2 * C], dim=1) - k
    best = torch.argmax(score * (im.nx + 2) - k, dim=1)
    dR = (im.alpha1 - im.alpha0) / im.nx
    Rb = im.alpha0 + best.double() * dR
    v = im.beta0 + torch.arange(im.ny, device=C.device).double() * (im.beta1 - im.beta0) / (im.ny - 1)
    al, be = Rb * torch.cos(v), Rb * torch.sin(v)
    c = 0.5 * (al.min() + al.max())
    R = torch.sqrt((al - c) ** 2 + be ** 2)
    w = torch.ones_like(R)
    w[0] = w[-1] = 0.5
    mean = (w * R).sum() / w.sum()
    A = 2.0 * torch.sqrt((w * (R - mean) ** 2).sum() / w.sum())
    return Rb, torch.stack([c.abs(), mean, A, al.min(), al.max()])


def exact(case, seed):
    kind = case["kind"]
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "initial":
        im = _image(case, seed)
        y = _start(im.a, im.incl, im.r_obs, *_grid(im, device))
        g, _, _ = _metric(im.a, y[1], y[2])
        E, L = -(g[0] * y[4] + g[1] * y[7]), g[1] * y[4] + g[4] * y[7]
        s, c = torch.sin(y[2]), torch.cos(y[2])
        Q = (g[3] * y[6]) ** 2 + c * c * (L * L / (s * s) - im.a ** 2 * E * E)
        null = torch.zeros_like(E)
        zero = torch.zeros((im.n, 4), dtype=torch.float64, device=device)
        return {"record": torch.cat([zero, y[:4].t(), y.t(), zero[:, :1]], dim=1),
                "invariants": torch.stack([E, L, Q, null], dim=1)}
    if kind == "image" and case["rule"] == "eq2" and case["out"] != "record":
        im = _image(case, seed)
        p, _ = _trace(im.a, _start(im.a, im.incl, im.r_obs, *_grid(im, device)), im.r_obs)
        return {"point": p[1:].t().contiguous(), "status": None}
    if kind == "ring":
        y, a, ims = [], [], _ring_images(case, seed)
        for im in ims:
            y.append(_start(im.a, im.incl, im.r_obs, *_grid(im, device)))
            a.append(torch.full((im.n,), im.a, dtype=torch.float64, device=device))
        _, cap = _trace(torch.cat(a), torch.cat(y, dim=1), ims[0].r_obs)
        rings = [_ring(im, x) for im, x in zip(ims, torch.split(cap, [im.n for im in ims]))]
        return {"metrics": torch.stack([m for _, m in rings]), "boundary": torch.cat([b for b, _ in rings]),
                "counts": None}
    return None
