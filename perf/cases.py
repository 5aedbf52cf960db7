"""The work a user has the solver do, as cases to be timed and compared.

A case is a plain dict; `prepare` builds what a user's program holds before the call (the image on
the device or in page-locked host memory, the markers, the solver handle), `run` makes one pass
through the public entry points and returns its outputs, `work` counts what such a pass cannot do
without, and `exact` gives the level set of one pseudo-time step in 64 bits from a plain torch
restatement of the equation (no multigrid, none of the package's solver code).

One pass of a handle is what a segmentation service does per image: `reset` on the next image and
its markers, one pseudo-time step to ||L(phi)|| / ||L(phi^n)|| <= tol, the level set and the mask.
Images are the seeded synthetic ones of the package (ellipses with ramps and noise; the disc and
square), scaled with the image size as its named workloads are.
"""
from __future__ import annotations

import math

import torch

from paper_1807_02137_gb300 import segmg, synth

# option texts of a case
PRECISION = {"f32": segmg.MG_F32, "f64": segmg.MG_F64, "mixed": segmg.MG_MIXED}
MODEL = {"sc": segmg.MG_MODEL_SC, "rc": segmg.MG_MODEL_RC}
SMOOTHER = {"hs2": segmg.MG_SMOOTH_FUSED, "gsline": segmg.MG_SMOOTH_GSLINE}
MAX_CYCLES = 60


def listed():
    return [
        # the smallest: the FP64 disc-and-square image of the accuracy checks, to 1e-8; every
        # grid is latency-bound
        {"name": "step_128_f64", "kind": "step", "n": 128, "m": 128, "precision": "f64", "model": "sc",
         "smoother": "hs2", "image": "disc", "tol": 1e-8},
        # a thumbnail or a region of interest, one image at a time: launches and chains count
        {"name": "step_256_f32", "kind": "step", "n": 256, "m": 256, "precision": "f32", "model": "sc",
         "smoother": "hs2", "image": "ellipses", "tol": 1e-6},
        # the headline workload's size: one ordinary image on a kept handle
        {"name": "step_1024_f32", "kind": "step", "n": 1024, "m": 1024, "precision": "f32", "model": "sc",
         "smoother": "hs2", "image": "ellipses", "tol": 1e-6},
        # the same image end to end: host image in, host mask out
        {"name": "host_1024_f32", "kind": "host", "n": 1024, "m": 1024, "precision": "f32", "model": "sc",
         "smoother": "hs2", "image": "ellipses", "tol": 1e-6},
        # the second model (area constraint) on a ragged size
        {"name": "step_rc_517x700_f32", "kind": "step", "n": 517, "m": 700, "precision": "f32", "model": "rc",
         "smoother": "hs2", "image": "ellipses", "tol": 1e-6},
        # a segmentation run on: several pseudo-time steps, the step control halving tau on the way
        {"name": "solve_512_f32", "kind": "solve", "n": 512, "m": 512, "precision": "f32", "model": "sc",
         "smoother": "hs2", "image": "ellipses", "tol": 1e-6, "steps": 4},
        # a large photograph or a tile of a scan: beyond L2
        {"name": "step_4096_f32", "kind": "step", "n": 4096, "m": 4096, "precision": "f32", "model": "sc",
         "smoother": "hs2", "image": "ellipses", "tol": 1e-6},
        # a whole-slide scan: the largest image, coefficients in BF16, non-power-of-two coarsening
        {"name": "step_25000_mixed", "kind": "step", "n": 25000, "m": 25000, "precision": "mixed", "model": "sc",
         "smoother": "hs2", "image": "ellipses", "tol": 1e-6},
        # many images of uneven sizes in one go
        {"name": "batch_16_f32", "kind": "batch", "precision": "f32", "model": "sc", "smoother": "hs2",
         "sizes": "256,256,256,256,512,512,512,512,768,768,768,1024,1024,1024,2048,2048", "tol": 1e-6},
        # the relaxation weights predicted by the conv net, accepted V-cycle by V-cycle
        {"name": "learned_2048_f32", "kind": "learned", "n": 2048, "m": 2048, "precision": "f32", "model": "sc",
         "smoother": "hs2", "image": "ellipses", "tol": 1e-6},
        # the paper's Algorithm 1 (line smoother), which comparisons of the algorithms run
        {"name": "step_gsline_1024_f32", "kind": "step", "n": 1024, "m": 1024, "precision": "f32", "model": "sc",
         "smoother": "gsline", "image": "ellipses", "tol": 1e-6},
    ]


# kind, precision, model, smoother, smallest and largest side (geometric mean of the two sides)
RANGES = [
    ("step", "f32", "sc", "hs2", 96, 6000),
    ("step", "f32", "sc", "hs2", 96, 6000),
    ("step", "f64", "sc", "hs2", 64, 400),
    ("step", "mixed", "sc", "hs2", 512, 9000),
    ("step", "f32", "rc", "hs2", 100, 1500),
    ("step", "f32", "sc", "gsline", 100, 1200),
    ("host", "f32", "sc", "hs2", 128, 3000),
    ("solve", "f32", "sc", "hs2", 128, 1000),
    ("learned", "f32", "sc", "hs2", 256, 3000),
    ("batch", "f32", "sc", "hs2", 200, 1500),
]


def draw(rng):
    kind, precision, model, smoother, lo, hi = rng.choice(RANGES)

    def side():
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    c = {"kind": kind, "precision": precision, "model": model, "smoother": smoother, "tol": 1e-6}
    if precision == "f64":
        c["tol"] = 1e-8
    if kind == "batch":
        c["sizes"] = ",".join(str(side()) for _ in range(rng.randint(4, 12)))
        return c
    s, aspect = side(), math.exp(rng.uniform(-0.4, 0.4))
    c.update(n=max(48, int(s * aspect)), m=max(48, int(s / aspect)), image="ellipses")
    if kind == "solve":
        c["steps"] = rng.randint(2, 4)
    return c


def image_of(image, n, m, precision, seed):
    """One image on the device and its markers (host), from the seed."""
    dt = torch.float64 if precision == "f64" else torch.float32
    if image == "disc":
        img, mk, _ = synth.disc_square(n, 0.05, seed)
        return torch.as_tensor(img, dtype=dt, device="cuda"), mk
    s = max(n, m) / 1024.0
    count = min(200, max(12, int(12 * s)))
    img, mk = synth.ellipses_device(n, m, count, (20.0 * s, 200.0 * s), 8, 0.05, seed, "cuda")
    return img.to(dt), mk


def params_of(case, n, m):
    return segmg.default_params(n, m, precision=PRECISION[case["precision"]], model=MODEL[case["model"]],
                                smoother=SMOOTHER[case["smoother"]])


def batch_images(case, seed):
    sizes = [int(s) for s in case["sizes"].split(",")]
    return [image_of("ellipses", s, s, case["precision"], seed * 64 + k) for k, s in enumerate(sizes)]


def net_weights(seed):
    """Parameters of the relaxation-weight net (5 -> 16 -> 16 -> 1 channels, 3x3): He-scaled, a
    small last layer, so that the predicted weights lie about 1 as trained ones do."""
    g = torch.Generator().manual_seed(seed)
    parts = []
    for cout, cin, scale in ((16, 5, 1.0), (16, 16, 1.0), (1, 16, 0.1)):
        parts.append(torch.randn(cout * cin * 9, generator=g) * (scale * math.sqrt(2.0 / (9 * cin))))
        parts.append(torch.zeros(cout))
    return torch.cat(parts).numpy()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        pairs = batch_images(case, seed)
        images, markers = [p[0] for p in pairs], [p[1] for p in pairs]
        params = [params_of(case, *im.shape) for im in images]
        return {"case": case, "images": images, "markers": markers,
                "batch": segmg.Batch(images, markers, params)}
    n, m = case["n"], case["m"]
    img, mk = image_of(case["image"], n, m, case["precision"], seed)
    p = params_of(case, n, m)
    if kind == "host":
        host = img.cpu().pin_memory().numpy()
        mask = torch.empty((n, m), dtype=torch.uint8).pin_memory().numpy()
        return {"case": case, "image": host, "markers": mk, "params": p, "mask": mask}
    s = segmg.Solver(img, mk, p)
    if kind == "learned":
        s.set_learned(net_weights(seed), mode=1, refresh=4)
    return {"case": case, "image": img, "markers": mk, "solver": s}


def run(state):
    case = state["case"]
    kind, tol = case["kind"], case["tol"]
    if kind == "host":
        mask, _, _ = segmg.segment_host(state["image"], state["markers"], state["params"], tol, MAX_CYCLES,
                                        mask_out=state["mask"])
        return {"mask": mask}
    if kind == "batch":
        b = state["batch"]
        b.reset(state["images"], state["markers"])
        b.solve_step(tol, MAX_CYCLES)
        solvers = [b.solver(i) for i in range(b.count)]
        return {"phi": [s.phi() for s in solvers], "mask": [s.mask() for s in solvers]}
    s = state["solver"]
    s.reset(state["image"], state["markers"])
    if kind == "solve":
        s.solve(tol, MAX_CYCLES, 0.0, case["steps"])
    else:
        s.solve_step(tol, MAX_CYCLES)
    return {"phi": s.phi(), "mask": s.mask()}


# Floating-point operations per cell of one V(2,2) cycle on one grid: four smoothing iterations of
# a snapshot (about 60) and four sweeps (about 18 each), a residual and the transfers (about 60);
# 4/3 of it over all grids.  A step takes about a dozen V-cycles.
CYCLE_FLOPS = 4.0 / 3.0 * (4 * (60 + 4 * 18) + 60)
CYCLES = 12


def work(case):
    """Bytes: the image in, the level set and the mask out, once each.  Operations: those of a
    dozen V-cycles per step."""
    item = 8 if case["precision"] == "f64" else 4
    if case["kind"] == "batch":
        cells = sum(int(s) ** 2 for s in case["sizes"].split(","))
    else:
        cells = case["n"] * case["m"]
    out = 1 if case["kind"] == "host" else item + 1
    steps = case.get("steps", 1)
    return {"bytes": float(cells * (item + out)), "flops": float(cells * CYCLE_FLOPS * CYCLES * steps)}


# ---- the 64-bit value of one step -------------------------------------------------------------

EXACT_CELLS = 1 << 21      # larger images would take too long
EPS, BETA, BETA_EDGE, SIGMA_BLUR, MU, LAM, THETA, NU, TAU = 1.0, 1e-6, 1.0, 1.0, 1.0, 10.0, 1.0, 1.0, 1.0


def _shift(a, di, dj):
    """a at (i + di, j + dj), indices clamped into the grid."""
    n, m = a.shape
    i = torch.arange(n, device=a.device).add(di).clamp(0, n - 1)
    j = torch.arange(m, device=a.device).add(dj).clamp(0, m - 1)
    return a[i][:, j] if di and dj else (a[i] if di else a[:, j])


def _blur(z, dim):
    """Gaussian taps of radius 3 sigma, half-sample mirror boundary."""
    r = int(math.ceil(3 * SIGMA_BLUR))
    taps = [math.exp(-t * t / (2 * SIGMA_BLUR ** 2)) for t in range(-r, r + 1)]
    n = z.shape[dim]
    out = torch.zeros_like(z)
    for t, w in zip(range(-r, r + 1), taps):
        i = torch.arange(n, device=z.device) + t
        i = torch.where(i < 0, -i - 1, i)
        i = torch.where(i >= n, 2 * n - i - 1, i)
        out += w / sum(taps) * z.index_select(dim, i)
    return out


def _hull(points):
    pts = sorted(set(map(tuple, points.tolist())))

    def half(seq):
        h = []
        for p in seq:
            while len(h) > 1 and ((h[-1][0] - h[-2][0]) * (p[1] - h[-2][1])
                                  - (h[-1][1] - h[-2][1]) * (p[0] - h[-2][0])) <= 0:
                h.pop()
            h.append(p)
        return h[:-1]

    return half(pts) + half(pts[::-1]) if len(pts) > 2 else []


def _initial(mk, n, m, dev):
    """Signed distance to the markers' convex hull (a disc when it has no area), and its area."""
    y = torch.arange(n, device=dev, dtype=torch.float64)[:, None]
    x = torch.arange(m, device=dev, dtype=torch.float64)[None, :]
    h = _hull(mk)
    area = 0.5 * sum(h[q][0] * h[(q + 1) % len(h)][1] - h[(q + 1) % len(h)][0] * h[q][1] for q in range(len(h)))
    if len(h) < 3 or area <= 0:
        r0 = 0.05 * max(n, m)
        return r0 - torch.sqrt((x - mk[:, 0].mean()) ** 2 + (y - mk[:, 1].mean()) ** 2), math.pi * r0 * r0
    dist = torch.full((n, m), 1e30, dtype=torch.float64, device=dev)
    inside = torch.ones((n, m), dtype=torch.bool, device=dev)
    for q in range(len(h)):
        (ax, ay), (bx, by) = h[q], h[(q + 1) % len(h)]
        ex, ey = bx - ax, by - ay
        inside &= ex * (y - ay) - ey * (x - ax) >= 0
        t = (((x - ax) * ex + (y - ay) * ey) / (ex * ex + ey * ey)).clamp(0, 1)
        dist = torch.minimum(dist, torch.sqrt((x - ax - t * ex) ** 2 + (y - ay - t * ey) ** 2))
    return torch.where(inside, dist, -dist), area


def _step_solution(z, mk, rc):
    """phi of one pseudo-time step: lagged diffusivity with a conjugate-gradient inner solve, to
    about 1e-9 of the change.  None when that is not reached."""
    n, m = z.shape
    dev = z.device
    zb = _blur(_blur(z, 1), 0)
    g = 1.0 / (1.0 + BETA_EDGE * 0.25 * ((_shift(zb, 0, 1) - _shift(zb, 0, -1)) ** 2
                                         + (_shift(zb, 1, 0) - _shift(zb, -1, 0)) ** 2))
    s2 = 1.0 / (2.0 * (0.05 * max(n, m)) ** 2)
    d = torch.ones_like(z)
    for px, py in mk.tolist():
        ex = torch.exp(-(torch.arange(m, device=dev, dtype=torch.float64) - px) ** 2 * s2)
        ey = torch.exp(-(torch.arange(n, device=dev, dtype=torch.float64) - py) ** 2 * s2)
        d *= 1.0 - ey[:, None] * ex[None, :]
    w = d * g if rc else g
    pn, area0 = _initial(mk, n, m, dev)

    def heaviside(p):
        return 0.5 + torch.atan(p / EPS) / math.pi

    H = heaviside(pn)
    c1, c2 = (H * z).sum() / H.sum(), ((1 - H) * z).sum() / (1 - H).sum()
    F = LAM * (z - c1) ** 2 - LAM * (z - c2) ** 2 + (0.0 if rc else THETA * d)

    def div(ax, ay, v):
        """sum over the existing faces of (face value) (v_X - v)"""
        out = torch.zeros_like(v)
        fy = ay * (v[1:] - v[:-1])
        fx = ax * (v[:, 1:] - v[:, :-1])
        out[:-1] += fy
        out[1:] -= fy
        out[:, :-1] += fx
        out[:, 1:] -= fx
        return out

    u = torch.zeros_like(z)
    last = None
    for outer in range(400):
        p = pn + u
        G = w / torch.sqrt(0.25 * ((_shift(p, 0, 1) - _shift(p, 0, -1)) ** 2
                                   + (_shift(p, 1, 0) - _shift(p, -1, 0)) ** 2) + BETA)
        ax, ay = MU * 0.5 * (G[:, 1:] + G[:, :-1]), MU * 0.5 * (G[1:] + G[:-1])
        b = div(ax, ay, pn) - F
        if rc:
            b = b - 2.0 * NU * (heaviside(p).sum() - area0) / (n * m)
        diag = torch.full_like(z, 1.0 / TAU)
        diag[:-1] += ay
        diag[1:] += ay
        diag[:, :-1] += ax
        diag[:, 1:] += ax
        r = b - (u / TAU - div(ax, ay, u))
        rn = float(r.norm())
        if last is None:
            last = rn
        if rn <= 1e-10 * last:
            return p
        # the inner system to a hundredth of this iterate's residual
        y = r / diag
        q, rz = y.clone(), (r * y).sum()
        for inner in range(1000):
            Aq = q / TAU - div(ax, ay, q)
            alpha = rz / (q * Aq).sum()
            u = u + alpha * q
            r = r - alpha * Aq
            if inner % 10 == 9 and float(r.norm()) <= 1e-2 * rn:
                break
            y = r / diag
            rz, old = (r * y).sum(), rz
            q = y + (rz / old) * q
    return None


def exact(case, seed):
    """The level set of one step from the method's equation in 64 bits; the mask has no such
    value.  None for images that would take too long, where the outputs come after several steps
    (each of whose step sizes the solver chooses), for several images and for a mask alone."""
    kind = case["kind"]
    if kind in ("batch", "solve", "host") or case["n"] * case["m"] > EXACT_CELLS:
        return None
    img, mk = image_of(case["image"], case["n"], case["m"], case["precision"], seed)
    phi = _step_solution(img.to(torch.float64), mk, case["model"] == "rc")
    return None if phi is None else {"phi": phi, "mask": None}
