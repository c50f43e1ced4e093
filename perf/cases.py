"""The work that this library is measured on: the calls of its users, over the
range of sizes, directions, precisions and pixel kinds they come in.

A program that images a radio observation sets the visibilities and the pixels
once and then, for as long as the problem lives, applies the operator and its
adjoint or solves for the image.  So ``prepare`` sets a problem up and ``run``
is one call.  Geometry, pixel layouts and gains come from the repository's own
generators (``synth``) at the sizes of its configurations, tests and benchmark;
every random choice (antenna positions, sources, noise, gains) follows the
seed.

Results.  FP64 results stay FP64.  A mixed-precision result holds an FP32
computation in an FP64 array; the program keeps it in single precision, as
images (FITS) and visibilities (complex64 measurement sets) are stored.
"""
import math

import numpy as np
import torch

from paper_1310_2078_gb300 import sl1m, synth

MIXED, FP64 = "mixed", "fp64"
PREC = {MIXED: sl1m.MIXED, FP64: sl1m.FP64}

# Power-iteration steps of a solve that finds its own step constant: a fixed
# number (the tolerance is never met), so every run takes the same steps.
POWER_STEPS = 10
NEVER = 1e-30


def _case(name, call, sky, n_pix, n_vis, extent, n_ant, n_times, radius, height, precision=MIXED,
          gains=False, iters=0):
    return {"name": name, "call": call, "sky": sky, "n_pix": n_pix, "n_vis": n_vis, "extent": extent,
            "n_ant": n_ant, "n_times": n_times, "radius": radius, "height": height, "precision": precision,
            "gains": gains, "iters": iters}


def listed():
    return [
        # the plain FP64 path: a whole small solve from host arrays, where launches count
        _case("solve-fp64-small", "solve", "grid", 32 * 32, 2208, 0.05, 24, 8, 500.0, 5.0, FP64, iters=20),
        # the smallest mixed calls: device pointers on a 32x32 grid ...
        _case("forward-small", "forward", "grid", 32 * 32, 2208, 0.05, 24, 8, 500.0, 5.0),
        # ... and a ragged pixel list through the host-pointer call
        _case("adjoint-ragged-host", "adjoint_host", "list", 1007, 2003, 0.3, 24, 8, 600.0, 10.0),
        # wide field with a strong w term (256x256 over +/-0.5): exact-phase tiles among the others
        _case("forward-wide", "forward", "grid", 256 * 256, 40320, 0.5, 64, 20, 2000.0, 50.0),
        _case("adjoint-wide", "adjoint", "grid", 256 * 256, 40320, 0.5, 64, 20, 2000.0, 50.0),
        # Dirac and three Gaussian scales on a jittered grid with per-antenna beams
        _case("forward-gains", "forward", "multiscale", 4 * 128 * 128, 32000, 0.25, 64, 16, 1000.0, 20.0, gains=True),
        _case("adjoint-gains", "adjoint", "multiscale", 4 * 128 * 128, 32000, 0.25, 64, 16, 1000.0, 20.0, gains=True),
        # the plain FP64 adjoint of a multiscale sky: the reference a user checks the mixed path against
        _case("adjoint-fp64", "adjoint", "multiscale", 4 * 64 * 64, 8064, 0.25, 64, 4, 1000.0, 20.0, FP64),
        # the paper's lambda-sweep setting (30 arcsec pixels, 36 antennas): the first steps of a solve
        _case("solve-table1", "solve", "grid", 1024 * 1024, 37800, 0.0745, 36, 60, 3000.0, 5.0, iters=5),
        # paper scale: one product with the operator and one with its adjoint
        _case("forward-paper-scale", "forward", "grid", 1024 * 1024, 406400, 0.3, 128, 50, 1000.0, 30.0),
        _case("adjoint-paper-scale", "adjoint", "grid", 1024 * 1024, 406400, 0.3, 128, 50, 1000.0, 30.0),
        # four requests of the serving mix (Dirac / Gaussian pixels, without / with gains) through the server
        _case("serve-mix", "serve", "mix", 4096, 6000, 0.1, 36, 10, 1000.0, 20.0, iters=25),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choice(["forward", "adjoint", "forward", "adjoint", "forward_host", "adjoint_host", "solve", "serve"])
    n_vis = int(_log_uniform(rng, 500, 406400))
    n_pix = int(_log_uniform(rng, 256, 1024 * 1024))
    sky = rng.choice(["grid", "grid", "list", "multiscale"])
    precision = FP64 if rng.random() < 0.2 else MIXED
    gains = rng.random() < 0.25
    iters = 0
    # the largest number of pairs of a pass, by what a pair costs
    most = 4.0e11
    if sky == "multiscale":
        most = 2.0e11
    if gains:
        most = 2.1e9
    if precision == FP64:
        most = 2.0e8
    if call == "solve":
        iters = rng.randrange(3, 25)
        most /= 2 * (iters + POWER_STEPS)
    if call == "serve":
        sky, precision, gains, iters = "mix", MIXED, False, rng.randrange(10, 40)
        n_vis, n_pix = int(_log_uniform(rng, 2000, 20000)), int(_log_uniform(rng, 1000, 16384))
        most = 1.0e8
    while n_vis * n_pix > most:
        n_vis, n_pix = max(500, int(0.8 * n_vis)), max(256, int(0.8 * n_pix))
        if n_vis == 500 and n_pix == 256:
            break
    # whole images and whole sets of scales
    if sky in ("grid", "mix"):
        n_pix = max(8, math.isqrt(n_pix)) ** 2
    elif sky == "multiscale":
        n_pix = 4 * max(8, math.isqrt(n_pix // 4)) ** 2
    n_ant = rng.randrange(24, 129)
    if gains:
        n_ant = min(n_ant, max(24, 5_000_000 // n_pix))
    n_times = -(-n_vis // (n_ant * (n_ant - 1) // 2))
    return {"call": call, "sky": sky, "n_pix": n_pix, "n_vis": n_vis, "extent": _log_uniform(rng, 0.05, 0.5),
            "n_ant": n_ant, "n_times": n_times, "radius": _log_uniform(rng, 500.0, 3000.0),
            "height": _log_uniform(rng, 5.0, 50.0), "precision": precision, "gains": gains, "iters": iters}


# ------------------------------------------------------------------ inputs

def _pixels(rng, case, sky):
    """Positions, Gaussian scales and kinds of the pixels, and the bright ones."""
    n_pix, extent = case["n_pix"], case["extent"]
    sigma = kind = None
    if sky == "list":
        lm = rng.uniform(-extent, extent, (n_pix, 2))
        inner = np.flatnonzero(np.abs(lm).max(axis=1) < 0.8 * extent)
        inner = inner if inner.size else np.arange(n_pix)
    elif sky == "multiscale":
        side = math.isqrt(n_pix // 4)
        delta = 2 * extent / side
        base = synth.regular_grid(side, extent)
        base = base + rng.uniform(-0.3 * delta, 0.3 * delta, base.shape)
        scales = [0.0, 1.0, 2.0, 4.0]
        lm = np.concatenate([base] * 4)
        sigma = np.repeat(np.array(scales) * delta, base.shape[0])
        kind = np.where(sigma == 0, synth.DIRAC, synth.GAUSS_WIDE).astype(np.int32)
        inner = synth.inner_pixels(side)
        inner = np.concatenate([inner + k * base.shape[0] for k in range(4)])
    else:
        side = math.isqrt(n_pix)
        lm = synth.regular_grid(side, extent)
        inner = synth.inner_pixels(side)
        if sky == "gauss":
            kind = np.full(n_pix, synth.GAUSS_WIDE, np.int32)
            sigma = np.full(n_pix, 1.5 * 2 * extent / side)
    return lm, sigma, kind, inner


def _inputs(case, seed, sky=None, gains=None):
    """One problem's inputs: arrays in host memory, as a program reads them."""
    rng = synth.rng_for(seed)
    sky = case["sky"] if sky is None else sky
    gains = case["gains"] if gains is None else gains
    enu = synth.antennas(rng, case["n_ant"], case["radius"], case["height"])
    uvw, ant = synth.uvw_tracks(enu, -30.0, case["n_times"])
    uvw, ant = uvw[:case["n_vis"]], ant[:case["n_vis"]]
    lm, sigma, kind, inner = _pixels(rng, case, sky)
    d = {"uvw": uvw, "ant": ant, "lm": lm, "sigma": sigma, "kind": kind, "gains": None}
    if gains:
        d["gains"] = synth.beam_gains(rng, lm, case["n_ant"])
    # an image as an iteration holds it: sources, and faint positive flux on a tenth of the pixels
    x = np.zeros(lm.shape[0])
    src = rng.choice(inner, size=min(50, max(1, inner.size // 8)), replace=False)
    faint = rng.choice(lm.shape[0], size=max(1, lm.shape[0] // 10), replace=False)
    x[faint] = rng.exponential(0.01, faint.size)
    x[src] = rng.exponential(1.0, src.size) + 0.1
    d["x"], d["src"] = x, src
    d["r"] = synth.complex_noise(rng, uvw.shape[0], 1.0)
    if case["call"] in ("solve", "serve"):       # measured data: the sources and noise
        d["vis"] = _measure(d) + synth.complex_noise(rng, uvw.shape[0], 0.01)
        d["lambda"] = 0.01 * uvw.shape[0] * float(x[src].max())
    return d


def _entries(d, rows, cols, dev="cuda"):
    """A[rows, cols] in FP64: the operator's entries as the paper writes them."""
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
    u, v, w = (t(d["uvw"][rows, i])[:, None] for i in range(3))
    l, m = (t(d["lm"][cols, i])[None, :] for i in range(2))
    r2 = l * l + m * m
    n = torch.sqrt(1.0 - r2)
    nm1 = -r2 / (1.0 + n)
    ph = u * l
    ph += v * m
    ph += w * nm1
    amp, beta = None, None
    if d["kind"] is not None:                    # wide-field Gaussians (a Dirac pixel is sigma = 0)
        s2 = t(d["sigma"][cols])[None, :] ** 2
        beta = w * s2
        id_ = 1.0 / (1.0 + beta * beta)
        amp = torch.exp(-math.pi * s2 * id_ * ((u - w * l) ** 2 + (v - w * m) ** 2)) * id_
        ph -= beta * beta * id_ * (u * l + v * m - 0.5 * w * r2) - 0.5 * id_ * beta * s2 * (u * u + v * v)
    ph -= torch.round(ph)
    ph *= -2.0 * math.pi
    a = torch.complex(torch.cos(ph), torch.sin(ph))
    del ph
    a /= n
    if amp is not None:
        a *= torch.complex(amp, amp * beta)
    if d["gains"] is not None:
        g = torch.as_tensor(d["gains"][cols], device=dev)
        ab = torch.as_tensor(d["ant"][rows].astype(np.int64), device=dev)
        a *= g[:, ab[:, 0]].T
        a *= g[:, ab[:, 1]].T.conj()
    return a


def _measure(d):
    a = _entries(d, slice(None), d["src"])
    return (a @ torch.as_tensor(d["x"][d["src"]], dtype=torch.complex128, device="cuda")).cpu().numpy()


def _problem(ctx, d):
    p = ctx.problem()
    p.set_visibilities(d["uvw"], d.get("vis"), None, d["ant"])
    p.set_pixels(d["lm"], d["sigma"], d["kind"])
    if d["gains"] is not None:
        p.set_gains(d["gains"])
    return p


# the serving mix: pixel kind and gains of the four requests
MIX = [("grid", False), ("gauss", False), ("grid", True), ("gauss", True)]


def _mix(case, seed):
    return [_inputs(case, 4 * seed + i, sky, gains) for i, (sky, gains) in enumerate(MIX)]


def prepare(case, seed):
    call = case["call"]
    stream = torch.cuda.Stream()
    ctx = sl1m.Context(0, stream=stream)
    s = {"case": case, "stream": stream, "ctx": ctx, "prec": PREC[case["precision"]]}
    if call == "serve":
        ds = _mix(case, seed)
        s["problems"] = [_problem(ctx, d) for d in ds]
        s["lambdas"] = [d["lambda"] for d in ds]
        ctx.server_start(precision=s["prec"])
        return s
    d = _inputs(case, seed)
    s["problem"] = _problem(ctx, d)
    if call == "solve":
        s["lambda"] = d["lambda"]
    elif call == "forward":
        s["x"] = torch.as_tensor(d["x"], device="cuda")
        s["out"] = torch.empty((d["uvw"].shape[0], 2), dtype=torch.float64, device="cuda")
    elif call == "adjoint":
        s["r"] = torch.view_as_real(torch.as_tensor(d["r"], device="cuda")).contiguous()
        s["out"] = torch.empty(d["lm"].shape[0], dtype=torch.float64, device="cuda")
    else:
        s["x"], s["r"] = d["x"], d["r"]
    return s


# -------------------------------------------------------------------- calls

def run(s):
    case, prec = s["case"], s["prec"]
    call = case["call"]
    single = prec == sl1m.MIXED
    if call == "serve":
        ctx = s["ctx"]
        tickets = [ctx.server_submit(p, lam, max_iter=case["iters"], power_max_iter=POWER_STEPS, power_tol=NEVER)
                   for p, lam in zip(s["problems"], s["lambdas"])]
        images = [ctx.server_wait(t, p)[0] for t, p in zip(tickets, s["problems"])]
        return [im.astype(np.float32) for im in images] if single else images
    p = s["problem"]
    if call == "solve":
        img, st = p.solve(s["lambda"], max_iter=case["iters"], power_max_iter=POWER_STEPS, power_tol=NEVER,
                          precision=prec)
        real = np.float32 if single else np.float64
        return {"image": img.astype(real), "E": real(st["E"]), "L": real(st["L"])}
    if call == "forward":
        p.forward_dev(s["x"], s["out"], prec)
    elif call == "adjoint":
        p.adjoint_dev(s["r"], s["out"], prec)
    elif call == "forward_host":
        vis = p.forward(s["x"], prec)
        return vis.astype(np.complex64) if single else vis
    else:
        img = p.adjoint(s["r"], prec)
        return img.astype(np.float32) if single else img
    if not single:
        return s["out"]
    with torch.cuda.stream(s["stream"]):
        return s["out"].float()


# ------------------------------------------------------- what a pass needs

def work(case):
    n_vis, n_pix, call = case["n_vis"], case["n_pix"], case["call"]
    # phase (3 multiply-adds), sine and cosine, and the accumulation (2
    # multiply-adds; the adjoint's real output needs one of each) per pair
    fwd, adj = 12, 9
    ops = {"forward": fwd, "forward_host": fwd, "adjoint": adj, "adjoint_host": adj}.get(call)
    if ops is None:
        ops = (case["iters"] + POWER_STEPS + 1) * fwd + (case["iters"] + POWER_STEPS) * adj
    problems = 4 if call == "serve" else 1
    # coordinates, data or residual, and the image, each once
    nbytes = n_vis * (24 + 16) + n_pix * (16 + 8)
    if case["gains"]:
        nbytes += n_pix * case["n_ant"] * 16
    return {"bytes": problems * nbytes, "flops": problems * n_vis * n_pix * ops}


# ------------------------------------------------- the same in 64-bit torch

MAX_PAIRS = 1.2e10            # about 10 s of FP64 sines and cosines
MAX_HELD = 3.0e9              # entries held as a matrix over a solve's steps


def _row_blocks(d, per_block=3.0e7):
    n_vis, n_pix = d["uvw"].shape[0], d["lm"].shape[0]
    step = max(1, int(per_block / n_pix))
    return [slice(i, min(n_vis, i + step)) for i in range(0, n_vis, step)]


class _Operator:
    """The operator in FP64, its entries kept when they are used again."""

    def __init__(self, d, keep):
        self.d = d
        self.rows = _row_blocks(d)
        self.held = [_entries(d, b, slice(None)) for b in self.rows] if keep else None

    def _block(self, i):
        return self.held[i] if self.held else _entries(self.d, self.rows[i], slice(None))

    def forward(self, x):
        xc = x.to(torch.complex128)
        return torch.cat([self._block(i) @ xc for i in range(len(self.rows))])

    def adjoint(self, r):
        g = torch.zeros(self.d["lm"].shape[0], dtype=torch.float64, device="cuda")
        for i, b in enumerate(self.rows):
            g += (r[b].conj() @ self._block(i)).real
        return g


def _fista(d, iters):
    """POWER_STEPS steps for L, then `iters` steps of the algorithm box from zero."""
    op = _Operator(d, True)
    n = d["lm"].shape[0]
    x = torch.full((n,), 1.0 / math.sqrt(n), dtype=torch.float64, device="cuda")
    L = 0.0
    for _ in range(POWER_STEPS):
        z = op.adjoint(op.forward(x))
        L = float(torch.linalg.vector_norm(z))
        x = z / L
    vis = torch.as_tensor(d["vis"], device="cuda")
    img = torch.zeros_like(x)
    y, t = img, 1.0
    for _ in range(iters):
        g = op.adjoint(op.forward(y) - vis)
        new = torch.clamp(y - g / L - d["lambda"] / L, min=0.0)
        t1 = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        y = new + ((t - 1.0) / t1) * (new - img)
        img, t = new, t1
    res = op.forward(img) - vis
    E = 0.5 * float((res.abs() ** 2).sum()) + d["lambda"] * float(img.sum())
    return img.cpu().numpy(), np.float64(E), np.float64(L)


def exact(case, seed):
    call, pairs = case["call"], float(case["n_vis"]) * case["n_pix"]
    if call == "serve":
        return [_fista(d, case["iters"])[0] for d in _mix(case, seed)] if pairs <= MAX_HELD else None
    if pairs > (MAX_HELD if call == "solve" else MAX_PAIRS):
        return None
    d = _inputs(case, seed)
    if call == "solve":
        img, E, L = _fista(d, case["iters"])
        return {"image": img, "E": E, "L": L}
    op = _Operator(d, False)
    if call.startswith("forward"):
        vis = op.forward(torch.as_tensor(d["x"], device="cuda"))
        return vis.cpu().numpy() if call == "forward_host" else torch.view_as_real(vis)
    img = op.adjoint(torch.as_tensor(d["r"], device="cuda"))
    return img.cpu().numpy() if call == "adjoint_host" else img
