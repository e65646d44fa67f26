"""The work that a program using this framework has it do, as cases for timing.

Every case goes through the public entry points of `paper_2507_00294_gb300.binding` and
`.surrogate`.  Units are those of `workloads.py`: a probe pitch of 0.5 nm, a probe sigma
near 0.1 nm, a dwell near 1 us, and a diffusion coefficient D of the case, each moved by a
few per cent by the seed, which also draws point lists, per-visit dwells and random orders.

The FP32-mixed path carries FP32 accuracy in its FP64 output buffer, so a program that
evaluates damage maps or doses in that precision keeps them in FP32 (`run` converts them);
FP64 results stay FP64.
"""
import math

import numpy as np
import torch

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import surrogate as sur
from paper_2507_00294_gb300 import workloads as w

PITCH = w.PITCH
ORDERS = {"raster": w.RASTER, "serpentine": w.SERPENTINE, "interleaved": w.INTERLEAVED, "random": w.RANDOM}
CANVAS = sur.CANVAS
DEV = "cuda:0"


def listed():
    return [
        # the paper's own 20 x 20 acquisition: the dose of each probe when its dwell starts, in
        # the reference precision -- the smallest call, all launches and latency
        dict(name="dose_20_fp64", kind="dose", nx=20, ny=20, order="raster", D=6e-14, timing="uniform",
             keep=1.0, prec="fp64"),
        # a small live view: the probe grid at the end of each of the 256 dwells
        dict(name="grid_16_every_dwell", kind="grid", nx=16, ny=16, order="raster", D=6e-14, timing="uniform",
             keep=1.0, cols=16, rows=16, step=1.0, n_t=256, snap="even", prec="mixed"),
        # the benchmark's field: a 64 x 64 raster on a 2x supersampled simulation grid after each row
        dict(name="grid_64_rows", kind="grid", nx=64, ny=64, order="raster", D=6e-14, timing="uniform",
             keep=1.0, cols=128, rows=128, step=0.5, n_t=64, snap="even", prec="mixed"),
        # an ordinary acquisition that is not ideal: odd sizes, every dwell its own length and a
        # flyback at each row, live frames between dwell boundaries, a grid finer than the probe's
        dict(name="grid_77x53_dwells", kind="grid", nx=77, ny=53, order="serpentine", D=2e-14, timing="dwells",
             keep=1.0, cols=131, rows=97, step=0.58, n_t=24, snap="frames", prec="mixed"),
        # the precision study's size: 65,536 visits, at the end of the scan and long after it
        dict(name="grid_256_interleaved", kind="grid", nx=256, ny=256, order="interleaved", D=1e-13,
             timing="uniform", keep=1.0, cols=256, rows=256, step=1.0, n_t=2, snap="late", prec="mixed"),
        # the reference precision on a simulation grid, as used to check the mixed path
        dict(name="grid_40_fp64", kind="grid", nx=40, ny=40, order="random", D=6e-14, timing="uniform",
             keep=0.8, cols=96, rows=81, step=0.5, n_t=12, snap="even", prec="fp64"),
        # scattered evaluation points (not a grid) over a subsampled random scan
        dict(name="points_64_random", kind="points", nx=64, ny=64, order="random", D=6e-14, timing="uniform",
             keep=0.6, n_pts=10007, n_t=33, snap="frames", prec="mixed"),
        # the dose of every probe of a large scan
        dict(name="dose_256", kind="dose", nx=256, ny=256, order="raster", D=6e-14, timing="uniform",
             keep=1.0, prec="mixed"),
        # the uneven batch of 512 scans, each on its probe grid at its end: one plan, run again
        dict(name="batch_grid_512", kind="batch_grid", n_scans=512, n_min=32, n_max=128, prec="mixed"),
        # the same kind of batch at each scan's own list of points (spot checks, regions of interest)
        dict(name="batch_points_256", kind="batch_points", n_scans=256, n_min=32, n_max=128, n_pts=997,
             prec="mixed"),
        # one hidden layer of the surrogate's training step: forward, both gradients, Adam
        dict(name="surrogate_layer_32", kind="layer", B=32, cin=32, cout=32, dilation=4),
        # the surrogate's inference on a batch of maps: input planes and all six layers
        dict(name="surrogate_infer_256", kind="infer", B=256),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "points", "dose", "dose", "batch_grid", "batch_points", "layer",
                       "infer"])
    if kind == "infer":
        return dict(kind=kind, B=rng.randint(16, 256))
    if kind == "layer":
        cin, cout = rng.choice([(16, 32), (32, 32), (32, 32), (32, 16)])
        return dict(kind=kind, B=rng.randint(8, 48), cin=cin, cout=cout, dilation=rng.randint(1, 32))
    if kind.startswith("batch"):
        c = dict(kind=kind, n_scans=int(_log(rng, 8, 512 if kind == "batch_grid" else 256)),
                 n_min=rng.randint(24, 48), n_max=rng.randint(64, 128), prec="mixed")
        if kind == "batch_points":
            c["n_pts"] = int(_log(rng, 64, 1000))
        return c
    fp64 = rng.random() < 0.25
    order = rng.choice(["raster", "raster", "serpentine", "interleaved", "random"])
    keep = rng.uniform(0.3, 1.0) if order == "random" else 1.0
    timing = rng.choice(["uniform", "uniform", "uniform", "dwells"])
    c = dict(kind=kind, order=order, D=_log(rng, 1e-15, 1e-12), timing=timing, keep=keep,
             prec="fp64" if fp64 else "mixed")
    hi = {"grid": 40 if fp64 else 160, "points": 32 if fp64 else 80,
          "dose": 48 if fp64 or timing == "dwells" else 256}[kind]
    c["nx"], c["ny"] = int(_log(rng, 12, hi)), int(_log(rng, 12, hi))
    if kind == "dose":
        return c
    c["snap"] = rng.choice(["even", "even", "frames", "late"])
    visits = c["nx"] * c["ny"] * keep
    most = 4e7 if fp64 else 2e9                     # causal pairs, about
    if kind == "grid":
        c["step"] = rng.choice([0.25, 0.5, 0.5, 1.0, round(rng.uniform(0.3, 1.2), 3)])
        c["cols"] = min(int(c["nx"] / c["step"]), 300) + rng.randint(0, 5)
        c["rows"] = min(int(c["ny"] / c["step"]), 300) + rng.randint(0, 5)
        pts = c["cols"] * c["rows"]
    else:
        c["n_pts"] = pts = int(_log(rng, 300, 4000 if fp64 else 20000))
        most /= 4
    most_t = max(1, int(2 * most / (visits * pts)))
    c["n_t"] = 2 if c["snap"] == "late" else max(1, min(most_t, int(_log(rng, 1, 128)), int(visits)))
    return c


# ------------------------------------------------------------------------------ inputs

def _physics(case, seed):
    rng = np.random.default_rng([seed, 1])
    return dict(D=case["D"] * 10.0 ** rng.uniform(-0.04, 0.04), dwell=1e-6 * 10.0 ** rng.uniform(-0.04, 0.04),
                sigma=w.SIGMA * rng.uniform(0.95, 1.05))


def _n_visits(case):
    n = case["nx"] * case["ny"]
    return max(int(math.floor(case["keep"] * n + 0.5)), 1) if case["keep"] < 1.0 else n


def _timing(case, seed, dwell):
    """(per-visit dwells or None, flyback): 'dwells' draws every dwell within a factor two and
    gives the orders that have rows a flyback."""
    if case["timing"] == "uniform":
        return None, 0.0
    rng = np.random.default_rng([seed, 2])
    tau = dwell * rng.uniform(0.7, 1.4, _n_visits(case))
    return tau, 5.3 * dwell if case["order"] in ("raster", "serpentine") else 0.0


def _spec(case, seed):
    p = _physics(case, seed)
    tau, flyback = _timing(case, seed, p["dwell"])
    return w.ScanSpec(case["nx"], case["ny"], sigma_m=p["sigma"], D_m2s=p["D"], dwell_s=p["dwell"],
                      order=ORDERS[case["order"]], interleave_stride=4 if case["order"] == "interleaved" else 1,
                      seed=seed, keep_fraction=case["keep"], dwell_per_visit=tau, flyback_s=flyback)


def _times(case, seed):
    """Snapshot times in nominal dwells: 'even' whole dwells spread over the scan (its row ends
    when there is one per row), 'frames' between dwell boundaries, 'late' the end and 16 x it."""
    n, n_t = _n_visits(case), case["n_t"]
    end = float(n)
    if case["timing"] != "uniform":
        p = _physics(case, seed)
        tau, flyback = _timing(case, seed, p["dwell"])
        end = (tau.sum() + flyback * (case["ny"] - 1)) / p["dwell"]
    if case["snap"] == "late":
        return np.array([end, 16.0 * end])
    t = np.arange(1, n_t + 1, dtype=np.float64) * (end / n_t)
    return np.maximum(np.rint(t), 1.0) if case["snap"] == "even" else t - 0.37


def _points(case, seed):
    """Scattered points over the scan's area and one pitch around it [m]."""
    rng = np.random.default_rng([seed, 3])
    ext = np.array([case["nx"] + 1.0, case["ny"] + 1.0])
    return (rng.random((case["n_pts"], 2)) * ext - 1.0) * PITCH


def _batch_specs(case, seed):
    """The uneven batch's scans: their sizes belong to the case, their physics and random
    orders come from the seed."""
    sizes, drawn = (w.batched_specs(case["n_scans"], seed=k, n_min=case["n_min"], n_max=case["n_max"])
                    for k in (4, 5 + seed % 1000003))
    return [a.with_(nx=q.nx, ny=q.ny, keep_fraction=q.keep_fraction) for q, a in zip(sizes, drawn)]


def _batch_points(case, specs, seed):
    rng = np.random.default_rng([seed, 4])
    return [rng.random((case["n_pts"], 2)) * (s.nx - 1) * PITCH for s in specs]


def _maps(case, seed):
    """Time maps [B, H, W] (1 / age of each visit in dwells, -1 where not visited) and scalars
    (standardised log D and log dwell, kappa) of random scans of 32^2 to 128^2 positions."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    B, n = case["B"], CANVAS * CANVAS
    rng = np.random.default_rng([seed, 5])
    side = rng.integers(32, CANVAS + 1, B)
    keep = rng.uniform(0.1, 1.0, B)
    iy, ix = torch.meshgrid(torch.arange(CANVAS, device=DEV), torch.arange(CANVAS, device=DEV), indexing="ij")
    side_t = torch.tensor(side, device=DEV)[:, None, None]
    inside = ((iy < side_t) & (ix < side_t)).view(B, n)
    rank = torch.where(inside, torch.rand((B, n), generator=gen, device=DEV), 2.0).argsort(1).argsort(1)
    visits = torch.tensor(np.maximum((side * side * keep).astype(np.int64), 1), device=DEV)[:, None]
    tmap = torch.where(rank < visits, 1.0 / (visits - rank).float(), -1.0).view(B, CANVAS, CANVAS).contiguous()
    logD, logt = rng.uniform(-15.0, -12.0, B), rng.uniform(-7.0, -5.0, B)
    scal = np.stack([(logD + 13.5) / 1.5, logt + 6.0, 10.0 ** (logD + logt) / PITCH ** 2], 1).astype(np.float32)
    return tmap, torch.from_numpy(scal).to(DEV)


def _layer(case, seed):
    """A layer in training: its input (behind a ReLU), weights, and the gradient of its output."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    B, ci, co = case["B"], case["cin"], case["cout"]
    bf = torch.bfloat16
    x = torch.relu(torch.randn((B, CANVAS, CANVAS, ci), generator=g, device=DEV)).to(bf)
    dz = (torch.randn((B, CANVAS, CANVAS, co), generator=g, device=DEV) * 1e-5).to(bf)
    wt = torch.randn((co, 9, ci), generator=g, device=DEV) * math.sqrt(2.0 / (9 * ci))
    bias = torch.randn(co, generator=g, device=DEV) * 0.05
    return x, dz, wt, bias


def _weights(seed):
    """Each layer's weights [cout, 9, cin] (its real channels; the padded ones zero) and biases."""
    rng = np.random.default_rng([seed, 6])
    out = []
    for k, (ci, co) in enumerate(sur.LAYERS):
        real_ci = sur.REAL_IN if k == 0 else ci
        real_co = sur.REAL_OUT if k == len(sur.LAYERS) - 1 else co
        wt, bias = np.zeros((co, 9, ci), np.float32), np.zeros(co, np.float32)
        wt[:real_co, :, :real_ci] = rng.standard_normal((real_co, 9, real_ci)) * math.sqrt(2.0 / (9 * real_ci))
        bias[:real_co] = rng.standard_normal(real_co) * 0.05
        out.append((torch.from_numpy(wt), torch.from_numpy(bias)))
    return out


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("dose", "grid", "points"):
        spec = _spec(case, seed)
        s["scan"] = b.Scan(spec)
        if kind == "dose":
            s["out"] = torch.empty(_n_visits(case), dtype=torch.float64, device=DEV)
            return s
        s["times"] = _times(case, seed) * spec.dwell_s
        if kind == "points":
            s["pts"] = torch.from_numpy(_points(case, seed)).to(DEV)
            n_pts = case["n_pts"]
        else:
            n_pts = case["cols"] * case["rows"]
        s["out"] = torch.empty((len(s["times"]), n_pts), dtype=torch.float64, device=DEV)
    elif kind.startswith("batch"):
        specs = _batch_specs(case, seed)
        scans = [b.Scan(q) for q in specs]
        times = np.array([w.n_visits(q) * q.dwell_s for q in specs])
        if kind == "batch_grid":
            s["plan"] = b.Batch(scans, None, times, case["prec"],
                                grids=[(0.0, 0.0, q.pitch_m, q.pitch_m, q.nx, q.ny) for q in specs])
            s["pts"] = None
        else:
            pts = _batch_points(case, specs, seed)
            offs = np.arange(len(specs) + 1) * case["n_pts"]
            s["plan"] = b.Batch(scans, offs, times, case["prec"])
            s["pts"] = torch.from_numpy(np.concatenate(pts)).to(DEV)
        s["out"] = torch.empty(s["plan"].total, dtype=torch.float64, device=DEV)
    elif kind == "layer":
        x, dz, wt, bias = _layer(case, seed)
        ci, co = case["cin"], case["cout"]
        bf = torch.bfloat16
        s.update(x=x, dz=dz, param=torch.cat([wt.reshape(-1), bias]), wb=wt.to(bf),
                 wf=wt.flip(1).permute(2, 1, 0).contiguous().to(bf), step=0)
        s["y"] = torch.empty((*x.shape[:3], co), dtype=bf, device=DEV)
        s["dx"] = torch.empty_like(x)
        s["part"] = torch.empty(608 * (co * 9 * ci + co), dtype=torch.float32, device=DEV)
        s["grad"] = torch.zeros_like(s["param"])
        s["m"], s["v"] = torch.zeros_like(s["param"]), torch.zeros_like(s["param"])
    else:
        s["tmap"], s["scal"] = _maps(case, seed)
        net = s["net"] = sur.Net(DEV)
        for k, (wt, bias) in enumerate(_weights(seed)):
            net.params[k].copy_(torch.cat([wt.reshape(-1), bias]))
            net.wb[k].copy_(wt)
            net.wf[k].copy_(wt.flip(1).permute(2, 1, 0))
        net.buffers(case["B"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "dose":
        out = b.dd_per_probe_dose(s["scan"], case["prec"], out=s["out"])
    elif kind == "grid":
        step = case["step"] * PITCH
        out = b.dd_field_on_grid(s["scan"], 0.0, 0.0, step, step, case["cols"], case["rows"], s["times"],
                                 case["prec"], out=s["out"])
    elif kind == "points":
        out = b.dd_field_at_times(s["scan"], s["pts"], s["times"], case["prec"], out=s["out"])
    elif kind.startswith("batch"):
        out = s["plan"].run(s["pts"], out=s["out"])
    elif kind == "layer":
        n, d = s["wb"].numel(), case["dilation"]
        s["step"] += 1
        b.dd_sur_conv3x3(s["x"], s["wb"], s["param"][n:], None, s["y"], 0, d)
        b.dd_sur_wgrad(s["x"], s["dz"], s["part"], s["grad"], d)
        b.dd_sur_conv3x3(s["dz"], s["wf"], None, s["x"], s["dx"], 2, d)
        p, g, m, v = s["param"], s["grad"], s["m"], s["v"]
        b.dd_sur_adam(p[:n], g[:n], m[:n], v[:n], 1e-3, s["step"], w_bf16=s["wb"], w_flip=s["wf"],
                      cin=case["cin"], cout=case["cout"])
        b.dd_sur_adam(p[n:], g[n:], m[n:], v[n:], 1e-3, s["step"])
        return dict(y=s["y"], dx=s["dx"], grad=g, param=p)
    else:
        return sur.predict(s["net"], s["tmap"], s["scal"], batch=case["B"])
    return out.float() if case["prec"] == "mixed" else out


# ------------------------------------------------------------------------------- work

def _pairs(case):
    """Causal (visit, point, snapshot) pairs of a field or dose case."""
    n = _n_visits(case)
    if case["kind"] == "dose":
        return n * (n - 1) / 2.0
    pts = case["n_pts"] if case["kind"] == "points" else case["cols"] * case["rows"]
    n_t = case["n_t"]
    return pts * (2.0 * n if case["snap"] == "late" else n * (n_t + 1) / 2.0)


def work(case):
    return {k: float(v) for k, v in _work(case).items()}


def _work(case):
    """The direct sum's pairs at the operations one needs at least: on a grid of points a
    multiply-add (the exponentials split into column and row factors), elsewhere the squared
    distance (3), the exponent (1), one exponential (1) and a multiply-add (2); visits (24 B),
    points (16 B) and weights read once, results written once."""
    kind = case["kind"]
    if kind == "infer":
        px = case["B"] * CANVAS * CANVAS
        taps = 9 * (sur.REAL_IN * 32 + 4 * 32 * 32 + 32 * sur.REAL_OUT)
        return {"bytes": px * 8.0, "flops": 2.0 * px * taps}
    if kind == "layer":
        px, ci, co = case["B"] * CANVAS * CANVAS, case["cin"], case["cout"]
        return {"bytes": 2.0 * px * (2 * ci + 2 * co) + 28.0 * 9 * ci * co, "flops": 3 * 2.0 * px * 9 * ci * co}
    if kind.startswith("batch"):
        m, k = case["n_max"] - case["n_min"], np.arange(case["n_min"], case["n_max"] + 1, dtype=np.float64)
        n2, n4 = (k ** 2).sum() / (m + 1), (k ** 4).sum() / (m + 1)
        if kind == "batch_grid":                   # keep fraction 0.55 on average
            return {"bytes": case["n_scans"] * (0.55 * 24 + 8) * n2, "flops": case["n_scans"] * 2 * 0.55 * n4}
        return {"bytes": case["n_scans"] * (0.55 * 24 * n2 + 24 * case["n_pts"]),
                "flops": case["n_scans"] * 7 * 0.55 * n2 * case["n_pts"]}
    n = _n_visits(case)
    if kind == "dose":
        return {"bytes": 32.0 * n, "flops": 7 * _pairs(case)}
    n_t = 2 if case["snap"] == "late" else case["n_t"]
    if kind == "grid":
        return {"bytes": 24.0 * n + 8.0 * n_t * case["cols"] * case["rows"], "flops": 2 * _pairs(case)}
    return {"bytes": 24.0 * n + (16 + 8.0 * n_t) * case["n_pts"], "flops": 7 * _pairs(case)}


# --------------------------------------------------------------- the same in 64 bits
#
# A visit's term E1(rho^2 / w1) - E1(rho^2 / w0) is the integral of exp(-(rho^2 / w1) e^y)
# over y in [0, ln(w1 / w0)] (u = (rho^2 / w1) e^y in E1's own integral), taken here by
# Gauss-Legendre with enough nodes for FP64 where the term matters.

def _splitmix_permutation(n, seed):
    """Fisher-Yates driven by SplitMix64: i from n - 1 down to 1 swaps with floor(u (i + 1) / 2^64)."""
    mask, x, p = (1 << 64) - 1, seed & ((1 << 64) - 1), list(range(n))
    for i in range(n - 1, 0, -1):
        x = (x + 0x9E3779B97F4A7C15) & mask
        z = x
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        z ^= z >> 31
        j = (z * (i + 1)) >> 64
        p[i], p[j] = p[j], p[i]
    return np.array(p, dtype=np.int64)


def _visit_xy(nx, ny, order, seed, n):
    """Grid positions (x, y) of the visits in visit order, in pitches."""
    idx = np.arange(nx * ny).reshape(ny, nx)
    if order == "serpentine":
        idx = idx.copy()
        idx[1::2] = idx[1::2, ::-1]
    elif order == "interleaved":
        idx = np.concatenate([idx[py::4, px::4].reshape(-1) for py in range(4) for px in range(4)])
    elif order == "random":
        idx = _splitmix_permutation(nx * ny, seed)[:n]
    idx = idx.reshape(-1)
    return (torch.from_numpy((idx % nx).astype(np.float64)).to(DEV),
            torch.from_numpy((idx // nx).astype(np.float64)).to(DEV))


def _starts(case, seed):
    """(start times, dwells) of the visits in nominal dwells."""
    n = _n_visits(case)
    dwell = _physics(case, seed)["dwell"]
    tau, flyback = _timing(case, seed, dwell)
    if tau is None:
        return np.arange(n, dtype=np.float64), np.ones(n)
    gap = np.zeros(n)
    if flyback:
        gap[case["nx"]::case["nx"]] = flyback
    return (np.concatenate([[0.0], np.cumsum(tau)[:-1]]) + np.cumsum(gap)) / dwell, tau / dwell


def _widths(age, tau, s, kappa):
    """1 / w1 and ln(w1 / w0) of visits of that age (> 0), all in pitches and dwells."""
    w1 = 2 * s + 4 * kappa * age
    return 1.0 / w1, -torch.log1p(-4 * kappa * torch.minimum(age, tau) / w1)


def _nodes(L):
    n = 7 if L <= 0.02 else 13 if L <= 0.3 else 32 if L <= 1.0 else 80
    u, wt = np.polynomial.legendre.leggauss(n)
    return [(0.5 * (1 + float(a)), 0.5 * float(c)) for a, c in zip(u, wt)]


def _by_length(L, most):
    """Index sets of visits, each with the largest ln(w1 / w0) that it holds."""
    edges = [0.0, 0.02, 0.3, 1.0, 1e9]
    for lo, hi in zip(edges, edges[1:]):
        at = torch.nonzero((L > lo) & (L <= hi)).view(-1)
        for part in at.split(most):
            if len(part):
                yield part, min(hi, 1e3)


def _grid_sum(px, py, x, y, iw, L):
    """Field on the grid of columns px and rows py from visits at (x, y): [rows * cols]."""
    F = torch.zeros((len(py), len(px)), dtype=torch.float64, device=DEV)
    for at, most in _by_length(L, 16384):
        dx2, dy2 = (px[None, :] - x[at, None]) ** 2, (py[None, :] - y[at, None]) ** 2
        for u, c in _nodes(most):
            q = (iw[at] * torch.exp(L[at] * u))[:, None]
            F += ((L[at] * c)[:, None] * torch.exp(-q * dy2)).T @ torch.exp(-q * dx2)
    return F.view(-1)


def _list_sum(px, py, x, y, iw, L):
    """Field at the points (px, py) from visits at (x, y)."""
    F = torch.zeros(len(px), dtype=torch.float64, device=DEV)
    for at, most in _by_length(L, max(256, int(3e7) // max(1, len(px)))):
        r2 = (px[:, None] - x[None, at]) ** 2 + (py[:, None] - y[None, at]) ** 2
        for u, c in _nodes(most):
            F += torch.exp(r2 * -(iw[at] * torch.exp(L[at] * u))) @ (L[at] * c)
    return F


def _exact_field(case, seed):
    p = _physics(case, seed)
    s, kappa = (p["sigma"] / PITCH) ** 2, p["D"] * p["dwell"] / PITCH ** 2
    pref = w.Q0 / (4 * math.pi * p["D"])
    n = _n_visits(case)
    x, y = _visit_xy(case["nx"], case["ny"], case["order"], seed, n)
    t0, tau = (torch.from_numpy(v).to(DEV) for v in _starts(case, seed))
    if case["kind"] == "dose":
        out = torch.zeros(n, dtype=torch.float64, device=DEV)
        for j0 in range(0, n, 256):
            j = torch.arange(j0, min(j0 + 256, n), device=DEV)
            for i0, i1 in ((0, max(0, j0 - 256)), (max(0, j0 - 256), min(j0 + 256, n))):
                for a in range(i0, i1, 32768):
                    i = torch.arange(a, min(a + 32768, i1), device=DEV)
                    age = t0[j, None] - t0[None, i]
                    live = age > 0.5 * float(tau.min())
                    iw, L = _widths(age.clamp_min(1e-3), tau[None, i].expand_as(age), s, kappa)
                    r2 = (x[j, None] - x[None, i]) ** 2 + (y[j, None] - y[None, i]) ** 2
                    a2, part = r2 * iw, torch.zeros_like(r2)
                    for u, c in _nodes(float(torch.where(live, L, 0.0).max())):
                        part += c * torch.exp(-a2 * torch.exp(L * u))
                    out[j] += torch.where(live, part * L, 0.0).sum(1)
        return out * pref
    t = torch.from_numpy(_times(case, seed)).to(DEV)
    if case["kind"] == "grid":
        k = np.arange(max(case["cols"], case["rows"])) * (case["step"] * PITCH) / PITCH
        px = torch.from_numpy(k[: case["cols"]].copy()).to(DEV)
        py = torch.from_numpy(k[: case["rows"]].copy()).to(DEV)
    else:
        pts = torch.from_numpy(_points(case, seed) / PITCH).to(DEV)
        px, py = pts[:, 0].contiguous(), pts[:, 1].contiguous()
    rows = []
    for tk in t:
        on = torch.nonzero(t0 < tk).view(-1)
        iw, L = _widths(tk - t0[on], tau[on], s, kappa)
        rows.append((_grid_sum if case["kind"] == "grid" else _list_sum)(px, py, x[on], y[on], iw, L) * pref)
    return torch.stack(rows)


def _exact_batch(case, seed):
    specs = _batch_specs(case, seed)
    pts = _batch_points(case, specs, seed) if case["kind"] == "batch_points" else None
    parts = []
    for k, q in enumerate(specs):
        n = max(int(math.floor(q.keep_fraction * q.nx * q.ny + 0.5)), 1)
        x, y = _visit_xy(q.nx, q.ny, "random", q.seed, n)
        s, kappa = (q.sigma_m / PITCH) ** 2, q.D_m2s * q.dwell_s / PITCH ** 2
        age = n - torch.arange(n, dtype=torch.float64, device=DEV)
        iw, L = _widths(age, torch.ones_like(age), s, kappa)
        pref = q.Q0 / (4 * math.pi * q.D_m2s)
        if pts is None:
            k1 = torch.arange(q.nx, dtype=torch.float64, device=DEV)
            parts.append(_grid_sum(k1, k1, x, y, iw, L) * pref)
        else:
            p = torch.from_numpy(pts[k] / PITCH).to(DEV)
            parts.append(_list_sum(p[:, 0].contiguous(), p[:, 1].contiguous(), x, y, iw, L) * pref)
    return torch.cat(parts)


def _taps(x, d):
    """The nine shifted views of [B, H, W, C] that a dilated 3 x 3 convolution reads."""
    B, H, W, C = x.shape
    z = torch.nn.functional.pad(x, (0, 0, d, d, d, d))
    return [z[:, ky * d: ky * d + H, kx * d: kx * d + W] for ky in range(3) for kx in range(3)]


def _conv(x, wt, d):
    return sum(v @ wt[:, k].T for k, v in enumerate(_taps(x, d)))


def _exact_layer(case, seed):
    x, dz, wt, bias = _layer(case, seed)
    ci, co, d = case["cin"], case["cout"], case["dilation"]
    x, dz, wb = x.double(), dz.double(), wt.to(torch.bfloat16).double()
    y = torch.cat([torch.relu(_conv(q, wb, d) + bias.double()) for q in x.split(8)])
    wf = wb.flip(1).permute(2, 1, 0)
    dx = torch.cat([_conv(q, wf, d) * (m > 0) for q, m in zip(dz.split(8), x.split(8))])
    gw = sum(torch.stack([g.reshape(-1, co).T @ v.reshape(-1, ci) for v in _taps(q, d)], 1)
             for q, g in zip(x.split(8), dz.split(8)))
    grad = torch.cat([gw.reshape(-1), dz.reshape(-1, co).sum(0)])
    p = torch.cat([wt.reshape(-1), bias]).double()
    # the first Adam step: both moments' corrections cancel
    return dict(y=y, dx=dx, grad=grad, param=p - 1e-3 * grad / (grad.abs() + 1e-8))


def _exact_infer(case, seed):
    """The network in 64 bits (its BF16 weights, no rounding of the activations)."""
    tmap, scal = (v.double() for v in _maps(case, seed))
    layers = [(wt.to(DEV).to(torch.bfloat16).double(), bias.to(DEV).double()) for wt, bias in _weights(seed)]
    out = []
    for q, c in zip(tmap.split(8), scal.split(8)):
        on = (q > 0).double()
        age = torch.where(q > 0, 1.0 / q.clamp_min(1e-9), 1.0).round()
        kap = c[:, 2, None, None]
        w0 = 2 * (w.SIGMA / PITCH) ** 2 + 4 * kap * (age - 1)
        bg = on * (age > sur.K_EXACT)
        own = torch.where(bg > 0, (torch.log10(torch.log1p(4 * kap / w0)) - sur.MU) / sur.SIGMA, 0.0)
        one = torch.ones_like(q)
        h = torch.stack([q * on, on, one * c[:, 0, None, None], one * c[:, 1, None, None], own, bg], -1)
        for k, (wt, bias) in enumerate(layers):
            h = _conv(h, wt[:, :, : h.shape[-1]], sur.DILATIONS[k]) + bias
            h = torch.relu(h) if k < len(layers) - 1 else h[..., 0]
        out.append(h)
    return torch.cat(out)


def exact(case, seed):
    with torch.no_grad():
        if case["kind"] in ("dose", "grid", "points"):
            return _exact_field(case, seed)
        if case["kind"].startswith("batch"):
            return _exact_batch(case, seed)
        return _exact_layer(case, seed) if case["kind"] == "layer" else _exact_infer(case, seed)
