"""Performance cases: what a user of this library has it do, over its real range.

Each case is one pass through the public entry points on inputs that are on
the GPU already, with a plan that a user's program keeps.  Samples are spread
so that every grid point has neighbours well above the density mask: a mask
bit that sits on its threshold would say nothing about the kernels.
"""
from __future__ import annotations

import itertools
import math
import statistics

import numpy as np
import torch

from paper_2204_07716_gb300 import fkreg

PROBE_SEED = 7


def listed():
    return [
        # bandwidth selection in one call at the size of the paper's own 1-D
        # example: 10 candidates, 200 samples; all latency
        {"name": "select-1d-200", "kind": "select", "d": 1, "order": 0, "n": 200, "g0": 100,
         "n_bw": 10, "s_lo": 0.03, "s_hi": 0.2, "probes": 10, "precision": "f64"},
        # the 1-D Nadaraya-Watson configuration, FP64 at nine digits: small
        # launches one after the other
        {"name": "nw1d-10k-f64", "kind": "smooth", "d": 1, "order": 0, "n": 10_000, "g0": 256,
         "sigma": 0.02, "precision": "f64", "tol": 1e-9, "rhs": 1, "complex": False},
        # an ordinary 2-D data set: estimate, log-variance, interval, values
        # at new points
        {"name": "ll2d-20k-interval", "kind": "interval", "d": 2, "order": 1, "n": 20_011,
         "g0": 100, "g1": 121, "sigma": 0.03, "new": 5003, "precision": "f32"},
        # 2-D local linear in FP64 at twelve digits, ragged sizes
        {"name": "ll2d-200k-f64", "kind": "smooth", "d": 2, "order": 1, "n": 200_003, "g0": 129,
         "g1": 161, "sigma": 0.02, "precision": "f64", "tol": 1e-12, "rhs": 1, "complex": False},
        # the headline configuration: fit, Monte-Carlo degrees of freedom,
        # GCV and the conditional variance of 10^6 clustered samples
        {"name": "ll2d-1M-step", "kind": "step", "d": 2, "order": 1, "n": 1_000_000, "g0": 256,
         "g1": 256, "sigma": 0.01, "probes": 10, "precision": "f32", "kernel": "gaussian"},
        # local quadratic, 2-D
        {"name": "lq2d-300k", "kind": "smooth", "d": 2, "order": 2, "n": 300_007, "g0": 128,
         "g1": 96, "sigma": 0.03, "precision": "f32", "tol": 1e-6, "rhs": 1, "complex": False},
        # local linear, 3-D
        {"name": "ll3d-300k", "kind": "smooth", "d": 3, "order": 1, "n": 300_001, "g0": 37,
         "g1": 41, "g2": 43, "sigma": 0.05, "precision": "f32", "tol": 1e-6, "rhs": 1,
         "complex": False},
        # the 3-D bandwidth sweep with Monte-Carlo degrees of freedom: the
        # largest job
        {"name": "nw3d-1M-sweep", "kind": "sweep", "d": 3, "order": 0, "n": 1_000_000, "g0": 64,
         "g1": 64, "g2": 64, "n_bw": 8, "s_lo": 0.015, "s_hi": 0.1, "probes": 32,
         "precision": "f32"},
        # the differentiable GCV score: value and gradients to x, y, log h
        {"name": "ll2d-2M-gcv-grad", "kind": "gcv", "d": 2, "order": 1, "n": 2_000_000, "g0": 512,
         "g1": 512, "sigma": 0.012, "probes": 10, "precision": "f32"},
        # the differentiable grid estimate in its default precision: forward
        # and backward
        {"name": "ll2d-50k-grid-grad", "kind": "grad", "d": 2, "order": 1, "n": 50_021, "g0": 128,
         "g1": 112, "sigma": 0.03, "precision": "f64"},
        # a compact kernel: exact direct sums, with degrees of freedom and
        # variance
        {"name": "epan2d-200k-step", "kind": "step", "d": 2, "order": 1, "n": 200_000, "g0": 256,
         "g1": 256, "sigma": 0.02, "probes": 10, "precision": "f32", "kernel": "epanechnikov"},
        # uneven complex problems replayed as one captured graph
        {"name": "batch-14-uneven", "kind": "batch", "problems": 14, "shapes": 5, "n_lo": 1000,
         "n_hi": 1_000_000, "g_hi": 1024},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _sigma(rng, n, d, lo=0.01, hi=0.08):
    """A bandwidth with some 60 samples or more under the kernel at the mean density."""
    least = (60.0 / (n * (2 * math.pi) ** (d / 2))) ** (1.0 / d)
    return round(min(0.2, max(_log(rng, lo, hi), least)), 5)


def draw(rng):
    kind = rng.choice(["select", "smooth", "smooth", "smooth", "interval", "step", "step", "sweep",
                       "gcv", "grad", "batch"])
    f32 = rng.random() < 0.65
    if kind == "select":
        c = {"d": 1, "order": rng.choice([0, 1]), "n": int(_log(rng, 100, 20_000)),
             "g0": int(_log(rng, 50, 600)), "n_bw": rng.randint(4, 16), "s_lo": 0.04, "s_hi": 0.2,
             "probes": rng.randint(4, 12), "precision": "f32" if f32 else "f64"}
    elif kind == "smooth":
        d = rng.choice([1, 2, 2, 3])
        f32 = f32 or d == 3
        n = int(_log(rng, 2000, (1_000_000 if d < 3 else 300_000) if f32 else 200_000))
        order = rng.choice([0, 1, 1, 2]) if d < 3 else rng.choice([0, 1])
        tol = 1e-6 if f32 else rng.choice([1e-6, 1e-9, 1e-12])
        lo = 0.02 if order == 2 else 0.01 if d < 3 else 0.03
        c = {"d": d, "order": order, "n": n, "sigma": _sigma(rng, n, d, lo),
             "precision": "f32" if f32 else "f64", "tol": tol, "rhs": rng.choice([1, 1, 2, 3]),
             "complex": rng.random() < 0.25}
        hi = {1: 1024, 2: 400, 3: 56}[d]
        c.update({f"g{j}": int(_log(rng, 24 if d == 3 else 60, hi)) for j in range(d)})
    elif kind == "interval":
        n = int(_log(rng, 3000, 1_000_000))
        c = {"d": 2, "order": rng.choice([0, 1]), "n": n, "g0": int(_log(rng, 60, 300)),
             "g1": int(_log(rng, 60, 300)), "sigma": _sigma(rng, n, 2),
             "new": int(_log(rng, 1000, 200_000)), "precision": "f32"}
    elif kind == "step":
        kernel = rng.choice(["gaussian", "gaussian", "gaussian", "epanechnikov", "triweight"])
        n = int(_log(rng, 20_000, 1_000_000 if kernel == "gaussian" else 200_000))
        c = {"d": 2, "order": rng.choice([0, 1, 1]), "n": n, "g0": int(_log(rng, 80, 300)),
             "g1": int(_log(rng, 80, 300)),
             "sigma": _sigma(rng, n, 2, 0.01, 0.04 if kernel == "gaussian" else 0.02),
             "probes": rng.randint(2, 10), "precision": "f32", "kernel": kernel}
        if kernel != "gaussian":  # a support with neighbours enough in the sparse corners
            c["sigma"] = round(max(c["sigma"], math.sqrt(600.0 / (n * math.pi))), 5)
    elif kind == "sweep":
        n = int(_log(rng, 100_000, 1_000_000))
        c = {"d": 3, "order": 0, "n": n, "n_bw": rng.randint(2, 8), "s_lo": 0.03, "s_hi": 0.1,
             "probes": rng.randint(4, 32), "precision": "f32"}
        c.update({f"g{j}": rng.randint(32, 64) for j in range(3)})
    elif kind == "gcv":
        n = int(_log(rng, 4000, 2_000_000))
        c = {"d": 2, "order": rng.choice([0, 1, 1]), "n": n, "g0": int(_log(rng, 100, 512)),
             "g1": int(_log(rng, 100, 512)), "sigma": _sigma(rng, n, 2),
             "probes": rng.randint(2, 10), "precision": "f32"}
    elif kind == "grad":
        n = int(_log(rng, 3000, 50_000 if not f32 else 200_000))
        c = {"d": 2, "order": rng.choice([0, 1, 1]), "n": n, "g0": int(_log(rng, 60, 160)),
             "g1": int(_log(rng, 60, 160)), "sigma": _sigma(rng, n, 2, 0.02),
             "precision": "f32" if f32 else "f64"}
    else:
        c = {"problems": rng.randint(4, 14), "shapes": rng.randrange(1, 1000), "n_lo": 1000,
             "n_hi": int(_log(rng, 20_000, 500_000)), "g_hi": rng.randint(200, 700)}
    return {"kind": kind, **c}


# ---- inputs ------------------------------------------------------------------------

def _grid(case):
    return tuple(int(case[f"g{j}"]) for j in range(case["d"]))


def _dtype(case):
    return torch.float32 if case["precision"] == "f32" else torch.float64


def _sigmas(case):
    """Bandwidth per axis (axis 1 half as wide again, as in the headline configuration)."""
    return [case["sigma"] * (1.0, 1.5, 1.2)[j] for j in range(case["d"])]


def _log_sigma(case):
    return torch.tensor([math.log(v) for v in _sigmas(case)], dtype=_dtype(case))


def _diag(sig):
    return np.diag(np.square(np.asarray(sig, dtype=np.float64)))[None]


def _sweep_h(case):
    s = np.logspace(math.log10(case["s_lo"]), math.log10(case["s_hi"]), case["n_bw"])
    return np.stack([np.eye(case["d"]) * v * v for v in s])


def _samples(n, d, gen, clustered):
    """Locations in the unit box: uniform, or three clusters over a uniform floor."""
    u = torch.rand(n, d, generator=gen, device="cuda", dtype=torch.float64)
    if not clustered:
        return u
    means = torch.tensor([[0.3, 0.3], [0.7, 0.4], [0.5, 0.75]], device="cuda", dtype=torch.float64)
    comp = torch.randint(0, 3, (n,), generator=gen, device="cuda")
    c = means[comp] + 0.1 * torch.randn(n, d, generator=gen, device="cuda", dtype=torch.float64)
    floor = torch.rand(n, 1, generator=gen, device="cuda") < 0.25
    return torch.where(floor, u, c.clamp(0.0, 1.0))


def _responses(x, rhs, cplx, gen):
    """[rhs, n]: a smooth surface plus noise that grows along axis 0."""
    n, d = x.shape
    out = []
    for r in range(rhs):
        m = torch.sin((4 + r) * x[:, 0])
        if d > 1:
            m = m * torch.cos(3 * x[:, 1])
        if d > 2:
            m = m + torch.exp(-((x - 0.5) ** 2).sum(1) / 0.05)
        e = torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)
        m = m + (0.1 + 0.2 * x[:, 0]) * e
        if cplx:
            e = torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)
            m = torch.complex(m, torch.cos(3 * x[:, 0]) + 0.1 * e)
        out.append(m)
    return torch.stack(out)


def _data(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + case["n"])
    x = _samples(case["n"], case["d"], gen, case["kind"] == "step")
    x = x.to(_dtype(case))
    cplx = bool(case.get("complex", False))
    y = _responses(x.double(), case.get("rhs", 1), cplx, gen)
    if cplx:
        y = y.to(torch.complex64 if case["precision"] == "f32" else torch.complex128)
    else:
        y = y.to(_dtype(case))
    return x, y, gen


def _problems(case):
    """Shapes of the uneven batch: (d, n, grid, bandwidths) per problem."""
    g = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["problems"]):
        d = int(g.integers(1, 3))
        n = int(round(math.exp(g.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        gn = tuple(int(round(math.exp(g.uniform(math.log(128), math.log(case["g_hi"])))))
                   for _ in range(d))
        sig = [max(1.06 * 0.2887 * n ** (-1.0 / (d + 4)), 2.5 / (gn[j] - 1)) for j in range(d)]
        out.append((d, n, gn, sig))
    return out


def _batch_data(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + 17)
    xs, ys = [], []
    for d, n, _, _ in _problems(case):
        x = torch.rand(n, d, generator=gen, device="cuda", dtype=torch.float32)
        f = 0.4 + 18.8 * x[:, 0].double()
        ph = torch.sin(2 * math.pi * x[:, 0].double() + seed % 7)
        e = torch.randn(2, n, generator=gen, device="cuda", dtype=torch.float64)
        ys.append(torch.complex(torch.cos(ph) / (1 + f) + 0.05 * e[0],
                                torch.sin(ph) / (1 + f) + 0.05 * e[1]).to(torch.complex64))
        xs.append(x)
    return xs, ys


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        xs, ys = _batch_data(case, seed)
        b = fkreg.Batch([dict(d=d, order=1, grid_n=gn, lo=(0.0,) * d, hi=(1.0,) * d, H=_diag(sig),
                              tol=1e-6, precision="f32", y_complex=True, max_n=n)
                         for d, n, gn, sig in _problems(case)])
        outs = b.capture(xs, ys, variance=True)
        return {"case": case, "batch": b, "outs": outs}
    x, y, gen = _data(case, seed)
    d, grid = case["d"], _grid(case)
    box = ((0.0,) * d, (1.0,) * d)
    s = {"case": case, "x": x, "y": y, "grid": grid, "box": box}
    if kind == "smooth":
        s["plan"] = fkreg.Plan(d, case["order"], grid, *box, _diag(_sigmas(case)), max_n=case["n"],
                               n_rhs=case["rhs"], tol=case["tol"], precision=case["precision"],
                               y_complex=case["complex"])
    elif kind == "interval":
        s["plan"] = fkreg.Plan(d, case["order"], grid, *box, _diag(_sigmas(case)), max_n=case["n"],
                               precision=case["precision"])
        s["new"] = torch.rand(case["new"], d, generator=gen, device="cuda", dtype=x.dtype)
    elif kind == "step":
        s["plan"] = fkreg.Plan(d, case["order"], grid, *box, _diag(_sigmas(case)), max_n=case["n"],
                               max_probes=case["probes"], precision=case["precision"],
                               kernel=case["kernel"])
    elif kind == "sweep":
        s["plan"] = fkreg.Sweep(d, case["order"], grid, *box, _sweep_h(case), max_n=case["n"],
                                max_probes=case["probes"], precision=case["precision"])
    elif kind == "select":
        s["hlist"] = _sweep_h(case)
    else:  # the differentiable calls keep their plan themselves
        s["x"] = x.requires_grad_()
        s["y"] = y.requires_grad_()
        s["log_sigma"] = _log_sigma(case).requires_grad_()
        if kind == "grad":
            w = torch.rand(1, *grid, generator=gen, device="cuda", dtype=torch.float64)
            s["weight"] = (w - 0.3).to(x.dtype)
    return s


# ---- one pass ----------------------------------------------------------------------

def _scalars(out, dtype):
    """The scalar results in the plan's own precision: they are as accurate as its fields."""
    return {k: out[k].to(dtype) for k in ("gcv", "trace") if k in out}


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "batch":
        s["batch"].launch()
        return s["outs"]
    if kind == "select":
        r = fkreg.cv_fkreg(s["x"], s["y"], s["hlist"], list(s["grid"]), *s["box"],
                           order=c["order"], n_probes=c["probes"], seed=PROBE_SEED,
                           precision=c["precision"], variance=True)
        t = np.float32 if c["precision"] == "f32" else np.float64
        return {"index": r["index"], "gcv": r["gcv"].astype(t), "trace": r["trace"].astype(t),
                "mhat_grid": r["mhat_grid"], "mask": r["mask"], "mhat_at_x": r["mhat_at_x"],
                "sigma2": r["sigma2"]}
    if kind == "gcv":
        v = fkreg.gcv(s["x"], s["y"][0], s["log_sigma"], s["grid"], *s["box"], order=c["order"],
                      n_probes=c["probes"], seed=PROBE_SEED, precision=c["precision"])
        dx, dy, dl = torch.autograd.grad(v, (s["x"], s["y"], s["log_sigma"]))
        return {"gcv": v.detach(), "dx": dx, "dy": dy, "dlogh": dl}
    if kind == "grad":
        m = fkreg.smooth_grid(s["x"], s["y"], s["log_sigma"], s["grid"], *s["box"],
                              order=c["order"], precision=c["precision"])
        dx, dy, dl = torch.autograd.grad(m, (s["x"], s["y"], s["log_sigma"]), s["weight"])
        return {"mhat_grid": m.detach(), "dx": dx, "dy": dy, "dlogh": dl}
    p = s["plan"]
    p.set_points(s["x"])
    if kind == "smooth":
        return p.smooth(s["y"], want=("mhat_grid", "mask", "mhat_at_x"))
    if kind == "interval":
        o = p.smooth(s["y"], want=("mhat_grid", "mhat_at_x"))
        v = p.log_variance(s["y"], o["mhat_at_x"])
        lo, hi = fkreg.interval(o["mhat_grid"], v["sigma2"], 0.05)
        new = fkreg.predict(o["mhat_grid"], s["grid"], *s["box"], s["new"], "linear")
        return {"mhat_grid": o["mhat_grid"], "mhat_at_x": o["mhat_at_x"],
                "v_at_x": v["v_at_x"], "lower": lo, "upper": hi, "new": new}
    o = p.df(s["y"], c["probes"], seed=PROBE_SEED, want=("mhat_grid", "mask", "mhat_at_x"))
    r = {"mask": o["mask"], "mhat_at_x": o["mhat_at_x"], **_scalars(o, _dtype(c))}
    if kind == "sweep":  # one entry per bandwidth
        r["mhat_grid"] = list(o["mhat_grid"].unbind(0))
    else:
        r["mhat_grid"] = o["mhat_grid"]
        r["sigma2"] = p.variance(s["y"], o["mhat_at_x"])
    return r


# ---- what a pass cannot do without -------------------------------------------------

def _nmono(d, deg):
    return math.comb(d + deg, d)


def _work_plan(d, order, n, cells, nbw, strengths, tol, size, at_samples, cplx=False):
    """Inputs once, outputs once; two flops per window cell for every strength spread and
    every field gathered (nine digits need a window of ten cells per axis)."""
    w = math.ceil(math.log10(1 / tol) - 1e-9) + 1
    ns, nt = _nmono(d, 2 * order), _nmono(d, order)
    fields = nbw * (ns + strengths * nt) if at_samples else 0
    flops = 2.0 * n * w ** d * (1 + strengths + fields)
    parts = 2 if cplx else 1
    return {"bytes": float(size * (n * (d + parts) + nbw * (cells + n) * parts)), "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for d, n, gn, _ in _problems(case):
            w = _work_plan(d, 1, n, math.prod(gn), 1, 2, 1e-6, 4, True, True)
            v = _work_plan(d, 1, n, math.prod(gn), 1, 0, 1e-6, 4, False)
            b += w["bytes"] + 4 * math.prod(gn)
            f += w["flops"] + v["flops"]
        return {"bytes": b, "flops": f}
    d, n, order = case["d"], case["n"], case["order"]
    cells, size = math.prod(_grid(case)), 4 if case["precision"] == "f32" else 8
    probes, nbw = case.get("probes", 0), case.get("n_bw", 1)
    tol = case.get("tol", 1e-6 if case["precision"] == "f32" else 1e-12)
    if case.get("kernel", "gaussian") != "gaussian":
        sg = _sigmas(case)
        pairs = (n + cells) * n * math.pi * sg[0] * sg[1]
        ns, nt = _nmono(d, 2 * order), _nmono(d, order)
        return {"bytes": float(size * (n * (d + 2) + 2 * cells)),
                "flops": 2.0 * pairs * (ns + nt * (1 + probes * n / (n + cells)))}
    cplx = bool(case.get("complex", False))
    strengths = case.get("rhs", 1) * (2 if cplx else 1) + probes
    w = _work_plan(d, order, n, cells, nbw, strengths, tol, size, kind != "grad", cplx)
    if kind in ("step", "select", "interval"):  # the variance pass
        w["bytes"] += size * cells
        w["flops"] += _work_plan(d, order, n, cells, 1, 0, tol, size, False)["flops"]
    if kind == "interval":
        w["bytes"] += size * (2 * cells + n + case["new"] * (d + 1))
    if kind in ("gcv", "grad"):  # the adjoint pass: gradients to every input
        w["bytes"] += size * n * (d + 1)
        w["flops"] *= 2
    return w


# ---- the same in 64 bits by direct sums --------------------------------------------

def _monos(d, deg):
    return [e for e in itertools.product(range(deg + 1), repeat=d) if sum(e) <= deg]


def _profile(r2, kernel):
    """The regression kernel without its constant (which cancels everywhere here)."""
    if kernel == "gaussian":
        return torch.exp(-0.5 * r2)
    u = (1.0 - r2).clamp_min(0.0)
    return u if kernel == "epanechnikov" else u ** 3


def _pair_sums(x, c, q, sig, order, kernel="gaussian"):
    """Moment sums at points q: {monomial: [Q, 1 + R]}, column 0 the density, by direct sums."""
    n, d = x.shape
    deg = 2 * order
    es = _monos(d, deg)
    x, q = (x - 0.5) / sig, (q - 0.5) / sig
    cols = torch.cat([torch.ones(1, n, device=x.device, dtype=x.dtype), c])
    w = torch.stack([torch.stack([x[:, j] ** e[j] for j in range(d)]).prod(0) for e in es])
    w = (w[:, None] * cols[None]).reshape(-1, n).T.contiguous()
    raw = []
    for part in q.split(max(1, (1 << 28) // n)):
        r2 = sum((part[:, None, j] - x[None, :, j]) ** 2 for j in range(d))
        raw.append((_profile(r2, kernel) @ w).reshape(len(part), len(es), -1))
    raw = torch.cat(raw)
    at = {e: raw[:, k] for k, e in enumerate(es)}
    out = {}
    for e in es:  # (x - q)^e by the binomial rule, axis by axis
        acc = 0
        for b in itertools.product(*[range(v + 1) for v in e]):
            f = math.prod(math.comb(e[j], b[j]) for j in range(d))
            sh = torch.stack([(-q[:, j]) ** (e[j] - b[j]) for j in range(d)]).prod(0)
            acc = acc + f * sh[:, None] * at[b]
        out[e] = acc
    return out


def _grid_sums(x, c, axes, sig, order):
    """The same at every grid point for the Gaussian, which is a product over the axes."""
    n, d = x.shape
    cols = torch.cat([torch.ones(1, n, device=x.device, dtype=x.dtype), c])
    es = _monos(d, 2 * order)
    out = dict.fromkeys(es, 0)
    for i in range(0, n, 250_000):
        f = []
        for j in range(d):
            z = (x[None, i:i + 250_000, j] - axes[j][:, None]) / sig[j]
            k = torch.exp(-0.5 * z * z)
            f.append([k * z ** p for p in range(2 * order + 1)])
        cc = cols[:, i:i + 250_000]
        for e in es:
            rows = cc if sum(e) <= order else cc[:1]
            if d == 1:
                v = rows @ f[0][e[0]].T
            else:
                last = f[1][e[1]]
                if d == 3:
                    last = (last[:, None] * f[2][e[2]][None]).reshape(-1, last.shape[1])
                v = torch.stack([(f[0][e[0]] * r) @ last.T for r in rows]).reshape(len(rows), -1)
            out[e] = out[e] + v
    return {e: v.T for e, v in out.items()}


def _fit(sums, d, order):
    """(estimates [R, Q], [S^-1]_11 [Q], the weights S^-1 e_1 [Q, p])."""
    un = _monos(d, order)
    add = lambda a, b: tuple(i + j for i, j in zip(a, b))  # noqa: E731
    m = torch.stack([torch.stack([sums[add(a, b)][:, 0] for b in un], -1) for a in un], -2)
    e1 = torch.zeros(m.shape[:-1], device=m.device, dtype=m.dtype)
    e1[:, un.index((0,) * d)] = 1.0
    a = torch.linalg.solve(m, e1)
    t = torch.stack([sums[e][:, 1:] for e in un], 1)
    return torch.einsum("qp,qpr->rq", a, t), a[:, un.index((0,) * d)], a


def _probes(n, count, single):
    """The documented probe generator: SplitMix64 words in Box-Muller pairs."""
    gamma = 0x9E3779B97F4A7C15
    wrap = lambda v: v - (1 << 64) if v >= 1 << 63 else v  # noqa: E731
    shr = lambda z, k: (z >> k) & ((1 << (64 - k)) - 1)  # noqa: E731

    def word(z):
        z = z + wrap(gamma)
        z = (z ^ shr(z, 30)) * wrap(0xBF58476D1CE4E5B9)
        z = (z ^ shr(z, 27)) * wrap(0x94D049BB133111EB)
        return z ^ shr(z, 31)

    i = torch.arange(n, device="cuda", dtype=torch.int64)
    bits = 24 if single else 53
    out = []
    for j in range((count + 1) // 2):
        base = ((i | (j << 40)) * 2) * wrap(gamma) + PROBE_SEED
        u1 = (shr(word(base), 64 - bits).double() + 1.0) * 2.0 ** -bits
        u2 = shr(word(base + wrap(gamma)), 64 - bits).double() * 2.0 ** -bits
        r = torch.sqrt(-2.0 * torch.log(u1))
        out += [r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)]
    return torch.stack(out[:count])


def _gcv(y, m, z, mz, a0):
    """(GCV, [Girard, Hutchinson, exact trace]) of one bandwidth."""
    n = y.shape[-1]
    g = n * ((z * mz).sum(1) / (z * z).sum(1)).mean()
    tr = torch.stack([g, (z * mz).sum(1).mean(), a0.sum()])
    return ((y - m) ** 2).mean() / (1 - g / n) ** 2, tr


def _afford(n, points, cols):
    return n * points * (60.0 + 2.0 * cols) < 6e12


def _axes(grid):
    return [torch.linspace(0, 1, g, device="cuda", dtype=torch.float64) for g in grid]


def _grid_any(x, c, grid, sig, order, kernel):
    if kernel == "gaussian":
        return _grid_sums(x, c, _axes(grid), sig, order)
    q = torch.cartesian_prod(*_axes(grid)).reshape(-1, len(grid))
    return _pair_sums(x, c, q, torch.as_tensor(sig, device="cuda", dtype=x.dtype), order, kernel)


def _ri(y):
    """Real rows of the responses: (re, im) pairs for complex ones."""
    if not y.is_complex():
        return y.double()
    y = y.to(torch.complex128)
    return torch.stack([y.real, y.imag], 1).reshape(-1, y.shape[-1])


def _back(m, y, *shape):
    return torch.complex(m[0::2], m[1::2]).reshape(shape) if y.is_complex() else m.reshape(shape)


def _exact_smooth(case, x, y):
    d, order, grid = case["d"], case["order"], _grid(case)
    c, sig = _ri(y), _sigmas(case)
    n, rhs = case["n"], y.shape[0]
    out = {"mask": None, "mhat_at_x": None}
    m = _fit(_grid_any(x, c, grid, sig, order, "gaussian"), d, order)[0]
    out["mhat_grid"] = _back(m, y, 1, rhs, *grid)
    if _afford(n, n, _nmono(d, 2 * order) * (1 + len(c))):
        st = torch.as_tensor(sig, device="cuda", dtype=torch.float64)
        m = _fit(_pair_sums(x, c, x, st, order), d, order)[0]
        out["mhat_at_x"] = _back(m, y, 1, rhs, n)
    return out


def _exact_df(case, x, y, sigs, kernel):
    """df and variance for each of the bandwidths `sigs`: a list of dicts."""
    d, order, grid, n = case["d"], case["order"], _grid(case), case["n"]
    z = _probes(n, case["probes"], case["precision"] == "f32")
    res = []
    for sig in sigs:
        gs = _grid_any(x, y, grid, sig, order, kernel)
        mg, _, ag = _fit(gs, d, order)
        r = {"mhat_grid": mg.reshape(1, *grid), "at": None, "gcv": None, "trace": None,
             "sigma2": None}
        if _afford(n, n, _nmono(d, 2 * order) * (2 + len(z))):
            st = torch.as_tensor(sig, device="cuda", dtype=torch.float64)
            m, a0, _ = _fit(_pair_sums(x, torch.cat([y, z]), x, st, order, kernel), d, order)
            r["at"] = m[:1]
            r["gcv"], r["trace"] = _gcv(y[0], m[0], z, m[1:], a0)
            v = _grid_any(x, (y - m[:1]) ** 2, grid, sig, order, kernel)
            t = torch.stack([v[e][:, 1] for e in _monos(d, order)], 1)
            r["sigma2"] = (ag * t).sum(1).reshape(1, *grid)
        res.append(r)
    return res


def _exact_interval(case, seed, x, y):
    d, order, grid, n = case["d"], case["order"], _grid(case), case["n"]
    sig = _sigmas(case)
    out = _exact_smooth({**case, "rhs": 1}, x, y)
    out.pop("mask")
    mg = out["mhat_grid"]
    gen = _data(case, seed)[2]
    q = torch.rand(case["new"], d, generator=gen, device="cuda", dtype=_dtype(case)).double()
    at, wt = [], []
    for j in range(d):
        u = q[:, j] * (grid[j] - 1)
        k = u.floor().clamp(0, grid[j] - 2)
        at.append(k.long())
        wt.append(u - k)
    v = 0
    for b in itertools.product((0, 1), repeat=d):
        w = torch.stack([wt[j] if b[j] else 1 - wt[j] for j in range(d)]).prod(0)
        v = v + w * mg[0, 0][tuple(at[j] + b[j] for j in range(d))]
    out["new"] = v.reshape(1, 1, -1)
    out["v_at_x"] = out["lower"] = out["upper"] = None
    if out["mhat_at_x"] is not None:
        r = (y - out["mhat_at_x"][0]) ** 2
        lr = torch.log(r + 1.0 / n)
        st = torch.as_tensor(sig, device="cuda", dtype=torch.float64)
        va = _fit(_pair_sums(x, lr, x, st, order), d, order)[0]
        vg = _fit(_grid_sums(x, lr, _axes(grid), sig, order), d, order)[0]
        s2 = torch.exp(vg) * (r * torch.exp(-va)).mean()
        h = statistics.NormalDist().inv_cdf(0.975) * torch.sqrt(s2).reshape(mg.shape)
        out.update({"v_at_x": va.reshape(1, 1, n), "lower": mg - h, "upper": mg + h})
    return out


def _exact_grad(case, x, y, weight):
    d, order, grid = case["d"], case["order"], _grid(case)
    x, y = x.requires_grad_(), y.requires_grad_()
    ls = _log_sigma(case).double().cuda().requires_grad_()
    m = _fit(_grid_sums(x, y, _axes(grid), torch.exp(ls), order), d, order)[0].reshape(1, *grid)
    dx, dy, dl = torch.autograd.grad(m, (x, y, ls), weight)
    return {"mhat_grid": m.detach(), "dx": dx, "dy": dy, "dlogh": dl}


def _exact_gcv(case, x, y):
    d, order, n = case["d"], case["order"], case["n"]
    z = _probes(n, case["probes"], True)
    x, y = x.requires_grad_(), y.requires_grad_()
    ls = _log_sigma(case).double().cuda().requires_grad_()
    m, a0, _ = _fit(_pair_sums(x, torch.cat([y, z]), x, torch.exp(ls), order), d, order)
    v = _gcv(y[0], m[0], z, m[1:], a0)[0]
    dx, dy, dl = torch.autograd.grad(v, (x, y, ls))
    return {"gcv": v.detach(), "dx": dx, "dy": dy, "dlogh": dl}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        xs, ys = _batch_data(case, seed)
        out = []
        for x, y, (d, n, gn, sig) in zip(xs, ys, _problems(case)):
            c = _ri(y[None])
            m, _, ag = _fit(_grid_sums(x.double(), c, _axes(gn), sig, 1), d, 1)
            r = {"mask": None, "mhat_at_x": None, "sigma2": None,
                 "mhat_grid": _back(m, y, 1, 1, *gn)}
            if _afford(n, 8 * n, 9):
                st = torch.as_tensor(sig, device="cuda", dtype=torch.float64)
                ma = _fit(_pair_sums(x.double(), c, x.double(), st, 1), d, 1)[0]
                r["mhat_at_x"] = _back(ma, y, 1, 1, n)
                v = _grid_sums(x.double(), ((c - ma) ** 2).sum(0, keepdim=True), _axes(gn), sig, 1)
                t = torch.stack([v[e][:, 1] for e in _monos(d, 1)], 1)
                r["sigma2"] = (ag * t).sum(1).reshape(1, 1, *gn)
            out.append(r)
        return out
    x, y, gen = _data(case, seed)
    x = x.double()
    if kind == "smooth":
        return _exact_smooth(case, x, y)
    y = y.double()
    if kind == "interval":
        return _exact_interval(case, seed, x, y)
    if kind == "grad":
        w = torch.rand(1, *_grid(case), generator=gen, device="cuda", dtype=torch.float64)
        return _exact_grad(case, x, y, (w - 0.3).to(_dtype(case)).double())
    if kind == "gcv":
        return _exact_gcv(case, x, y) if case["n"] <= 6000 else None
    if kind == "step":
        r = _exact_df(case, x, y, [_sigmas(case)], case["kernel"])[0]
        return {"mask": None, "mhat_grid": r["mhat_grid"][None],
                "mhat_at_x": None if r["at"] is None else r["at"][None],
                "gcv": None if r["gcv"] is None else r["gcv"].reshape(1, 1),
                "trace": None if r["trace"] is None else r["trace"].reshape(1, 3),
                "sigma2": None if r["sigma2"] is None else r["sigma2"][None]}
    sigs = [[math.sqrt(v) for v in np.diag(h)] for h in _sweep_h(case)]
    if kind == "select":
        rs = _exact_df(case, x, y, sigs, "gaussian")
        if rs[0]["gcv"] is None:
            return None
        gcv = torch.stack([r["gcv"] for r in rs])
        k = int(torch.nonzero(gcv <= gcv.min()).max())
        return {"index": None, "gcv": gcv, "trace": torch.stack([r["trace"] for r in rs]),
                "mhat_grid": rs[k]["mhat_grid"], "mask": None, "mhat_at_x": rs[k]["at"],
                "sigma2": rs[k]["sigma2"]}
    # the sweep: the grid estimates of its narrowest and widest bandwidth
    pick = [0, len(sigs) - 1]
    grids = [None] * len(sigs)
    for b in pick:
        s = _grid_sums(x, y, _axes(_grid(case)), sigs[b], 0)
        grids[b] = _fit(s, case["d"], 0)[0].reshape(1, *_grid(case))
    return {"mask": None, "mhat_at_x": None, "gcv": None, "trace": None, "mhat_grid": grids}
