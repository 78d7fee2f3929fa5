"""Direct sums at the edges of their groups, runs and strength chunks: n around
multiples of the 32 targets of a group, strength counts around multiples of
four and at the instantiated chunk sizes, every kernel, a correlated H; and a
response that is not finite stays inside the supports that hold its sample.

Bars as in test_gpu_parity (FP64 1e-10, FP32 1e-5 of the oracle's direct sums).
"""
import numpy as np
import pytest

import oracle
from paper_2204_07716_gb300 import inputs
from parity_util import mhat_error

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2204_07716_gb300 import build
    build.build()
    oracle.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def plan(w, n_rhs, kernel, **kw):
    from paper_2204_07716_gb300.fkreg import Plan
    return Plan(w.d, w.order, w.grid_n, w.lo, w.hi, w.H, max_n=w.n, n_rhs=n_rhs, tol=w.tol,
                precision=w.precision, kernel=kernel, **kw)


# d, order, precision, n, responses, kernel, full H
CASES = [
    (1, 0, "f32", 31, 1, "uniform", False),
    (1, 1, "f32", 1025, 5, "triangle", False),
    (1, 2, "f64", 600, 13, "biweight", False),
    (2, 0, "f32", 2049, 33, "triweight", True),
    (2, 0, "f64", 1000, 40, "epanechnikov", False),
    (2, 1, "f32", 3000, 4, "epanechnikov", True),
    (2, 1, "f32", 2500, 12, "triweight", False),
    (2, 1, "f32", 2500, 13, "biweight", False),
    (2, 2, "f32", 4000, 5, "epanechnikov", False),
    (3, 0, "f32", 3001, 36, "gaussian_direct", False),
    (3, 0, "f32", 2000, 60, "epanechnikov", True),
    (3, 1, "f32", 4000, 9, "biweight", False),
    (3, 1, "f64", 2500, 2, "gaussian_direct", True),
]


@pytest.mark.parametrize("d,order,prec,n,rhs,kernel,full_h", CASES)
def test_sums_at_chunk_edges(d, order, prec, n, rhs, kernel, full_h):
    sig = {1: 0.08, 2: 0.15, 3: 0.3}[d] * (0.2 if kernel == "gaussian_direct" else 1.0)
    grid = {1: 70, 2: 21, 3: 11}[d]
    w = inputs.random_small(900 + 10 * d + order, d, n, grid, order, [sig], precision=prec,
                            tol=1e-12 if prec == "f64" else 1e-6, n_rhs=rhs, full_h=full_h)
    dt = torch.float32 if prec == "f32" else torch.float64
    p = plan(w, rhs, kernel)
    p.set_points(torch.tensor(w.x, dtype=dt))
    out = p.smooth(torch.tensor(w.y, dtype=dt), want=("mhat_grid", "mask", "mhat_at_x"))
    p.sync()
    ft = np.float32 if prec == "f32" else np.float64
    x, y = w.x.astype(ft).astype(np.float64), w.y.astype(ft).astype(np.float64)
    H, bar = w.H[0], 1e-10 if prec == "f64" else 1e-5
    for q, got, ok in ((oracle.grid_points(w.grid_n, w.lo, w.hi), out["mhat_grid"], out["mask"]),
                       (x, out["mhat_at_x"], None)):
        if kernel == "gaussian_direct":
            r = oracle.smooth_at(x, y, H, order, q)
            a = np.abs(oracle.moment_sums(x, np.abs(y), H, 0, q)[:, :, 0])
        else:
            r = oracle.smooth_at_compact(x, y, H, order, q, kernel)
            a = np.abs(oracle.moment_sums_compact(x, np.abs(y), H, 0, q, kernel)[:, :, 0])
        a = a if a.shape[0] == q.shape[0] else a.T
        valid = None if ok is None else ok[0].reshape(-1).cpu().numpy().astype(bool)
        for k in (0, rhs // 2, rhs - 1):
            m = got[0, k].reshape(-1).cpu().numpy()
            assert mhat_error(m, r["mhat"][:, k], r["s"][:, 0], a[:, k], valid) < bar


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_values_that_are_not_finite_stay_in_their_supports(prec):
    w = inputs.random_small(951, 2, 3000, 24, 1, [0.1], precision=prec,
                            tol=1e-12 if prec == "f64" else 1e-6, n_rhs=2)
    dt = torch.float32 if prec == "f32" else torch.float64
    p = plan(w, 2, "epanechnikov")
    x = torch.tensor(w.x, dtype=dt)
    p.set_points(x)
    y = torch.tensor(w.y, dtype=dt)
    ref = p.smooth(y, want=("mhat_at_x",))["mhat_at_x"][0].clone()
    y[0, 7], y[1, 90] = float("nan"), float("inf")
    got = p.smooth(y, want=("mhat_at_x",))["mhat_at_x"][0]
    p.sync()
    xd = x.double().cpu()
    for r, i in ((0, 7), (1, 90)):
        dist = torch.sqrt(((xd - xd[i]) ** 2).sum(1)) / 0.1
        far, near = dist > 1.001, dist < 0.999
        assert torch.allclose(got[r].cpu()[far], ref[r].cpu()[far], rtol=1e-5, atol=1e-5)
        assert not torch.isfinite(got[r].cpu()[near]).any()
    # a later pass with finite values is clean again
    y = torch.tensor(w.y, dtype=dt)
    again = p.smooth(y, want=("mhat_at_x",))["mhat_at_x"][0]
    p.sync()
    assert torch.isfinite(again).all()
