"""1-D plans whose transforms the library computes itself: grid estimate and
values at the samples against the oracle for transform lengths with every
radix, odd lattice lengths, and lengths on both sides of the 4096-point limit
(above it the transforms are cuFFT's).
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


# grid points, sigma, precision, tol: nf from 28 to beyond 4096, L odd and even
CASES = [(2, 0.4, "f64", 1e-12), (17, 0.3, "f32", 1e-6), (47, 0.1, "f64", 1e-9),
         (100, 0.05, "f64", 1e-12), (121, 0.05, "f32", 1e-6), (333, 0.02, "f64", 1e-12),
         (1000, 0.004, "f32", 1e-6), (2000, 0.0035, "f64", 1e-9), (5000, 0.002, "f32", 1e-6)]


@pytest.mark.parametrize("grid,sigma,prec,tol", CASES)
def test_transform_lengths(grid, sigma, prec, tol):
    from paper_2204_07716_gb300.fkreg import Plan
    n = 6000
    w = inputs.random_small(1000 + grid, 1, n, grid, 1, [sigma], precision=prec, tol=tol, n_rhs=2)
    dt = torch.float32 if prec == "f32" else torch.float64
    p = Plan(1, 1, w.grid_n, w.lo, w.hi, w.H, max_n=n, n_rhs=2, tol=tol, precision=prec)
    p.set_points(torch.tensor(w.x, dtype=dt))
    out = p.smooth(torch.tensor(w.y, dtype=dt), want=("mhat_grid", "mask", "mhat_at_x"))
    p.sync()
    ft = np.float32 if prec == "f32" else np.float64
    x, y = w.x.astype(ft).astype(np.float64), w.y.astype(ft).astype(np.float64)
    bar = {1e-12: 1e-10, 1e-9: 1e-8, 1e-6: 1e-5}[tol]
    gp = oracle.grid_points(w.grid_n, w.lo, w.hi)
    for q, got, ok in ((gp, out["mhat_grid"], out["mask"]), (x, out["mhat_at_x"], None)):
        r = oracle.smooth_at(x, y, w.H[0], 1, q)
        a = oracle.scale_field(x, y, w.H[0], q)
        valid = None if ok is None else ok[0].reshape(-1).cpu().numpy().astype(bool)
        for k in range(2):
            m = got[0, k].reshape(-1).cpu().numpy()
            assert mhat_error(m, r["mhat"][:, k], r["s"][:, 0], a[:, k], valid) < bar
