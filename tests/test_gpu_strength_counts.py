"""Grid estimate and values at the samples for strength counts around every
launch size of the spreading (counts are responses plus the density) and field
counts around the units of a cell record, against the oracle.

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


CASES = [(2, "f32", r) for r in (2, 3, 4, 7, 8, 11, 12, 15, 16, 24, 38)]
CASES += [(1, "f32", r) for r in (2, 8, 13, 20)] + [(2, "f64", r) for r in (2, 4, 6)]
CASES += [(3, "f32", 4)]


@pytest.mark.parametrize("d,prec,rhs", CASES)
def test_every_response(d, prec, rhs):
    from paper_2204_07716_gb300.fkreg import Plan
    tol = 1e-6 if prec == "f32" else 1e-12
    n, grid, sigma = 3001, {1: 45, 2: 19, 3: 8}[d], {1: 0.05, 2: 0.1, 3: 0.25}[d]
    w = inputs.random_small(1300 + 50 * d + rhs, d, n, grid, 0, [sigma], precision=prec, tol=tol,
                            n_rhs=rhs)
    ft = np.float32 if prec == "f32" else np.float64
    dt = torch.float32 if prec == "f32" else torch.float64
    p = Plan(d, 0, w.grid_n, w.lo, w.hi, w.H, max_n=n, n_rhs=rhs, tol=tol, precision=prec)
    p.set_points(torch.tensor(w.x, dtype=dt))
    out = p.smooth(torch.tensor(w.y, dtype=dt), want=("mhat_grid", "mask", "mhat_at_x"))
    p.sync()
    x, y = (v.astype(ft).astype(np.float64) for v in (w.x, w.y))
    bar = 1e-5 if prec == "f32" else 1e-10
    for q, got, ok in ((oracle.grid_points(w.grid_n, w.lo, w.hi), out["mhat_grid"], out["mask"]),
                       (x[::7], out["mhat_at_x"][:, :, ::7], None)):
        r = oracle.smooth_at(x, y, w.H[0], 0, q)
        a = oracle.scale_field(x, y, w.H[0], q)
        valid = None if ok is None else ok[0].reshape(-1).cpu().numpy().astype(bool)
        for k in range(rhs):
            m = got[0, k].reshape(-1).cpu().numpy()
            assert mhat_error(m, r["mhat"][:, k], r["s"][:, 0], a[:, k], valid) < bar
