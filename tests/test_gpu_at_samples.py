"""The at-sample pass at the sizes where its lane-per-sample gathers can go
wrong: every instantiated window width in both precisions, 1-D plans of one
bin and of many (tile set), 2-D windows staged in shared memory and read from
the grid, 3-D local linear, orders 0 to 2, group remainders (n around
multiples of 32 and of a block) and more fields than one pass holds.

Bars as in test_gpu_parity: FP64 at tol 1e-12 within 1e-10 of the oracle, at
1e-9 within 1e-8, at 1e-6 within 1e-5, FP32 at tol 1e-6 within 1e-5.
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


# d, order, precision, tol, n, probes, tile
CASES = [
    (1, 0, "f64", 1e-9, 1, 0, 0),
    (1, 1, "f64", 1e-12, 33, 2, 0),
    (1, 2, "f64", 1e-6, 1025, 3, 0),
    (1, 1, "f64", 1e-12, 2049, 20, 64),     # more fields than one FP64 pass
    (1, 1, "f32", 1e-6, 257, 4, 0),
    (1, 2, "f32", 1e-6, 1500, 25, 0),       # more fields than one FP32 pass
    (2, 0, "f64", 1e-6, 1023, 1, 0),
    (2, 1, "f64", 1e-9, 2000, 2, 0),
    (2, 1, "f64", 1e-12, 4001, 3, 0),
    (2, 1, "f64", 1e-12, 1500, 18, 0),      # window too large to stage
    (2, 2, "f64", 1e-12, 3000, 1, 0),
    (2, 2, "f32", 1e-6, 3001, 2, 0),
    (2, 2, "f32", 1e-6, 2500, 9, 0),        # several passes, staged
    (3, 1, "f32", 1e-6, 3000, 2, 0),
    (3, 1, "f64", 1e-6, 2500, 1, 0),
]


@pytest.mark.parametrize("d,order,prec,tol,n,probes,tile", CASES)
def test_values_traces_at_samples(d, order, prec, tol, n, probes, tile):
    from paper_2204_07716_gb300.fkreg import Plan
    bar = {1e-12: 1e-10, 1e-9: 1e-8, 1e-6: 1e-5}[tol]
    sig = {1: 0.05, 2: 0.12, 3: 0.2}[d]
    w = inputs.random_small(700 + 10 * d + order, d, n, 20, order, [sig], precision=prec, tol=tol)
    dt = torch.float32 if prec == "f32" else torch.float64
    p = Plan(d, order, w.grid_n, w.lo, w.hi, w.H, max_n=n, max_probes=max(probes, 1), tol=tol,
             precision=prec, tile=tile)
    p.set_points(torch.tensor(w.x, dtype=dt))
    x = w.x.astype(np.float32).astype(np.float64) if prec == "f32" else w.x
    y = w.y.astype(np.float32).astype(np.float64) if prec == "f32" else w.y
    z = np.zeros((0, n))
    if probes:
        z = oracle.probes(11, probes, n).astype(np.float32).astype(np.float64)
        out = p.df(torch.tensor(y, dtype=dt), probes, probes=torch.tensor(z, dtype=dt),
                   want=("mhat_at_x",))
    else:
        out = p.smooth(torch.tensor(y, dtype=dt), want=("mhat_at_x",))
    p.sync()
    if order > 0 and n < 30:
        return
    c = np.concatenate([y, z])
    r = oracle.smooth_at(x, c, w.H[0], order, x)
    ay = oracle.scale_field(x, c, w.H[0], x)
    mh = out["mhat_at_x"][0, 0].cpu().numpy()
    assert mhat_error(mh, r["mhat"][:, 0], r["s"][:, 0], ay[:, 0]) < bar
    if probes:
        hutch = float(np.mean(np.sum(z * r["mhat"][:, 1:].T, axis=1)))
        scale = float(np.mean(np.sum(np.abs(z * r["mhat"][:, 1:].T), axis=1)))
        assert abs(out["trace"][0, 1].item() - hutch) < 20 * bar * scale
        assert out["trace"][0, 2].item() == pytest.approx(oracle.trace_exact(x, w.H[0], order),
                                                          rel=20 * bar)
