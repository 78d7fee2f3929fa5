"""FP64 direct sums: every instantiated number of strength chunks and its neighbours, at the
samples and on the grid, with groups of 32 samples that span rows of bins (most of their
candidates lie in no lane's support), against the oracle's sums.

Bar as in test_gpu_direct_sums (1e-10).
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


@pytest.mark.parametrize("d,order,rhs,kernel,full_h", [
    (1, 0, 5, "epanechnikov", False), (1, 0, 13, "triangle", False), (1, 1, 9, "biweight", False),
    (2, 0, 4, "uniform", False), (2, 0, 12, "epanechnikov", True), (2, 0, 36, "triweight", False),
    (2, 0, 37, "epanechnikov", False), (2, 1, 5, "epanechnikov", False), (2, 2, 3, "biweight", True),
    (3, 0, 5, "triweight", False), (3, 0, 13, "epanechnikov", False), (3, 1, 3, "triangle", False)])
def test_strength_chunks(d, order, rhs, kernel, full_h):
    from paper_2204_07716_gb300.fkreg import Plan
    n, grid = {1: 1000, 2: 1500, 3: 2500}[d], {1: 200, 2: 40, 3: 12}[d]
    w = inputs.random_small(1400 + 10 * d + order, d, n, grid, order, [{1: 0.05, 2: 0.15, 3: 0.3}[d]],
                            n_rhs=rhs, full_h=full_h)
    p = Plan(d, order, w.grid_n, w.lo, w.hi, w.H, max_n=n, n_rhs=rhs, precision="f64", kernel=kernel)
    p.set_points(torch.tensor(w.x))
    out = p.smooth(torch.tensor(w.y), want=("mhat_grid", "mask", "mhat_at_x"))
    p.sync()
    H = w.H[0]
    for q, got, ok in ((oracle.grid_points(w.grid_n, w.lo, w.hi), out["mhat_grid"], out["mask"]),
                       (w.x, out["mhat_at_x"], None)):
        r = oracle.smooth_at_compact(w.x, w.y, H, order, q, kernel)
        a = oracle.moment_sums_compact(w.x, np.abs(w.y), H, 0, q, kernel)[:, :, 0]
        valid = None if ok is None else ok[0].reshape(-1).cpu().numpy().astype(bool)
        for k in (0, rhs // 2, rhs - 1):
            m = got[0, k].reshape(-1).cpu().numpy()
            assert mhat_error(m, r["mhat"][:, k], r["s"][:, 0], a[:, k], valid) < 1e-10
