"""3-D spreading of FP32 plans (lanes over the window cells): tile sizes that
give padded rows of each kind, fine grids that take the vector flush and ones
that don't (the last axis or the tiles not multiples of four cells), and
sub-problems from one sample to several per bin, against the oracle.

Bars as in test_gpu_parity (FP32 1e-5 of the oracle's direct sums).
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


# n, tile (0: the planner's 16), grid, sigma, responses; nf is 84, 70, 84, 60, 70, 54, 84
CASES = [(1, 0, 9, 0.08, 1), (3001, 0, 9, 0.1, 2), (20_011, 8, 9, 0.08, 1),
         (9000, 20, 12, 0.12, 3), (9000, 6, 9, 0.1, 1), (40_003, 24, 9, 0.2, 2),
         (5000, 5, 9, 0.08, 1)]


@pytest.mark.parametrize("n,tile,grid,sigma,rhs", CASES)
def test_grid_estimate(n, tile, grid, sigma, rhs):
    from paper_2204_07716_gb300.fkreg import Plan
    w = inputs.random_small(1200 + tile, 3, n, grid, 0, [sigma], precision="f32", tol=1e-6,
                            n_rhs=rhs)
    w.x[::5] = w.x[0]      # runs of samples that share a window
    p = Plan(3, 0, w.grid_n, w.lo, w.hi, w.H, max_n=n, n_rhs=rhs, tol=1e-6, precision="f32",
             tile=tile)
    p.set_points(torch.tensor(w.x, dtype=torch.float32))
    out = p.smooth(torch.tensor(w.y, dtype=torch.float32), want=("mhat_grid", "mask"))
    p.sync()
    x, y = (v.astype(np.float32).astype(np.float64) for v in (w.x, w.y))
    q = oracle.grid_points(w.grid_n, w.lo, w.hi)
    r = oracle.smooth_at(x, y, w.H[0], 0, q)
    a = oracle.scale_field(x, y, w.H[0], q)
    ok = out["mask"][0].reshape(-1).cpu().numpy().astype(bool)
    for k in range(rhs):
        m = out["mhat_grid"][0, k].reshape(-1).cpu().numpy()
        assert mhat_error(m, r["mhat"][:, k], r["s"][:, 0], a[:, k], ok) < 1e-5
