"""Lengths of the lattice transforms: those that go to cuFFT are even on the last axis.

cuFFT packs two rows of a batch of odd real length into one complex transform, and the
fields of a batch (1, z, z^2, ...) differ in scale by the units of the box: an odd length
puts the rounding of the large fields onto the small ones.  The GPU cases would have had
odd lengths; the estimates meet the same bars as everywhere (FP32 1e-5, FP64 1e-10).
"""
import numpy as np
import pytest

import oracle
from paper_2204_07716_gb300 import fkreg, inputs
from parity_util import mhat_error


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2204_07716_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("d", [1, 2, 3])
def test_last_axis_is_even_where_cufft_transforms_it(d):
    rng = np.random.default_rng(d)
    hi, odd = {1: 40_000, 2: 3000, 3: 200}[d], 0
    for _ in range(200):
        grid = [int(np.exp(rng.uniform(np.log(8), np.log(hi)))) for _ in range(d)]
        sig = [max(0.02, 3.0 / g) if d > 1 else 12.0 / g for g in grid]
        g = fkreg.geometry(d=d, order=1, grid_n=grid, lo=(0.0,) * d, hi=(1.0,) * d,
                           H=np.diag(np.square(sig)), tol=1e-6, precision="f32")
        last = g["ldft"][d - 1]
        odd += any(v % 2 for v in g["ldft"])
        assert last % 2 == 0 or (d == 1 and last <= 4096), (grid, g["ldft"])
        for j, v in enumerate(g["ldft"]):  # still the next 7-smooth length that holds the tail
            assert (v - grid[j] + 1) / (grid[j] - 1) >= 5.2 * sig[j]
    assert odd > 0  # other axes, and short 1-D lengths, stay as they are


# box edge, grid, bandwidth / box edge per axis, order, precision, tol, scale of the second response
CASES = [(1.0, (10_000,), (0.0015,), 1, "f32", 1e-6, 1.0),    # 10125 points
         (1.0, (5000,), (0.002,), 1, "f64", 1e-12, 1.0),      # 5103 points
         (1.0, (4990,), (0.002,), 2, "f64", 1e-9, 1.0),       # 5103 points
         (1e-3, (24, 80), (0.1, 0.05), 1, "f32", 1e-6, 1.0),  # last axis 105
         (1e-3, (17, 1000), (0.2, 0.004), 1, "f32", 1e-6, 1.0),   # last axis 1029
         (1.0, (24, 80), (0.1, 0.05), 0, "f32", 1e-6, 1e-6),  # a response a million times smaller
         (1e-3, (10, 10, 80), (0.2, 0.2, 0.05), 1, "f32", 1e-6, 1.0)]


@pytest.mark.gpu
@pytest.mark.parametrize("edge,grid,sig,order,prec,tol,scale", CASES)
def test_fields_of_unlike_scale(edge, grid, sig, order, prec, tol, scale):
    torch = pytest.importorskip("torch")
    d, n = len(grid), 6000
    ft = np.float32 if prec == "f32" else np.float64
    w = inputs.random_small(1200 + grid[-1], d, n, grid, order, [0.1], n_rhs=2)
    x = (edge * w.x).astype(ft)
    y = (w.y * np.array([[1.0], [scale]])).astype(ft)
    H = np.diag(np.square(edge * np.asarray(sig)))
    lo, hi = (0.0,) * d, (edge,) * d
    p = fkreg.Plan(d, order, grid, lo, hi, H[None], max_n=n, n_rhs=2, tol=tol, precision=prec)
    p.set_points(torch.tensor(x))
    out = p.smooth(torch.tensor(y), want=("mhat_grid", "mask"))
    p.sync()
    x, y = x.astype(np.float64), y.astype(np.float64)
    q = oracle.grid_points(grid, lo, hi)
    r = oracle.smooth_at(x, y, H, order, q)
    a = oracle.scale_field(x, y, H, q)
    valid = out["mask"][0].reshape(-1).cpu().numpy().astype(bool)
    bar = {1e-12: 1e-10, 1e-9: 1e-8, 1e-6: 1e-5}[tol]
    for k in range(2):
        m = out["mhat_grid"][0, k].reshape(-1).cpu().numpy()
        assert mhat_error(m, r["mhat"][:, k], r["s"][:, 0], a[:, k], valid) < bar
