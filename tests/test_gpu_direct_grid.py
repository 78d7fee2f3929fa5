"""Grid fields of the direct sums against the oracle, on both sides of the rule that picks
the kernel: patches of 32 points (many patches, few samples inside a support) and a warp
to each point (1-D, coarse grids, wide supports), at strength counts around the
instantiated sizes, with ragged patches; and bandwidths of one plan that fall on
different sides, each in its own slice of the fields.

Bars of the fields' natural size as in test_gpu_direct_sums: FP64 1e-10, FP32 1e-5.
"""
import numpy as np
import pytest

import oracle
from paper_2204_07716_gb300 import inputs
from parity_util import field_error, field_scale_sigma, sample_grid_indices

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2204_07716_gb300 import build
    build.build()
    oracle.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def check(d, order, prec, n, grid, sigmas, rhs, kernel, full_h=False):
    from paper_2204_07716_gb300.fkreg import Plan
    w = inputs.random_small(1300 + 10 * d + order, d, n, grid, order, sigmas, precision=prec,
                            n_rhs=rhs, full_h=full_h)
    dt = torch.float32 if prec == "f32" else torch.float64
    p = Plan(d, order, w.grid_n, w.lo, w.hi, w.H, max_n=n, n_rhs=rhs, precision=prec, kernel=kernel)
    p.set_points(torch.tensor(w.x, dtype=dt))
    mom = p.smooth(torch.tensor(w.y, dtype=dt), want=("moments",))["moments"]
    p.sync()
    ft = np.float32 if prec == "f32" else np.float64
    x, y = w.x.astype(ft).astype(np.float64), w.y.astype(ft).astype(np.float64)
    idx = sample_grid_indices(w.grid_n, 300, seed=d)
    q = oracle.grid_points(w.grid_n, w.lo, w.hi)[idx]
    bar = 1e-10 if prec == "f64" else 1e-5
    es, et = oracle.monomials(d, 2 * order), oracle.monomials(d, order)
    for b, H in enumerate(w.H):
        got = mom[b].reshape(mom.shape[1], -1).double().cpu().numpy()[:, idx]
        one = np.ones((1, n))
        s = oracle.moment_sums_compact(x, one, H, 2 * order, q, kernel)[:, 0, :]
        for k, e in enumerate(es):
            assert field_error(got[k], s[:, k], s[:, 0], field_scale_sigma(H, e)) < bar, (b, k)
        for r in {0, rhs // 2, rhs - 1}:
            t = oracle.moment_sums_compact(x, y[r:r + 1], H, order, q, kernel)[:, 0, :]
            a = oracle.moment_sums_compact(x, np.abs(y[r:r + 1]), H, 0, q, kernel)[:, 0, 0]
            for k, e in enumerate(et):
                g = got[len(es) + r * len(et) + k]
                assert field_error(g, t[:, k], a, field_scale_sigma(H, e)) < bar, (b, r, k)


# patches: 0.35 reach inside max(1, 608 / patches) < inside + 400 (FP32), reach inside
# max(1, 608 / patches) < inside + 200 (FP64), on the GB300's 152 SMs
@pytest.mark.parametrize("d,order,prec,n,grid,sigma,rhs,kernel,full_h", [
    (2, 0, "f32", 3000, (90, 70), 0.08, 5, "triweight", False),
    (2, 1, "f32", 3000, (90, 70), 0.08, 1, "epanechnikov", False),
    (2, 1, "f32", 3000, (89, 73), 0.08, 4, "biweight", True),
    (2, 1, "f32", 3000, (90, 70), 0.08, 13, "epanechnikov", False),
    (2, 2, "f32", 3000, (90, 70), 0.08, 2, "triweight", False),
    (2, 1, "f64", 1500, (121, 97), 0.06, 1, "epanechnikov", False),
    (2, 0, "f64", 1500, (121, 97), 0.06, 12, "triangle", True),
    (2, 2, "f64", 1500, (121, 97), 0.06, 5, "biweight", False),
    (3, 1, "f32", 3000, (22, 25, 21), 0.15, 3, "epanechnikov", False),
    (3, 0, "f64", 3000, (22, 25, 21), 0.12, 5, "triweight", False),
])
def test_patches(d, order, prec, n, grid, sigma, rhs, kernel, full_h):
    check(d, order, prec, n, grid, [sigma], rhs, kernel, full_h)


@pytest.mark.parametrize("d,order,prec,n,grid,sigma,rhs,kernel,full_h", [
    (1, 0, "f32", 4000, (33,), 0.01, 12, "epanechnikov", False),
    (1, 1, "f64", 4000, (250,), 0.1, 8, "triweight", False),
    (1, 2, "f32", 3000, (70,), 0.08, 5, "biweight", False),
    (2, 1, "f32", 5000, (9, 13), 0.1, 1, "epanechnikov", True),
    (2, 1, "f64", 5000, (40, 31), 0.2, 6, "triangle", False),
    (2, 2, "f32", 5000, (16, 17), 0.15, 8, "triweight", False),
    (3, 1, "f64", 4000, (8, 9, 7), 0.25, 5, "epanechnikov", True),
    (3, 0, "f32", 4000, (10, 9, 11), 0.2, 36, "biweight", False),
])
def test_points(d, order, prec, n, grid, sigma, rhs, kernel, full_h):
    check(d, order, prec, n, grid, [sigma], rhs, kernel, full_h)


def test_bandwidths_on_both_sides():
    check(2, 1, "f32", 6000, (90, 70), [0.05, 0.3, 0.04, 0.03, 0.35], 2, "epanechnikov")
