"""The bin sort around the tile sizes of its scatters, bit for bit against
numpy's stable sort of the keys computed on the CPU: n at the edges of a
1024-key tile and of the range that takes them, one 8-bit and two 10-bit digit
plans, FP32 and FP64.
"""
import numpy as np
import pytest

from paper_2204_07716_gb300 import inputs
from test_gpu_parity import cpu_keys

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2204_07716_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 70_001, 524_288, 524_289])
@pytest.mark.parametrize("d,sigma,prec", [(1, 0.02, "f64"), (2, 0.05, "f32"), (2, 0.012, "f32")])
def test_permutation(n, d, sigma, prec):
    from paper_2204_07716_gb300.fkreg import Plan
    w = inputs.random_small(1100 + d, d, n, 60, 0, [sigma], precision=prec,
                            tol=1e-9 if prec == "f64" else 1e-6)
    p = Plan(d, 0, w.grid_n, w.lo, w.hi, w.H, max_n=n + 500, tol=w.tol, precision=prec)
    p.set_points(torch.tensor(w.x, dtype=torch.float32 if prec == "f32" else torch.float64))
    perm, bstart = p.get_sort()
    p.sync()
    key, bins = cpu_keys(w.x, p.geom, prec)
    assert np.array_equal(perm.cpu().numpy().astype(np.int64), np.argsort(key, kind="stable"))
    counts = np.bincount(bins, minlength=int(np.prod(p.geom["nbins"])))
    assert np.array_equal(bstart.cpu().numpy()[1:].astype(np.int64), np.cumsum(counts))
