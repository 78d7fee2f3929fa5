"""Scalars of the direct sums with many more groups of 32 samples than a GPU holds blocks:
blocks take groups as they get free, yet RSS, traces and GCV repeat bit for bit and
agree with plain FP64 sums over all pairs.

Bars against FP64, as for the values (FP64 1e-10, FP32 1e-5 of the sums of magnitudes):
with S|.| the smoother of magnitudes, |d mhat| <= bar S|y|, so |d RSS| <= 2 bar sum |r| S|y|
(and its square), |d w'Sw| <= bar |w|'S|w|, and each term of the exact trace is a kernel
value over a sum of positive terms.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2204_07716_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def samples(n, prec, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand(n, 2, generator=g, device="cuda", dtype=torch.float64)
    c = 0.4 + 0.05 * torch.randn(n, 2, generator=g, device="cuda", dtype=torch.float64)
    x = torch.where(torch.rand(n, 1, generator=g, device="cuda") < 0.2, c.clamp(0, 1), x)
    y = torch.sin(5 * x[:, 0]) + 0.3 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    t = torch.float32 if prec == "f32" else torch.float64
    return x.to(t), y.to(t)


def plan(n, prec, order, sigma, probes):
    import numpy as np
    from paper_2204_07716_gb300.fkreg import Plan
    return Plan(2, order, (40, 50), (0.0, 0.0), (1.0, 1.0), np.eye(2)[None] * sigma**2, max_n=n,
                max_probes=probes, precision=prec, kernel="epanechnikov")


@pytest.mark.parametrize("prec,n", [("f32", 150_001), ("f64", 90_000)])
def test_scalars_repeat(prec, n):
    x, y = samples(n, prec, 5)
    p = plan(n, prec, 1, 0.02, 3)
    p.set_points(x)
    runs = [{k: v.clone() for k, v in p.df(y, 3, seed=11, want=("mhat_at_x",)).items()}
            for _ in range(6)]
    p.sync()
    for k in ("rss", "trace", "gcv", "mhat_at_x"):
        assert all(torch.equal(r[k], runs[0][k]) for r in runs[1:]), k


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_scalars_of_many_groups(prec):
    n, sigma, probes = 60_001, 0.015, 2
    x, y = samples(n, prec, 6)
    z = torch.randn(probes, n, generator=torch.Generator(device="cuda").manual_seed(7),
                    device="cuda", dtype=torch.float64).to(x.dtype)
    p = plan(n, prec, 0, sigma, probes)
    p.set_points(x)
    out = p.df(y, probes, probes=z, want=("mhat_at_x",))
    p.sync()
    xd = x.double() / sigma
    v = torch.cat([y.double()[None], z.double()])
    v = torch.cat([v, v.abs()]).T  # strengths, then their magnitudes
    sv, s0 = torch.empty(n, v.shape[1], device="cuda", dtype=torch.float64), torch.empty(
        n, device="cuda", dtype=torch.float64)
    for i in range(0, n, 1000):
        d = (xd[i:i + 1000, None, 0] - xd[None, :, 0]) ** 2 + (xd[i:i + 1000, None, 1] - xd[None, :, 1]) ** 2
        k = (1.0 - d).clamp_min(0.0)
        s0[i:i + 1000] = k.sum(1)
        sv[i:i + 1000] = k @ v
    sv /= s0[:, None]
    bar = 1e-10 if prec == "f64" else 1e-5
    r = v[:, 0] - sv[:, 0]
    a = sv[:, 1 + probes]
    assert abs(out["rss"].item() - (r * r).sum().item()) <= (
        2 * bar * (r.abs() * a).sum() + bar**2 * (a * a).sum()).item()
    w, sw = v[:, 1:1 + probes], sv[:, 1:1 + probes]
    mag = (v[:, 2 + probes:] * sv[:, 2 + probes:]).sum(0)
    wsw, ww = (w * sw).sum(0), (w * w).sum(0)
    got = out["trace"][0].double()
    assert abs(got[0] - n * (wsw / ww).mean()) <= bar * n * (mag / ww).mean()
    assert abs(got[1] - wsw.mean()) <= bar * mag.mean()
    exact = (1.0 / s0).sum()
    assert abs(got[2] - exact) <= bar * exact
