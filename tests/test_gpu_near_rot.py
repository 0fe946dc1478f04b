"""Float32 near field that evaluates each unordered pair once (up to 8
right-hand sides) against the dense sum in float64.

Bound per entry: a float32 kernel value carries the rounding of d squares, the
approximate root and exponential (2^-22 each, |phi'| r <= 1) and, for the
Gaussian, of three terms that cancel (their size over the box, below 8 here);
charges round once, sums of at most 512 terms stay in float32 before float64
takes over: (512 / 2 + 4 d + 32) 2^-23 of the terms' magnitudes covers it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


# leaves of 32 sites (a warp's width), around it, ragged, at 256 slots; and
# leaves below 32 or above 256, which keep the one-CTA-per-leaf kernel
@pytest.mark.parametrize("n,leaf", [(32, 32), (33, 64), (65, 64), (1000, 100), (1025, 256), (2048, 256), (999, 20),
                                    (1300, 512)])
@pytest.mark.parametrize("kernel,d,r,prec", [("exp", 1, 1, "fp32"), ("exp", 16, 1, "mixed"), ("matern32", 8, 4, "fp32"),
                                             ("matern32", 11, 3, "mixed"), ("gauss", 10, 8, "fp32"),
                                             ("gauss", 19, 5, "mixed"), ("exp", 4, 2, "fp32")])
def test_near_field_matches_dense(n, leaf, kernel, d, r, prec):
    from paper_2402_09531_gb300 import Plan
    g = torch.Generator(device="cuda").manual_seed(n + d)
    pts = torch.rand((n, d), dtype=torch.float64, device="cuda", generator=g) / torch.arange(
        1, d + 1, dtype=torch.float64, device="cuda")
    pts[n // 2] = pts[0]
    x = torch.randn((r, n), dtype=torch.float64, device="cuda", generator=g)
    p = Plan(d, kernel=kernel, gamma=np.ones(d), q=1.0, eta=1e9, leaf_size=leaf, precision=prec, max_rhs=r)
    p.tree_build(pts)
    y, y2 = torch.empty_like(x), torch.empty_like(x)
    p.matvec(x, y)
    r2 = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    for k in range(d):
        df = pts[:, k:k + 1] - pts[:, k]
        r2 += df * df
    t = r2.sqrt()
    phi = {"gauss": lambda: (-0.5 * r2).exp(), "exp": lambda: (-t).exp(),
           "matern32": lambda: (1 + np.sqrt(3.0) * t) * (-np.sqrt(3.0) * t).exp()}[kernel]()
    tol = (256 + 4 * d + 32) * 2.0 ** -23 * (x.abs() @ phi)
    # the float32 coordinates of the exponential's coincident and close pairs: |r| is off by 2^-23 |x|
    assert bool(((y - x @ phi).abs() <= tol).all()), float(((y - x @ phi).abs() / tol).max())
    p.matvec(x, y2)
    assert torch.equal(y, y2)
    bad = x.clone()
    bad[0, n // 3] = float("nan")
    p.matvec(bad, y2)
    assert bool(torch.isnan(y2[0]).all())
    if r > 1:
        assert torch.equal(y2[1:], y[1:])
