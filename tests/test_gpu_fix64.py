"""Float64 sums in fixed point (near field and couplings of float64 plans)
against the dense sum in float64.

Bound per entry: the fixed-point kernel value is within 2 units of 2^-56 and a
charge within 2^-56 of its column's (or group's) largest, at most doubled by
the power of two above it: n 2^-54 max|x| over n terms.  The reference's own
terms carry the rounding of d squares, the root, the argument and the
exponential, |phi'| r <= 1 of it: below 2^-53 (d + 12) of a term's magnitude,
and its sums and the library's add log-depth to n roundings of 2^-53.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def dense(kernel, sigma, pts, x):
    r2 = torch.zeros((pts.shape[0], pts.shape[0]), dtype=torch.float64, device="cuda")
    for k in range(pts.shape[1]):
        df = pts[:, k:k + 1] - pts[:, k]
        r2 += df * df
    t = r2.sqrt() / sigma
    if kernel == "gauss":
        phi = (-0.5 * t * t).exp()
    elif kernel == "exp":
        phi = (-t).exp()
    else:
        phi = (1.0 + np.sqrt(3.0) * t) * (-np.sqrt(3.0) * t).exp()
    return phi, x @ phi


def setup(n, d, r, leaf, kernel="exp", sigma=1.0, eta=1e9, seed=3, shift=0.0):
    from paper_2402_09531_gb300 import Plan
    g = torch.Generator(device="cuda").manual_seed(seed)
    pts = torch.rand((n, d), dtype=torch.float64, device="cuda", generator=g) * (1.0 / torch.arange(
        1, d + 1, dtype=torch.float64, device="cuda")) + shift
    if n > 3:
        pts[n // 2] = pts[0]                 # a duplicate, and a pair far below the units of the format
        pts[n // 3] = pts[1] * (1 + 1e-15)
    x = torch.randn((r, n), dtype=torch.float64, device="cuda", generator=g)
    p = Plan(d, kernel=kernel, sigma=sigma, gamma=np.ones(d), q=1.0, eta=eta, leaf_size=leaf, precision="fp64",
             max_rhs=r)
    p.tree_build(pts)
    return p, pts, x


def check(p, pts, x, kernel, sigma):
    y = torch.empty_like(x)
    p.matvec(x, y)
    phi, ref = dense(kernel, sigma, pts, x)
    n, d = pts.shape
    tol = 2.0 ** -53 * (d + 12 + n) * (x.abs() @ phi) + n * 2.0 ** -54 * x.abs().amax(1, keepdim=True)
    assert bool(((y - ref).abs() <= tol).all()), float(((y - ref).abs() / tol).max())
    return y


# leaves of one warp's width and around it, ragged, at and beyond 128 slots
@pytest.mark.parametrize("n,leaf", [(1, 64), (2, 2), (31, 64), (32, 32), (33, 64), (129, 64), (257, 128), (1000, 100),
                                    (1500, 200), (777, 20), (4100, 128)])
@pytest.mark.parametrize("kernel,d,r", [("exp", 1, 1), ("matern32", 8, 4), ("gauss", 10, 5), ("exp", 16, 16),
                                        ("matern32", 11, 2), ("gauss", 17, 1)])
def test_near_field_matches_dense(n, leaf, kernel, d, r):
    p, pts, x = setup(n, d, r, leaf, kernel)
    check(p, pts, x, kernel, 1.0)


# box sizes against the length scale on both sides of the format's range, and
# a box far from the origin
@pytest.mark.parametrize("kernel", ["exp", "matern32", "gauss"])
@pytest.mark.parametrize("sigma,shift", [(0.01, 0.0), (0.1, 0.0), (0.3, 0.0), (1e4, 0.0), (0.7, 1000.0)])
def test_range_of_length_scales(kernel, sigma, shift):
    p, pts, x = setup(600, 5, 2, 64, kernel, sigma, shift=shift)
    check(p, pts, x, kernel, sigma)


@pytest.mark.parametrize("r", [1, 9])
def test_charges_of_any_magnitude(r):
    p, pts, x = setup(700, 4, r, 64)
    for f in (1e-300, 1e300):
        check(p, pts, x * f, "exp", 1.0)
    x[:, 5] = 1e8
    check(p, pts, x, "exp", 1.0)
    x.zero_()
    y = torch.full_like(x, 3.0)
    p.matvec(x, y)
    assert bool((y == 0).all())


@pytest.mark.parametrize("n,leaf,r,eta", [(700, 64, 1, 1e9), (700, 64, 3, 1e9), (700, 256, 9, 1e9), (3000, 64, 1, 1.0)])
def test_not_finite_charges_and_the_product_after(n, leaf, r, eta):
    p, pts, x = setup(n, 4, r, leaf, eta=eta)
    good, y = torch.empty_like(x), torch.empty_like(x)
    p.matvec(x, good)
    bad = x.clone()
    bad[0, 7] = float("inf")
    p.matvec(bad, y)
    if eta > 1e6:
        assert bool((y[0] == float("inf")).all())            # phi > 0 for every pair
    else:
        assert not bool(torch.isfinite(y[0, 7]))
    bad[0, 7] = float("nan")
    p.matvec(bad, y)
    assert bool(torch.isnan(y[0]).all())
    p.matvec(x, y)                                            # nothing of it is left
    assert torch.equal(y, good)


@pytest.mark.parametrize("q,d,r", [(0.0, 2, 1), (2.0, 4, 1), (3.0, 3, 4), (4.0, 4, 16)])
def test_couplings_match_the_oracle(q, d, r):
    """Node sets from one node to more than a warp's width."""
    import dwfmm_inputs as di
    from oracle import dwfmm_oracle as o
    from paper_2402_09531_gb300 import Plan
    gamma = np.ones(d)
    w = di.Workload("t", d=d, n=1300, gamma=gamma, kernel="exp", q=q, leaf=16, nrhs=r, seed=9)
    X, f = di.sites_and_rhs(w)
    pb = o.make_problem(X, w.kernel, o.weights_inv_gamma(gamma), q, w.leaf, 1.0)
    ref = o.fmm_matvec(pb, f)
    p = Plan(d, kernel="exp", gamma=gamma, q=q, eta=1.0, leaf_size=16, precision="fp64", max_rhs=r)
    p.set_nodes(pb.exp_.nodes)
    p.tree_build(X)
    assert p.info()[1] > 0
    y = torch.empty((r, w.n), dtype=torch.float64, device="cuda")
    p.matvec(torch.as_tensor(f, device="cuda"), y)
    err = np.linalg.norm(y.cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= 1e-12
