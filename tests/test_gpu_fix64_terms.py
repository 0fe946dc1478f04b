"""Float64 products term by term: a small kernel value, a small charge beside a
large one, keep float64's relative accuracy.

Bound per entry, of the terms' magnitudes: the library's kernel value is within
2^-52, and its coordinates are rounded to at most 2^-58 of the diagonal, which
moves w < 2^5 by sqrt(d) 2^-53 (exponential, Matern) or twice that (Gaussian).
The reference's carries the rounding of d squares, the root, the argument (up to
22) and the exponential: 22 (d / 2 + 3) 2^-53 for the first two, 22 (d + 4) 2^-53
for the Gaussian.  Sums add at most n roundings each.  (22 (d + 4) + 2 n + 16)
2^-53 covers it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def kernel_matrix(kernel, sigma, pts):
    r2 = torch.zeros((pts.shape[0], pts.shape[0]), dtype=torch.float64, device="cuda")
    for k in range(pts.shape[1]):
        df = pts[:, k:k + 1] - pts[:, k]
        r2 += df * df
    t = r2.sqrt() / sigma
    if kernel == "gauss":
        return (-0.5 * t * t).exp()
    if kernel == "exp":
        return (-t).exp()
    return (1.0 + np.sqrt(3.0) * t) * (-np.sqrt(3.0) * t).exp()


# boxes near the top of the format's range (diagonals just below 4 sigma, 8 sigma,
# 16 sigma), where the smallest kernel values are below 2^-11
SIGMA = {"exp": 0.062, "matern32": 0.124, "gauss": 0.248}


def setup(kernel, d, r, leaf, n=600):
    from paper_2402_09531_gb300 import Plan
    g = torch.Generator(device="cuda").manual_seed(d + leaf)
    pts = torch.rand((n, d), dtype=torch.float64, device="cuda", generator=g) * (0.985 / d ** 0.5)
    pts[0], pts[1] = 0.0, 0.985 / d ** 0.5
    p = Plan(d, kernel=kernel, sigma=SIGMA[kernel], gamma=np.ones(d), q=1.0, eta=1e9, leaf_size=leaf, precision="fp64",
             max_rhs=r)
    p.tree_build(pts)
    return p, kernel_matrix(kernel, SIGMA[kernel], pts), g


def check(p, phi, x, d):
    y = torch.empty_like(x)
    p.matvec(x, y)
    for yr, xr in zip(y, x):
        ref, size = (phi * xr).sum(1), (phi * xr.abs()).sum(1)
        tol = 2.0 ** -53 * (22 * (d + 4) + 2 * x.shape[1] + 16) * size
        assert bool(((yr - ref).abs() <= tol).all()), float(((yr - ref).abs() / tol).max())


# the symmetric form (leaves of 37 sites), the list form (leaves below 32; 9 columns)
@pytest.mark.parametrize("r,leaf", [(1, 64), (3, 64), (2, 16), (9, 64), (16, 16)])
@pytest.mark.parametrize("kernel,d", [("exp", 1), ("exp", 4), ("matern32", 8), ("gauss", 10), ("gauss", 16)])
def test_unit_vectors_and_mixed_magnitudes(kernel, d, r, leaf):
    p, phi, g = setup(kernel, d, r, leaf)
    n = phi.shape[0]
    assert float(phi.min()) < 2.0 ** -11
    x = torch.zeros((r, n), dtype=torch.float64, device="cuda")
    for k in range(r):
        x[k, k] = 1.0                      # columns of K
    check(p, phi, x, d)
    x = torch.randn((r, n), dtype=torch.float64, device="cuda", generator=g)
    x[0, 1] = 1e17                         # one large charge among small ones
    check(p, phi, x, d)
    x *= 10.0 ** (40 * torch.rand((r, n), dtype=torch.float64, device="cuda", generator=g) - 20)
    check(p, phi, x, d)
    x[:, 2] = 1e-310                       # below the normal range
    check(p, phi, x, d)


@pytest.mark.parametrize("r", [1, 4, 16])
def test_small_couplings_of_a_unit_vector(r):
    """One node a cluster: the far field of a unit vector is a single kernel
    value, down to 2^-14."""
    import dwfmm_inputs as di
    from oracle import dwfmm_oracle as o
    from paper_2402_09531_gb300 import Plan
    d, gamma = 4, np.full(4, 0.98 * 4.0)
    w = di.Workload("t", d=d, n=1300, gamma=gamma, kernel="exp", q=0.0, leaf=16, nrhs=r, seed=9)
    X, f = di.sites_and_rhs(w)
    f[:] = 0.0
    for k in range(r):
        f[k, 10 * k] = 1.0
    pb = o.make_problem(X, w.kernel, o.weights_inv_gamma(gamma), w.q, w.leaf, 1.0)
    ref = o.fmm_matvec(pb, f)
    p = Plan(d, kernel="exp", gamma=gamma, q=0.0, eta=1.0, leaf_size=16, precision="fp64", max_rhs=r)
    p.set_nodes(pb.exp_.nodes)
    p.tree_build(X)
    assert p.info()[1] > 0
    y = torch.empty((r, w.n), dtype=torch.float64, device="cuda")
    p.matvec(torch.as_tensor(f, device="cuda"), y)
    assert ref.min() < 2.0 ** -13
    assert np.max(np.abs(y.cpu().numpy() / ref - 1.0)) <= 2.0 ** -53 * (22 * (d + 4) + 64)
