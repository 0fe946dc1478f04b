"""Direct sums and evaluation at new points against the dense sum in float64,
at the edges of their tiles, parts and paths.

Float32 bound per entry: d squares, the approximate root and exponential (2^-22
each, |phi'| r <= 1), charges rounded once, sums of at most 256 terms before a
compensated sum takes them: (256 / 2 + 4 d + 32) 2^-23 of the terms'
magnitudes.  Float64: 2^-53 (d + 12 + n) of them.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def phi_matrix(kernel, a, b):
    r2 = torch.zeros((a.shape[0], b.shape[0]), dtype=torch.float64, device="cuda")
    for k in range(a.shape[1]):
        df = a[:, k:k + 1] - b[:, k]
        r2 += df * df
    t = r2.sqrt()
    return {"gauss": lambda: (-0.5 * r2).exp(), "exp": lambda: (-t).exp(),
            "matern32": lambda: (1 + np.sqrt(3.0) * t) * (-np.sqrt(3.0) * t).exp()}[kernel]()


def points(n, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand((n, d), dtype=torch.float64, device="cuda", generator=g) / torch.arange(
        1, d + 1, dtype=torch.float64, device="cuda"), g


@pytest.mark.parametrize("n", [1, 31, 33, 255, 257, 1025, 1536, 1537, 3000])
@pytest.mark.parametrize("kernel,d,r", [("exp", 1, 1), ("matern32", 6, 3), ("gauss", 10, 8), ("exp", 16, 16)])
def test_direct_sum(n, kernel, d, r):
    import paper_2402_09531_gb300 as pkg
    pts, g = points(n, d, n + d)
    wide = torch.full((n, d + 3), 7.0, dtype=torch.float64, device="cuda")   # leading dimensions above the sizes
    wide[:, :d] = pts
    x = torch.randn((r, n + 5), dtype=torch.float64, device="cuda", generator=g)
    y = torch.full((r, n + 2), -1.0, dtype=torch.float64, device="cuda")
    s = torch.cuda.current_stream().cuda_stream

    def call(xx, yy):
        return pkg.lib().dwfmm_direct_sum_noalloc(pkg.KERNELS[kernel], 1.0, wide.data_ptr(), n, d, wide.stride(0),
                                                  xx.data_ptr(), yy.data_ptr(), r, xx.stride(0), yy.stride(0), s)
    assert call(x, y) == 0
    phi = phi_matrix(kernel, pts, pts)
    tol = (128 + 4 * d + 32) * 2.0 ** -23 * (x[:, :n].abs() @ phi)
    assert bool(((y[:, :n] - x[:, :n] @ phi).abs() <= tol).all())
    assert bool((y[:, n:] == -1.0).all())
    over = x.clone()                                  # y over x: the charges are read before y is written
    assert call(over, over) == 0
    assert torch.equal(over[:, :n], y[:, :n]) or bool(((over[:, :n] - x[:, :n] @ phi).abs() <= tol).all())
    assert torch.equal(over[:, n:], x[:, n:])


@pytest.mark.parametrize("prec", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("n,nt,leaf,r", [(50, 1, 64, 1), (3000, 1, 64, 3), (3000, 257, 128, 9), (700, 4000, 32, 2)])
def test_evaluate(prec, n, nt, leaf, r):
    from paper_2402_09531_gb300 import Plan
    d = 5
    pts, g = points(n, d, n)
    tg = torch.rand((nt, d), dtype=torch.float64, device="cuda", generator=g) * 1.5 - 0.25   # inside the box and around
    c = torch.randn((r, n), dtype=torch.float64, device="cuda", generator=g)
    p = Plan(d, kernel="matern32", gamma=np.ones(d), q=1.0, leaf_size=leaf, precision=prec, max_rhs=r)
    p.tree_build(pts)
    out = torch.full((r, nt), float("nan"), dtype=torch.float64, device="cuda")
    p.evaluate(tg, c, out)
    phi = phi_matrix("matern32", tg, pts)
    per = 2.0 ** -53 * (d + 12 + n) if prec == "fp64" else (128 + 4 * d + 32) * 2.0 ** -23
    tol = per * (c.abs() @ phi.t())
    assert bool(((out - c @ phi.t()).abs() <= tol).all())
    again = torch.full_like(out, float("nan"))        # another size in between: workspaces are kept
    p.evaluate(tg[:1], c, again[:, :1].contiguous())
    p.evaluate(tg, c, again)
    assert torch.equal(again, out)


def test_evaluate_many_target_blocks_one_right_hand_side():
    """More CTAs than the GPU holds at once, four warps each: the compensation
    of one right-hand side has to be cleared by the threads that use it."""
    from paper_2402_09531_gb300 import Plan
    n, nt, d = 4000, 60001, 10
    pts, g = points(n, d, 5)
    tg = points(nt, d, 6)[0]
    c = torch.randn((1, n), dtype=torch.float64, device="cuda", generator=g)
    p = Plan(d, kernel="gauss", gamma=np.ones(d), q=1.0, leaf_size=256, precision="fp32", max_rhs=1)
    p.tree_build(pts)
    out = torch.empty((1, nt), dtype=torch.float64, device="cuda")
    p.evaluate(tg, c, out)
    phi = phi_matrix("gauss", tg, pts)
    tol = (128 + 4 * d + 32) * 2.0 ** -23 * (c.abs() @ phi.t())
    assert bool(((out - c @ phi.t()).abs() <= tol).all())
