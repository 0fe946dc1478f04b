"""Workspaces whose size follows the right-hand sides, under graphs that hold
their addresses."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def setup(prec, n=1500, d=4, r=16, leaf=64, kernel="matern32", eta=1e9, seed=11):
    from paper_2402_09531_gb300 import Plan
    g = torch.Generator(device="cuda").manual_seed(seed)
    pts = torch.rand((n, d), dtype=torch.float64, device="cuda", generator=g)
    x = torch.randn((r, n), dtype=torch.float64, device="cuda", generator=g)
    p = Plan(d, kernel=kernel, gamma=np.ones(d), q=1.0, eta=eta, leaf_size=leaf, precision=prec, max_rhs=16)
    p.tree_build(pts)
    return p, pts, x


@pytest.mark.parametrize("prec", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("first,wide", [(1, 2), (1, 8), (4, 16)])
def test_solve_replayed_after_a_wider_product(prec, first, wide):
    """The kept iterations of a solve are replayed after a product (and an
    incremental step) that needed larger workspaces."""
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        p, pts, x = setup(prec)
        f = x[:first].contiguous()
        got = []
        for _ in range(2):
            c = torch.zeros_like(f)
            status, its, _ = p.solve(1e-1, f, c, rtol=1e-10, maxit=3000)
            assert status == 0 and its > 32     # three runs of 16 iterations: plain, captured, replayed
            got.append(c)
            y = torch.empty_like(x[:wide])
            p.matvec(x[:wide].contiguous(), y)
            p.cg_begin(1e-1, f, rtol=1e-10)
            p.cg_step(1)
        q, _, _ = setup(prec)
        c = torch.zeros_like(f)
        q.solve(1e-1, f, c, rtol=1e-10, maxit=3000)
        stream.synchronize()
        assert torch.equal(got[0], got[1]) and torch.equal(got[0], c)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_tree_build_waits_for_products_on_other_streams(prec):
    """New sites on another stream do not touch the tree that a product is
    still reading."""
    p, pts, x = setup(prec, n=60000, d=8, r=4, leaf=128, kernel="exp", eta=1.0)
    want, y = torch.empty_like(x), torch.empty_like(x)
    p.matvec(x, want)
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    other = pts.flip(0).contiguous() * 0.5
    torch.cuda.synchronize()
    for _ in range(3):
        with torch.cuda.stream(a):
            p.matvec(x, y)
        with torch.cuda.stream(b):
            p.tree_build(other)
            p.tree_build(pts)
        torch.cuda.synchronize()
        assert torch.equal(y, want)


# partial sums of 42 MB (float32) or 84 MB (float64) a right-hand side
@pytest.mark.parametrize("prec,r,engines", [("fp64", 4, ("fp64_list", "fp64_symmetric")), ("fp32", 8, None),
                                            ("mixed", 8, None)])
def test_products_without_memory_for_partial_sums(prec, r, engines):
    """The list kernel runs where the pairs' partial sums cannot be allocated."""
    p, pts, x = setup(prec, n=40000, d=8, leaf=128, kernel="exp")
    want = torch.empty_like(x)
    p.matvec(x, want)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    block = torch.empty(torch.cuda.mem_get_info()[0] - (160 << 20), dtype=torch.uint8, device="cuda")
    y = torch.empty_like(x[:r])
    bound = 1e-13 if prec == "fp64" else 1e-5
    try:
        p.matvec(x[:r].contiguous(), y)
        torch.cuda.synchronize()
        few = p.near_engine()
    finally:
        del block
        torch.cuda.empty_cache()
    assert float(torch.linalg.norm(y - want[:r]) / torch.linalg.norm(want[:r])) <= bound
    y2 = torch.empty_like(y)
    p.matvec(x[:r].contiguous(), y2)
    assert float(torch.linalg.norm(y2 - want[:r]) / torch.linalg.norm(want[:r])) <= bound
    if engines:
        assert (few, p.near_engine()) == engines


@pytest.mark.parametrize("prec,first,r", [("fp64", 1, 4), ("fp64", 1, 16), ("fp32", 1, 8), ("fp32", 1, 12),
                                          ("mixed", 2, 8), ("mixed", 9, 16)])
def test_capture_of_a_wider_product(prec, first, r):
    """A product with more right-hand sides than any before, captured; and the
    same graph after its workspaces grew outside."""
    p, pts, x = setup(prec)
    y, want = torch.empty_like(x), torch.empty_like(x)
    p.matvec(x[:first].contiguous(), y[:first].contiguous())
    torch.cuda.synchronize()
    xr, yr = x[:r].contiguous(), torch.empty_like(x[:r])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        p.matvec(xr, yr)
    yr.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    got = yr.clone()
    p.matvec(xr, want[:r])
    bound = 1e-13 if prec == "fp64" else 1e-5
    assert float(torch.linalg.norm(got - want[:r]) / torch.linalg.norm(want[:r])) <= bound
    p.matvec(x, want)
    yr.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(yr, got)


@pytest.mark.parametrize("prec,n,nrhs", [("fp64", 20000, 1), ("mixed", 20000, 4), ("fp32", 3000, 1)])
def test_admission_estimate_covers_a_request(prec, n, nrhs):
    """Device memory of a plan that multiplied, iterated and took a residual."""
    from paper_2402_09531_gb300 import Plan
    from paper_2402_09531_gb300.serving import estimate_bytes
    d = 16
    gamma = 2.0 ** -np.arange(d)
    g = torch.Generator(device="cuda").manual_seed(2)
    pts = (2 * torch.rand((n, d), dtype=torch.float64, device="cuda", generator=g) - 1) * torch.as_tensor(gamma, device="cuda")
    f = torch.randn((nrhs, n), dtype=torch.float64, device="cuda", generator=g)
    c, y = torch.zeros_like(f), torch.empty_like(f)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    p = Plan(d, kernel="exp", gamma=gamma, q=6.0, leaf_size=128, precision=prec, max_rhs=nrhs)
    p.tree_build(pts)
    p.matvec(f, y)
    p.cg_begin(10.0, f)
    p.cg_step(2)
    p.cg_result(c)
    p.residual(10.0, f, c)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    assert used <= estimate_bytes(n, d, nrhs, 128, p.info()[0]), used
