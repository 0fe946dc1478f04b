"""A float64 plan's blocking solve and its incremental CG are one method: the same
iterates, bit for bit (33 iterations turn a change of the operator's last bits
into one of 1e-12 to 4e-12 of the solution)."""
import numpy as np
import pytest

import dwfmm_inputs as di

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("kernel,n,nrhs,leaf,seed", [("matern32", 2000, 2, 64, 0), ("matern32", 2000, 2, 64, 4),
                                                     ("exp", 1500, 1, 64, 1), ("gauss", 1100, 5, 200, 2)])
def test_incremental_iterates_are_the_solves(kernel, n, nrhs, leaf, seed):
    from paper_2402_09531_gb300 import Plan
    w = di.scaled(di.small_exp_d4(), n, nrhs=nrhs)
    w.seed = seed
    X, f = di.sites_and_rhs(w)
    fd, Xd = torch.from_numpy(f).cuda(), torch.from_numpy(X).cuda()
    plans = [Plan(d=4, kernel=kernel, gamma=w.gamma, q=4.0, leaf_size=leaf, precision="fp64", max_rhs=nrhs)
             for _ in range(2)]
    for p in plans:
        p.tree_build(Xd)
    c, inc = torch.zeros_like(fd), torch.zeros_like(fd)
    status, its, _ = plans[0].solve(5.0, fd, c, rtol=1e-10, maxit=500)
    assert status == 0
    plans[1].cg_begin(5.0, fd, rtol=1e-10)
    plans[1].cg_step(its)
    plans[1].cg_result(inc)
    torch.cuda.synchronize()
    _, status, iters, _ = plans[1].cg_poll()
    assert np.all(status == 1) and int(iters.max()) == its
    assert torch.equal(c, inc)


def test_iterations_after_a_new_tree_need_a_new_begin():
    """The vectors of the iterations go with the tree: refused on the host."""
    from paper_2402_09531_gb300 import DwfmmError, Plan
    p = Plan(d=3, kernel="exp", gamma=np.ones(3), q=1.0, leaf_size=64, precision="fp32", max_rhs=1)
    g = torch.Generator(device="cuda").manual_seed(1)
    pts = torch.rand((500, 3), dtype=torch.float64, device="cuda", generator=g)
    f = torch.randn((1, 500), dtype=torch.float64, device="cuda", generator=g)
    p.tree_build(pts)
    p.cg_begin(1.0, f)
    p.cg_step(2)
    p.tree_build(pts)
    for call in (lambda: p.cg_step(1), lambda: p.cg_result(torch.empty_like(f))):
        with pytest.raises(DwfmmError) as e:
            call()
        assert e.value.status == 7
    p.cg_begin(1.0, f)
    p.cg_step(2)
    torch.cuda.synchronize()
