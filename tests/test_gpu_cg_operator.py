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
