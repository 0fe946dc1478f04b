"""Batches whose problems need different shared memory in the passes over the
tree.  The points that share a Legendre table halve as its rows pass 79 and
159 values, so the problem with the larger index set takes less of it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


# degrees 0 .. q in the first dimension only: q + 1 values a table row for d = 1,
# q + d for the others
@pytest.mark.parametrize("q,r", [(77, (8, 8)), (77, (2, 3)), (77, (1, 9)), (78, (8, 8))])
@pytest.mark.parametrize("engine", ["graph", "persistent"])
def test_batch_of_index_sets_around_a_change_of_table(q, r, engine):
    from paper_2402_09531_gb300 import Batch, Plan
    g = torch.Generator(device="cuda").manual_seed(q)
    plans, xs = [], []
    for d, n, k in ((1, 3000, r[0]), (2, 2500, r[1])):
        gamma = np.array([1.0, 1e-4])[:d]
        pts = (2 * torch.rand((n, d), dtype=torch.float64, device="cuda", generator=g) - 1) * torch.as_tensor(
            gamma, device="cuda")
        p = Plan(d, kernel="exp", gamma=gamma, q=float(q), leaf_size=128, precision="fp32", max_rhs=k)
        p.tree_build(pts)
        assert p.info()[0] == q + 1 and p.info()[1] > 0
        plans.append(p)
        xs.append(torch.randn((k, n), dtype=torch.float64, device="cuda", generator=g))
    b = Batch(plans, list(r))
    b.set_engine(engine)
    ys = [torch.full_like(x, float("nan")) for x in xs]
    b.matvec(xs, ys)
    for p, x, y in zip(plans, xs, ys):
        want = torch.empty_like(x)
        p.matvec(x, want)
        assert float(torch.linalg.norm(y - want) / torch.linalg.norm(want)) <= 1e-6
    b.close()


def test_product_between_batched_iterations():
    """The iterations go on with their own vectors after the batch multiplied
    the caller's."""
    from paper_2402_09531_gb300 import Batch, Plan
    g = torch.Generator(device="cuda").manual_seed(5)
    plans, fs = [], []
    for n in (900, 1300):
        p = Plan(4, kernel="matern32", gamma=np.ones(4), q=2.0, leaf_size=64, precision="fp32", max_rhs=2)
        p.tree_build(torch.rand((n, 4), dtype=torch.float64, device="cuda", generator=g))
        plans.append(p)
        fs.append(torch.randn((2, n), dtype=torch.float64, device="cuda", generator=g))
    b = Batch(plans, [2, 2])
    got = []
    for between in (False, True):
        for p, f in zip(plans, fs):
            p.cg_begin(1.0, f, rtol=1e-12)
        ys = [torch.full_like(f, float("nan")) for f in fs]
        b.matvec(fs, ys)
        keep = [y.clone() for y in ys]
        b.cg_step(3)
        if between:
            b.matvec(fs, ys)
        b.cg_step(3)
        cs = [torch.empty_like(f) for f in fs]
        for p, c in zip(plans, cs):
            p.cg_result(c)
        torch.cuda.synchronize()
        assert all(torch.equal(y, k) for y, k in zip(ys, keep))
        got.append(cs)
    assert all(torch.equal(a, c) for a, c in zip(*got))
    b.close()


@pytest.mark.parametrize("r", [(1, 3, 8), (2, 12), (16, 5)])
def test_batched_iterations_with_several_classes(r):
    """Iterations of a batch whose right-hand sides fall into several classes
    (products evaluate each pair once, the iterations run the list form)."""
    from paper_2402_09531_gb300 import Batch, Plan
    g = torch.Generator(device="cuda").manual_seed(8)
    plans, fs = [], []
    for i, k in enumerate(r):
        n = 1100 + 300 * i
        p = Plan(4, kernel="matern32", gamma=np.ones(4), q=2.0, leaf_size=64, precision="fp32", max_rhs=k)
        p.tree_build(torch.rand((n, 4), dtype=torch.float64, device="cuda", generator=g))
        plans.append(p)
        fs.append(torch.randn((k, n), dtype=torch.float64, device="cuda", generator=g))
    b = Batch(plans, list(r))
    got = []
    for step in (b.cg_step, lambda it: [p.cg_step(it) for p in plans]):
        for p, f in zip(plans, fs):
            p.cg_begin(50.0, f, rtol=1e-12)
        step(2)
        step(3)
        cs = [torch.empty_like(f) for f in fs]
        for p, c in zip(plans, cs):
            p.cg_result(c)
        torch.cuda.synchronize()
        got.append(cs)
    # five iterations with a condition number of about 20: the float32 operator's
    # rounding (256 2^-24 of a row's sum) enters each of them
    for x, y in zip(*got):
        assert float(torch.linalg.norm(x - y) / torch.linalg.norm(y)) <= 1e-4
    b.close()
