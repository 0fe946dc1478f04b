"""Trees whose levels are split by one CTA per cluster, and larger ones, against
the oracle's tree: clusters around the kernel's widths, ties, duplicates and
both zeros; a plan rebuilt with other sizes equals a fresh plan."""
import numpy as np
import pytest

import dwfmm_inputs as di
from oracle import dwfmm_oracle as o

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def sites(n, d, kind):
    rng = np.random.default_rng(n + d)
    X = rng.random((n, d)) - 0.5
    if kind == "ties":
        X = np.round(X * 4) / 4 * np.where(rng.random((n, d)) < 0.5, 1.0, -1.0)   # few values, +0.0 and -0.0
    elif kind == "equal":
        X[:] = X[0]
    elif kind == "close":
        X = 1.0 + np.arange(n)[:, None] * 2.0 ** -52 * np.arange(1, d + 1)          # keys that differ in the last bits
    elif kind == "wide":
        X *= 10.0 ** rng.integers(-300, 300, (n, d))
    return X


def build(plan, X):
    plan.tree_build(torch.from_numpy(X).cuda())
    return plan.export_tree(), plan.export_lists()


@pytest.mark.parametrize("n,d,leaf,kind", [(1, 3, 4, "plain"), (3, 1, 2, "plain"), (33, 2, 2, "ties"), (1025, 5, 8, "plain"),
                                           (5632, 2, 64, "plain"), (5633, 9, 64, "ties"), (3000, 3, 16, "equal"),
                                           (3000, 2, 16, "close"), (4000, 4, 32, "wide"), (32769, 3, 128, "ties"),
                                           (70001, 2, 512, "plain")])
def test_tree_matches_oracle(n, d, leaf, kind):
    from paper_2402_09531_gb300 import Plan
    X = sites(n, d, kind)
    t = o.build_tree(X, leaf)
    p = Plan(d, gamma=np.ones(d), q=1.0, leaf_size=leaf, precision="fp32", max_rhs=1)
    g, _ = build(p, X)
    assert g["depth"] == t.depth
    np.testing.assert_array_equal(g["perm"], t.perm)
    np.testing.assert_array_equal(g["begin"], t.begin)
    np.testing.assert_array_equal(g["lo"], t.lo)
    np.testing.assert_array_equal(g["hi"], t.hi)


def test_rebuilt_plan_equals_a_fresh_one():
    from paper_2402_09531_gb300 import Plan
    w = di.small_exp_d4()

    def plan():
        return Plan(4, kernel="exp", gamma=w.gamma, q=4.0, leaf_size=64, precision="mixed", max_rhs=2)
    p = plan()
    for n in (3000, 9000, 700, 70000, 20, 3001):
        X = sites(n, 4, "plain") * w.gamma
        x = torch.from_numpy(np.random.default_rng(n).standard_normal((2, n))).cuda()
        q = plan()
        got, want = build(p, X), build(q, X)
        for k in want[0]:
            np.testing.assert_array_equal(got[0][k], want[0][k])
        for a, b in zip(got[1], want[1]):
            np.testing.assert_array_equal(a, b)
        y, z = torch.empty_like(x), torch.empty_like(x)
        p.matvec(x, y)
        q.matvec(x, z)
        assert torch.equal(y, z)
