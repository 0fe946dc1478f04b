"""Workloads that stand for what programs do with this library.

Each case is one pass through the public entry points of
``paper_2402_09531_gb300.dwfmm``: a matrix-vector product, a product on sites
that just arrived (tree build included), conjugate gradient iterations, a
batch of uneven problems, the interpolant at new points, an allocation-free
direct sum.  ``prepare`` makes what the program holds before the call (sites
and right-hand sides on the GPU, the plan, its tree, the batch), ``run`` is
the call, ``exact`` the dense sum in float64 with plain torch.  The compressed
product differs from the dense one by the method's own compression error, the
direct sums only by rounding.

The library hands every result over in float64 buffers.  Plans in ``fp32`` and
``mixed`` compute to float32 accuracy, and a program that chose them keeps
float32 results: ``run`` returns those as float32.
"""
from __future__ import annotations

import functools
import math

import torch

from paper_2402_09531_gb300 import dwfmm

# Site and expansion parameters of the library's workloads: dimension weights
# gamma_k (sites are uniform in prod_k [-gamma_k, gamma_k]), kernel, degree q
# of the index set, sites per leaf.
FAMILIES = {
    "exp_d4": dict(d=4, gamma="halving", kernel="exp", q=4.0, leaf=64),
    "matern_d8": dict(d=8, gamma="inverse_square", kernel="matern32", q=6.0, leaf=128),
    "gauss_d10": dict(d=10, gamma="sqrt_half", kernel="gauss", q=8.0, leaf=256),
    "matern_d12": dict(d=12, gamma="inverse_square", kernel="matern32", q=5.0, leaf=128),
    "exp_d16": dict(d=16, gamma="half_powers", kernel="exp", q=6.0, leaf=128),
}
LAMBDA = 1e-2      # ridge of the conjugate gradient cases


def _gamma(rule: str, d: int) -> list[float]:
    if rule == "halving":
        return [2.0 ** -k for k in range(d)]
    if rule == "inverse_square":
        return [1.0 / (k * k) for k in range(1, d + 1)]
    if rule == "sqrt_half":
        return [2.0 ** (-0.5 * k) for k in range(d)]
    return [2.0 ** -k for k in range(1, d + 1)]


def listed() -> list[dict]:
    return [
        # one right-hand side on a few thousand sites: the smallest product,
        # bound by launches and latency
        dict(name="matvec_fp64_exp_d4_n4096_r1", kind="matvec", family="exp_d4", precision="fp64", n=4096, nrhs=1),
        # the plain float64 operator at size: what a float64 solve calls at
        # every iteration
        dict(name="matvec_fp64_matern_d8_n262144_r1", kind="matvec", family="matern_d8", precision="fp64", n=262144,
             nrhs=1),
        # a block of right-hand sides against the float64 operator: the
        # residual that iterative refinement of a mixed solve recomputes
        dict(name="matvec_fp64_gauss_d10_n12289_r16", kind="matvec", family="gauss_d10", precision="fp64", n=12289,
             nrhs=16),
        # the headline product: a million sites, 16 right-hand sides
        dict(name="matvec_mixed_gauss_d10_n1048576_r16", kind="matvec", family="gauss_d10", precision="mixed",
             n=1048576, nrhs=16),
        # a served request's operator: one right-hand side, many dimensions
        dict(name="matvec_mixed_exp_d16_n50021_r1", kind="matvec", family="exp_d16", precision="mixed", n=50021,
             nrhs=1),
        # a few right-hand sides in float32
        dict(name="matvec_fp32_matern_d8_n100003_r4", kind="matvec", family="matern_d8", precision="fp32", n=100003,
             nrhs=4),
        # a block of right-hand sides under a kernel that is not the Gaussian
        dict(name="matvec_mixed_matern_d12_n65536_r16", kind="matvec", family="matern_d12", precision="mixed",
             n=65536, nrhs=16),
        # sites that just arrived: tree, lists and expansion data are built,
        # then one product
        dict(name="new_sites_mixed_exp_d16_n20011_r1", kind="new_sites", family="exp_d16", precision="mixed", n=20011,
             nrhs=1),
        # a slice of a served solve: conjugate gradient iterations of a small
        # request on its own stream
        dict(name="cg_mixed_exp_d16_n3001_i8", kind="cg", family="exp_d16", precision="mixed", n=3001, nrhs=1,
             iterations=8),
        # many uneven problems in one fused product
        dict(name="batch_fp32_matern_p16", kind="batch", precision="fp32", problems=16, n_min=2048, n_max=32768,
             picks=4),
        # prediction: the interpolant of a solved system at new points
        dict(name="evaluate_mixed_gauss_d10_n131072_t10007_r1", kind="evaluate", family="gauss_d10",
             precision="mixed", n=131072, targets=10007, nrhs=1),
        # exact product of a small set of sites without any allocation
        dict(name="direct_matern_d6_n1021_r3", kind="direct", kernel="matern32", d=6, n=1021, nrhs=3),
    ]


def _log(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["matvec", "matvec", "matvec", "matvec", "new_sites", "cg", "batch", "evaluate", "direct"])
    family = rng.choice(sorted(FAMILIES))
    precision = rng.choice(["fp64", "fp32", "mixed"])
    nrhs = rng.choice([1, 1, 1, 2, 3, 4, 5, 7, 8, 9, 12, 16])
    if kind == "matvec":
        n = _log(rng, 1000, 300000 if precision != "fp64" else (60000 if nrhs <= 4 else 20000))
        return dict(kind=kind, family=family, precision=precision, n=n, nrhs=nrhs)
    if kind == "new_sites":
        return dict(kind=kind, family=family, precision=precision, n=_log(rng, 1000, 20000), nrhs=nrhs)
    if kind == "cg":
        return dict(kind=kind, family=family, precision=precision, n=_log(rng, 1000, 8000), nrhs=rng.choice([1, 1, 2]),
                    iterations=rng.randint(4, 8))
    if kind == "batch":
        return dict(kind=kind, precision=rng.choice(["fp32", "mixed"]), problems=rng.randint(2, 16), n_min=2048,
                    n_max=32768, picks=rng.randrange(1 << 20))
    if kind == "evaluate":
        return dict(kind=kind, family=family, precision=precision, n=_log(rng, 1000, 20000 if precision == "fp64" else
                                                                           100000),
                    targets=_log(rng, 100, 10000), nrhs=nrhs)
    return dict(kind="direct", kernel=rng.choice(["exp", "matern32", "gauss"]), d=rng.randint(2, 16),
                n=_log(rng, 100, 8192), nrhs=nrhs)


def _problems(case: dict) -> list[tuple[int, int, int]]:
    """(d, n, nrhs) of a batch's problems: n log-uniform, d in 6..12, 1..8
    right-hand sides (a part of the case, not of the seed)."""
    import random
    rng = random.Random(case["picks"])
    return [(rng.randint(6, 12), _log(rng, case["n_min"], case["n_max"]), rng.randint(1, 8))
            for _ in range(case["problems"])]


def _generator(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _sites(n: int, gamma: list[float], g: torch.Generator) -> torch.Tensor:
    u = torch.rand((n, len(gamma)), dtype=torch.float64, device="cuda", generator=g)
    return (2.0 * u - 1.0) * torch.tensor(gamma, dtype=torch.float64, device="cuda")


def _rhs(r: int, n: int, g: torch.Generator) -> torch.Tensor:
    return torch.randn((r, n), dtype=torch.float64, device="cuda", generator=g)


def _inputs(case: dict, seed: int):
    """[(sites, right-hand sides)] of the case's problems, and the targets of
    an evaluation."""
    g = _generator(seed)
    kind = case["kind"]
    if kind == "batch":
        return [(_sites(n, _gamma("inverse_square", d), g), _rhs(r, n, g)) for d, n, r in _problems(case)], None
    if kind == "direct":
        gamma = _gamma("inverse_square", case["d"])
    else:
        f = FAMILIES[case["family"]]
        gamma = _gamma(f["gamma"], f["d"])
    pts, x = _sites(case["n"], gamma, g), _rhs(case["nrhs"], case["n"], g)
    return [(pts, x)], _sites(case["targets"], gamma, g) if kind == "evaluate" else None


def _plan(family: str, precision: str, nrhs: int) -> dwfmm.Plan:
    f = FAMILIES[family]
    return dwfmm.Plan(f["d"], kernel=f["kernel"], gamma=_gamma(f["gamma"], f["d"]), q=f["q"], leaf_size=f["leaf"],
                      precision=precision, max_rhs=nrhs)


class _State:
    pass


def prepare(case: dict, seed: int) -> _State:
    s = _State()
    s.case, s.kind = case, case["kind"]
    problems, targets = _inputs(case, seed)
    s.pts, s.x = problems[0]
    s.y = torch.empty_like(s.x)
    s.wide = case.get("precision") == "fp64"
    if s.kind == "direct":
        return s
    if s.kind == "batch":
        s.xs = [x for _, x in problems]
        s.plans = []
        for (d, _, r), (pts, _) in zip(_problems(case), problems):
            p = dwfmm.Plan(d, kernel="matern32", gamma=_gamma("inverse_square", d), q=5.0, leaf_size=128,
                           precision=case["precision"], max_rhs=r)
            p.tree_build(pts)
            s.plans.append(p)
        s.y = torch.empty(sum(x.numel() for x in s.xs), dtype=torch.float64, device="cuda")
        parts = torch.split(s.y, [x.numel() for x in s.xs])
        s.ys = [p.view_as(x) for p, x in zip(parts, s.xs)]
        s.batch = dwfmm.Batch(s.plans, [x.shape[0] for x in s.xs])
        return s
    s.plan = _plan(case["family"], case["precision"], case["nrhs"])
    if s.kind != "new_sites":
        s.plan.tree_build(s.pts)
    if s.kind == "cg":
        s.stream = torch.cuda.Stream()
    if s.kind == "evaluate":
        s.targets = targets
        s.y = torch.empty((case["nrhs"], targets.shape[0]), dtype=torch.float64, device="cuda")
    return s


def _direct(s: _State) -> None:
    c = s.case
    st = dwfmm.lib().dwfmm_direct_sum_noalloc(
        dwfmm.KERNELS[c["kernel"]], 1.0, s.pts.data_ptr(), c["n"], c["d"], s.pts.stride(0), s.x.data_ptr(),
        s.y.data_ptr(), c["nrhs"], s.x.stride(0), s.y.stride(0), torch.cuda.current_stream().cuda_stream)
    if st != dwfmm.OK:
        raise dwfmm.DwfmmError(st, "direct sum")


def run(s: _State) -> torch.Tensor:
    if s.kind == "matvec":
        s.plan.matvec(s.x, s.y)
    elif s.kind == "new_sites":
        s.plan.tree_build(s.pts)
        s.plan.matvec(s.x, s.y)
    elif s.kind == "cg":
        s.stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s.stream):
            s.plan.cg_begin(LAMBDA, s.x, rtol=1e-12)
            s.plan.cg_step(s.case["iterations"])
            s.plan.cg_result(s.y)
        torch.cuda.current_stream().wait_stream(s.stream)
    elif s.kind == "batch":
        s.batch.matvec(s.xs, s.ys)
    elif s.kind == "evaluate":
        s.plan.evaluate(s.targets, s.x, s.y)
    else:
        _direct(s)
    return s.y if s.wide else s.y.float()


@functools.lru_cache(maxsize=None)
def _counts(family: str, n: int) -> tuple[float, float]:
    """Ordered site pairs of the near field and node pairs of the couplings."""
    plan = _plan(family, "fp32", 1)
    plan.tree_build(_sites(n, _gamma(FAMILIES[family]["gamma"], FAMILIES[family]["d"]), _generator(0)))
    n_x, n_far, n_near, depth = plan.info()
    plan.close()
    return n_near * (n / 2.0 ** depth) ** 2, n_far * float(n_x) ** 2


def _pair_flops(d: int, r: int) -> float:
    """Per ordered pair of a symmetric sum: the kernel value is shared by both
    orders (3d + 4), 2 per right-hand side."""
    return (3 * d + 4) / 2.0 + 2.0 * r


def work(case: dict) -> dict:
    if case["kind"] == "batch":
        # every pair of a problem once, close to what its near field and couplings hold at these sizes
        w = [(8.0 * n * (d + 2 * r), n * n * _pair_flops(d, r)) for d, n, r in _problems(case)]
        return {"bytes": sum(b for b, _ in w), "flops": sum(f for _, f in w)}
    n, r = case["n"], case["nrhs"]
    if case["kind"] == "direct":
        return {"bytes": 8.0 * n * (case["d"] + 2 * r), "flops": n * n * _pair_flops(case["d"], r)}
    d = FAMILIES[case["family"]]["d"]
    if case["kind"] == "evaluate":
        t = case["targets"]
        return {"bytes": 8.0 * (n * (d + r) + t * (d + r)), "flops": float(n) * t * (3 * d + 4 + 2 * r)}
    near, far = _counts(case["family"], n)
    return {"bytes": 8.0 * n * (d + 2 * r), "flops": case.get("iterations", 1) * (near + far) * _pair_flops(d, r)}


# -- the dense sums in float64 ------------------------------------------------

def _dense(kernel: str, targets: torch.Tensor, sites: torch.Tensor, x: torch.Tensor) -> torch.Tensor:
    """(R, nt): sum_j phi(|t - x_j|) x_j, a block of targets at a time."""
    out = torch.empty((x.shape[0], targets.shape[0]), dtype=torch.float64, device=x.device)
    step = max(1, (1 << 28) // sites.shape[0])
    st = sites.t().contiguous()
    for a in range(0, targets.shape[0], step):
        t = targets[a:a + step]
        r2 = torch.zeros((t.shape[0], sites.shape[0]), dtype=torch.float64, device=x.device)
        for k in range(t.shape[1]):
            df = t[:, k:k + 1] - st[k]
            r2.addcmul_(df, df)
        if kernel == "gauss":
            phi = r2.mul_(-0.5).exp_()
        elif kernel == "exp":
            phi = r2.sqrt_().neg_().exp_()
        else:
            r = r2.sqrt_().mul_(math.sqrt(3.0))
            phi = (-r).exp_().mul_(r.add_(1.0))
        out[:, a:a + step] = x @ phi.t()
    return out


def exact(case: dict, seed: int):
    if case["kind"] == "cg":
        # the iterates belong to the compressed operator: a few steps blow its difference from the dense one up
        return None
    if case["kind"] != "batch":
        pairs = float(case["n"]) * case.get("targets", case["n"])
        if pairs > 8e10:
            return None   # a minute and more
    problems, targets = _inputs(case, seed)
    if case["kind"] == "batch":
        return torch.cat([_dense("matern32", pts, pts, x).reshape(-1) for pts, x in problems])
    pts, x = problems[0]
    kernel = case["kernel"] if case["kind"] == "direct" else FAMILIES[case["family"]]["kernel"]
    if case["kind"] == "evaluate":
        return _dense(kernel, targets, pts, x)
    return _dense(kernel, pts, pts, x)
