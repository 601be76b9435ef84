"""The work that users of this library have it do, as cases that can be timed.

A case is one pass through the public entry points on inputs that are already
on the GPU: an evaluation f_i = sum_j sigma_j K(x_i - y_j) on a tree and an
operator set that the program keeps, a batch of such evaluations, or the
Morton sort of a point set.  Points are the test sets of the paper's Section
5.2 (cube, sphere) and the clustered mixture of `workloads.gaussian_mixture`;
sizes, tolerances and depths are those of the benchmark and the tests.  One
operator set serves every state of a kernel, depth and tolerance, as it does
in a program: it depends on none of the points.
"""
from __future__ import annotations

import math

import torch

from paper_1408_0210_gb300 import eifmm as E
from paper_1408_0210_gb300 import workloads as wl

LO, SIDE = (0.0, 0.0, 0.0), 1.0
# EIM ranks of the operator sets (1/r; the config-3 kernel at 1e-6 is about 280)
RANK = {1e-4: 126, 1e-5: 161, 1e-6: 193, 1e-7: 256}
EXACT_PAIRS = 1.2e11  # about the pairs that torch sums in FP64 within 20 s


def _case(name, **more):
    c = dict(do="evaluate", kernel="inv_r", points="cube", n=1 << 20, targets=0, depth=5, eps=1e-4, rhs=1,
             prec="mixed", normal=False)
    c.update(more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small problem inside a larger program: launches and latency
        _case("mixed_e5_3k", n=3000, depth=3, eps=1e-5),
        # a reference solution in double precision on a small set
        _case("fp64_e6_4k", n=4096, depth=3, eps=1e-6, prec="fp64"),
        # the headline: single-precision accuracy on a million points, every time step
        _case("mixed_e4_1m"),
        # the same size where six digits are asked for: the FP64 far field
        _case("mixed_e6_1m", eps=1e-6),
        # seven digits: FP64 near field too, the largest rank
        _case("mixed_e7_1m", eps=1e-7),
        # double precision throughout, the comparison run of every accuracy study
        _case("fp64_e4_1m", prec="fp64"),
        # many charges on one geometry (block solvers, several fields), odd count
        _case("mixed_e6_262k_rhs7", n=262144, eps=1e-6, rhs=7),
        # many uneven independent problems in one call
        _case("batch_e6_12", do="batch", n=131072, problems=12, n_min=16384, eps=1e-6),
        # clustered points and an anisotropic kernel without a closed-form expansion
        _case("config3_e6_1m", kernel="config3", points="mixture", eps=1e-6),
        # points on a surface: a deep tree, most of whose leaves are empty
        _case("sphere_e4_1m", points="sphere", n=992046, depth=7),
        # the largest: 16 million points, five digits, charges N(0, 1)
        _case("mixed_e5_16m", n=1 << 24, depth=7, eps=1e-5, normal=True),
        # moving points: the Morton sort of every time step, into kept arrays
        _case("sort_1m", do="sort", n=1 << 20, depth=5),
    ]


def _depth(n):
    """About 32 points a leaf, as the benchmark chooses it."""
    return min(5, max(3, math.ceil(math.log(n / 32, 8))))


def draw(rng):
    n = int(round(math.exp(rng.uniform(math.log(2000), math.log(1 << 20)))))
    depth = _depth(n)
    kind = rng.random()
    if kind < 0.15:
        return _case(None, do="sort", points=rng.choice(["cube", "mixture", "sphere"]), n=n, depth=rng.randint(3, 7))
    if kind < 0.25:
        n = min(n, 131072)
        return _case(None, do="batch", n=n, n_min=max(1000, n // 8), problems=rng.randint(2, 12),
                     eps=rng.choice([1e-4, 1e-5, 1e-6]), prec="mixed")
    prec = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    eps = rng.choice([1e-4, 1e-5, 1e-6, 1e-7])
    # FP64 far fields take their time in proportion to the right-hand sides
    most = 16 if prec == "mixed" and eps >= 1e-5 else 8 if depth < 5 else 1 if prec == "fp64" else 3
    rhs = rng.choice([1, 1, rng.randint(1, most)])
    points = rng.choice(["cube", "cube", "mixture", "sphere"])
    kernel = "config3" if points == "mixture" and eps == 1e-6 and rhs == 1 and rng.random() < 0.5 else "inv_r"
    if points == "sphere":  # a surface fills few leaves: one level deeper keeps them small
        depth = min(6, depth + 1) if rhs == 1 and eps == 1e-4 and prec == "mixed" else depth
    if points == "mixture" and n > 300000 and prec == "fp64":
        n //= 4
    targets = rng.choice([0, 0, 0, n // rng.randint(1, 5) + 1])
    return _case(None, kernel=kernel, points=points, n=n, targets=targets, depth=depth, eps=eps, rhs=rhs, prec=prec,
                 normal=rng.random() < 0.5)


# ------------------------------------------------------------------ inputs --
def _generator(seed):
    return torch.Generator("cuda").manual_seed(int(seed))


def _points(kind, n, g):
    o = dict(dtype=torch.float64, device="cuda", generator=g)
    if kind == "cube":
        return torch.rand(n, 3, **o)
    if kind == "sphere":
        v = torch.randn(n, 3, **o)
        return (0.5 + 0.5 * v / v.norm(dim=1, keepdim=True)).clamp_(0.0, 1.0)
    centres = 0.2 + 0.6 * torch.rand(8, 3, **o)
    which = torch.randint(0, 8, (n,), device="cuda", generator=g)
    return (centres[which] + 0.05 * torch.randn(n, 3, **o)).clamp_(0.0, 1.0)


def _sigma(n, rhs, normal, g):
    """Column-major n x rhs charges (a vector for one column)."""
    o = dict(dtype=torch.float64, device="cuda", generator=g)
    s = torch.randn(rhs, n, **o) if normal else 2.0 * torch.rand(rhs, n, **o) - 1.0
    return s[0] if rhs == 1 else s.T


def _inputs(case, seed):
    """[(sources, targets or None, sigma)]: one for an evaluation, several for a batch."""
    g = _generator(seed)
    if case["do"] != "batch":
        x = _points(case["points"], case["n"], g)
        y = _points(case["points"], case["targets"], g) if case["targets"] else None
        return [(x, y, _sigma(case["n"], case["rhs"], case["normal"], g))]
    # the sizes are part of the case: they do not change with the seed
    sizes = wl.batch_sizes(case["problems"], case["n_min"], case["n"], 40)
    return [(_points(case["points"], n, g), None, _sigma(n, 1, case["normal"], g)) for n in sizes]


_operators = {}  # the operator set in use


def _ops(case, depth):
    key = (case["kernel"], depth, case["eps"])
    if key not in _operators:
        _operators.clear()
        _operators[key] = E.eifmm_ops_build(case["kernel"], SIDE, depth, case["eps"])
    return _operators[key]


def prepare(case, seed):
    if case["do"] == "sort":
        n, leaves = case["n"], 8 ** case["depth"]
        new = lambda m: torch.empty(m, dtype=torch.int32, device="cuda")  # noqa: E731
        return dict(case=case, x=_points(case["points"], n, _generator(seed)), out=(new(n), new(n), new(leaves + 1)))
    items = _inputs(case, seed)
    depths = [_depth(len(x)) if case["do"] == "batch" else case["depth"] for x, _, _ in items]
    ops = _ops(case, max(depths))
    trees = [E.eifmm_tree_build(x, y, LO, SIDE, d, y is None) for (x, y, _), d in zip(items, depths)]
    fs = []
    for x, y, _ in items:
        m = len(x) if y is None else len(y)
        f = torch.zeros(case["rhs"], m, dtype=torch.float64, device="cuda")
        fs.append(f[0] if case["rhs"] == 1 else f.T)
    return dict(case=case, ops=ops, trees=trees, points=items, sigma=[s for _, _, s in items], f=fs)


def run(state):
    case, stream = state["case"], torch.cuda.current_stream()
    if case["do"] == "sort":
        return E.eifmm_tree_sort_static(state["x"], LO, SIDE, case["depth"], *state["out"], stream=stream)
    if case["do"] == "batch":
        E.eifmm_evaluate_batched(state["trees"], state["sigma"], state["f"], state["ops"], case["prec"], stream)
        return state["f"]
    E.eifmm_evaluate(state["trees"][0], state["ops"], state["sigma"][0], state["f"][0], case["prec"], stream)
    return state["f"][0]


# -------------------------------------------------------------------- work --
def _far_pairs(k, points):
    """Pairs of boxes in the interaction lists of level k (a surface fills about one layer of the boxes)."""
    n = 1 << k
    a = sum(min(n - 1, 2 * (i >> 1) + 3) - max(0, 2 * (i >> 1) - 2) + 1 for i in range(n))
    b = sum(min(n - 1, i + 1) - max(0, i - 1) + 1 for i in range(n))
    return (a ** 3 - b ** 3) if points != "sphere" else 3.0 * n * n * 27


def _evaluate_work(case, n, m, depth):
    """Two flops a product; a kernel value counts 8 flops (the distance and 1/r)."""
    d, rhs = (280 if case["kernel"] == "config3" else RANK[case["eps"]]), case["rhs"]
    leaves = 8 ** depth if case["points"] != "sphere" else 3 * 4 ** depth
    neighbours = 27 if case["points"] != "sphere" else 9
    near = float(m) * max(1.0, neighbours * n / leaves)
    flops = sum(2.0 * d * d * rhs * _far_pairs(k, case["points"]) for k in range(2, depth + 1))
    flops += sum(4.0 * d * d * rhs * leaves / 8 ** k for k in range(depth - 1)) + 2.0 * d * d * rhs * leaves
    flops += (float(n) + m) * d * (8 + 2 * rhs) + near * (8 + 2 * rhs)
    size = 8 if case["prec"] == "fp64" or case["eps"] < 1e-5 else 4
    operators = (depth - 1) * 316.0 * d * d * size
    return 24.0 * (n + (m if case["targets"] else 0)) + 8.0 * rhs * (n + m), operators, flops


def work(case):
    if case["do"] == "sort":  # points in; keys, permutation and leaf offsets out
        return {"bytes": 24.0 * case["n"] + 8.0 * case["n"] + 4.0 * (8 ** case["depth"] + 1), "flops": 6.0 * case["n"]}
    if case["do"] == "batch":
        w = [_evaluate_work(case, n, n, _depth(n))
             for n in wl.batch_sizes(case["problems"], case["n_min"], case["n"], 40)]
        # the problems share one operator set
        return {"bytes": sum(b for b, _, _ in w) + max(o for _, o, _ in w), "flops": sum(f for _, _, f in w)}
    b, o, f = _evaluate_work(case, case["n"], case["targets"] or case["n"], case["depth"])
    return {"bytes": b + o, "flops": f}


# ------------------------------------------------------------------- exact --
def _direct(x, y, s):
    """sum_j s_j / |t_i - x_j| in FP64, the pairs of coinciding points left out when targets are the sources."""
    t = x if y is None else y
    s2 = s[:, None] if s.dim() == 1 else s
    f = torch.empty(len(t), s2.shape[1], dtype=torch.float64, device=x.device)
    step = max(1, (1 << 27) // len(x))
    for a in range(0, len(t), step):
        b = min(len(t), a + step)
        r2 = torch.zeros(b - a, len(x), dtype=torch.float64, device=x.device)
        for k in range(3):
            r2 += (t[a:b, k:k + 1] - x[None, :, k]).square_()
        if y is None:
            r2[torch.arange(b - a, device=x.device), torch.arange(a, b, device=x.device)] = math.inf
        f[a:b] = r2.rsqrt_() @ s2
    return f[:, 0] if s.dim() == 1 else f.T.contiguous().T


def exact(case, seed):
    """The direct sum.  None for the sort (whole numbers), for sizes whose direct sum takes too long, and for the
    config-3 kernel, whose boxes are not well separated along y: the method itself stays near 1e-1 of the sum."""
    if case["do"] == "sort" or case["kernel"] != "inv_r":
        return None
    if case["do"] == "batch":
        sizes = wl.batch_sizes(case["problems"], case["n_min"], case["n"], 40)
        if sum(float(n) * n for n in sizes) > EXACT_PAIRS:
            return None
        return [_direct(x, y, s) for x, y, s in _inputs(case, seed)]
    if float(case["n"]) * (case["targets"] or case["n"]) > EXACT_PAIRS:
        return None
    (x, y, s), = _inputs(case, seed)
    return _direct(x, y, s)
