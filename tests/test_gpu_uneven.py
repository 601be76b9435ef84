"""The FP64 far field on uneven problems: charges of order 1 in one corner of the
cube and 1e-14 in the opposite one, every step compared with the CPU EIFMM box by
box, so that a weak box has to keep its own digits.

exp(-r^2) on a cube of edge 8 leaves the weak corner to its own charges (the strong
ones are at e^-48 there) and the M2L to the FP64 pipes or FP32 pairs; 1/r carries the
strong ones everywhere, and its M2L runs in residues.

Tolerances: W, l and f are sums of at most 8 d and 189 d products in FP64 on both
sides, each sum with errors of 189 d 2^-53 (8e-12 at d = 340) of its absolute terms;
these exceed the results by 7 (exp) and 19 (1/r) at level 4, positive charges: 1e-9
for a box or a target.  g: 10 * 189 d 2^-53 of the absolute terms, summed here.
FP32 pairs (tier 4): 2^-46 a product instead."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1408_0210_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu
DEPTH, N = 4, 4000


@pytest.fixture(scope="module")
def E():
    from paper_1408_0210_gb300 import eifmm
    eifmm.lib()
    return eifmm


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def coords(box, level):
    return [sum(((box >> (3 * i + a)) & 1) << i for i in range(level)) for a in range(3)]


def abs_terms(orc, kern, L, lv, k, W, boxes):
    """sum |T^delta| |W| over the interaction list of every box."""
    d = lv["d"]
    Kd = orc.m2l_operators(kern, L, k, lv)
    delta = np.stack([orc.apply_delta(lv["Gamma"], lv["B"], e) for e in np.eye(d)], 1)
    T, out = {}, {}
    for b in boxes:
        out[b], c = np.zeros(d), coords(b, k)
        for J in orc.interaction_list(k, b):
            if J < 0 or not W[J].any():
                continue
            t = [x - y for x, y in zip(coords(int(J), k), c)]
            slot = t[0] + 3 + 7 * (t[1] + 3) + 49 * (t[2] + 3)
            if slot not in T:
                T[slot] = np.abs(Kd[slot] @ delta)
            out[b] += T[slot] @ np.abs(W[J])
    return out


@pytest.mark.parametrize("kern,L,prec", [("exp_r2", 8.0, "fp64"), ("exp_r2", 8.0, "mixed"), ("inv_r", 1.0, "fp64")])
def test_weak_boxes_keep_their_digits(E, orc, kern, L, prec):
    lv = orc.build_levels(kern, L, DEPTH, 1e-6)
    x = L * np.concatenate([0.25 * wl.uniform_cube(N // 2, 31), 0.75 + 0.25 * wl.uniform_cube(N // 2, 32)])
    s = np.abs(wl.sigma_uniform(N, 1, 33)) + 0.5
    s[N // 2:] *= 1e-14
    f2, dm = orc.eifmm(kern, L, [0, 0, 0], DEPTH, lv, x, x, s, dump=True)
    ops = E.eifmm_ops_load(kern, L, DEPTH, lv)
    ops.plan(4)
    tree = E.eifmm_tree_build(dev(x), None, (0, 0, 0), L, DEPTH, True)
    f = torch.zeros(N, dtype=torch.float64, device="cuda")
    E.eifmm_evaluate(tree, ops, dev(s[:, 0]), f, prec)
    assert (np.abs(f.cpu().numpy() - f2[:, 0]) <= 1e-9 * f2[:, 0]).all()
    for k in range(2, DEPTH + 1):
        a, b = E.eifmm_debug_export(tree, 0, k, lv[k]["d"])[:, 0], dm["W"][k][:, 0]
        assert (np.abs(a - b).max(1) <= 1e-9 * np.abs(b).max(1)).all(), k
    d = lv[DEPTH]["d"]
    W, g = dm["W"][DEPTH][:, 0], E.eifmm_debug_export(tree, 2, DEPTH, d)[:, 0]
    boxes = [int(b) for b in np.flatnonzero(W.any(1))]
    boxes = boxes[:3] + boxes[-3:]  # of the strong corner and of the weak one
    unit = 2.0 ** -53 if prec == "fp64" else 2.0 ** -46
    for b, t in abs_terms(orc, kern, L, lv[DEPTH], DEPTH, W, boxes).items():
        assert t.max() > 0
        assert (np.abs(g[b] - dm["g"][DEPTH][b, 0]) <= 10 * 189 * d * unit * t.max()).all(), b
    # step 6 by its backward error, box by box: A^t lhat = l
    X, Y = lv[DEPTH]["X"], lv[DEPTH]["Y"]
    A = orc.kernel(kern, (X[:, None] - Y[None]).reshape(-1, 3)).reshape(d, d)
    lh, ll = (E.eifmm_debug_export(tree, w, DEPTH, d)[:, 0] for w in (4, 3))
    assert (np.abs(lh @ A - ll).max(1) <= 1e-12 * (np.abs(lh) @ np.abs(A)).max(1)).all()



def test_pair_arithmetic_m2l(E):
    """A steep kernel's M2L in tiers 3 and 4 runs in FP32 pairs: against the FP64 pipes
    (option m2l_fp64) 1e-10 of the leaf level's largest g (a product is good to 2^-47,
    the absolute terms are 7 times the result, 22,000 terms), and not the same bits."""
    x, s = 8.0 * wl.uniform_cube(N, 38), dev(wl.sigma_uniform(N, 1, 39)[:, 0])
    ops = E.eifmm_ops_build("exp_r2", 8.0, DEPTH, 1e-6)
    tree = E.eifmm_tree_build(dev(x), None, (0, 0, 0), 8.0, DEPTH, True)
    d = ops.error_estimate(DEPTH)[1]
    for tier in (3, 4):
        ops.plan(tier)
        g = {}
        for fp64 in (True, False):
            tree.set_option("m2l_fp64", fp64)
            E.eifmm_evaluate(tree, ops, s, torch.zeros(N, dtype=torch.float64, device="cuda"), "mixed")
            g[fp64] = E.eifmm_debug_export(tree, 2, DEPTH, d)
        diff = np.abs(g[True] - g[False]).max()
        assert 0.0 < diff <= 1e-10 * np.abs(g[True]).max()


def ints(a, e):
    """a 2^e as exact integers."""
    return np.array([int(Fraction(float(v)) * 2 ** e) for v in a.ravel()], dtype=object).reshape(a.shape)


# Operators without rounding: Gamma = B = 1 (Delta = 1), K(z) = |z|^2 and nodes on a
# grid, so that T^delta = K^delta is exact.  The exported W then gives g exactly, and
# the residue M2L's error is the rounding of W, for these boxes (even ones and weak
# ones) at most 2^-53 of the largest W of the interaction list for every term, and one
# or two of the sum (each 2^-53 of the absolute terms): together below 2^-51 of that W
# times the row sums of |T|.
@pytest.mark.parametrize("depth,d,weak", [(4, 8, (1.0,)), (4, 17, (1.0,)), (4, 8, (2.0 ** -30,)), (4, 17, (2.0 ** -30,)),
                                          (4, 8, (2.0 ** -55,)), (4, 17, (2.0 ** -55,)),
                                          (5, 17, (2.0 ** -55, 1.0, 2.0 ** -20))])  # several tiles and columns
def test_residue_m2l_is_exact_to_its_rounding(E, orc, depth, d, weak):
    rng = np.random.default_rng(7)
    lv = {}
    for k in range(2, depth + 1):
        p = rng.integers(-128, 128, (2, d, 3)) / 256.0 * 2.0 ** -k
        lv[k] = dict(d=d, X=p[0], Y=p[1], Gamma=np.eye(d), B=np.eye(d), eps_est=1e-6)
    x = np.concatenate([0.25 * wl.uniform_cube(N // 2, 35), 0.75 + 0.25 * wl.uniform_cube(N // 2, 36)])
    R = len(weak)
    s = wl.sigma_uniform(N, R, 37)
    s[N // 2:] *= np.array(weak)
    ops = E.eifmm_ops_load("quad", 1.0, depth, lv)
    tree = E.eifmm_tree_build(dev(x), None, (0, 0, 0), 1.0, depth, True)
    f = torch.zeros(R, N, dtype=torch.float64, device="cuda")
    E.eifmm_evaluate(tree, ops, dev(s.T).T if R > 1 else dev(s[:, 0]), f.T if R > 1 else f[0], "fp64")
    for k in (2, depth):
        Ws, gs = (E.eifmm_debug_export(tree, w, k, d, R) for w in (0, 2))
        Kd = orc.m2l_operators("quad", 1.0, k, lv[k])
        boxes = np.flatnonzero(Ws[:, 0].any(1))
        for r in range(R):
            W, g = Ws[:, r], gs[:, r]
            for b in (int(boxes[0]), int(boxes[1]), int(boxes[-2]), int(boxes[-1])):
                total, largest, rows = np.zeros(d, dtype=object), 0.0, np.zeros(d)
                for J in orc.interaction_list(k, b):
                    if J < 0 or not W[J].any():
                        continue
                    t = [p - q for p, q in zip(coords(int(J), k), coords(b, k))]
                    T = Kd[t[0] + 3 + 7 * (t[1] + 3) + 49 * (t[2] + 3)]
                    total += ints(T, 60) @ ints(W[J], 200)
                    largest, rows = max(largest, np.abs(W[J]).max()), rows + np.abs(T).sum(1)
                err = [abs(float(Fraction(int(v), 2 ** 260) - Fraction(float(w)))) for v, w in zip(total, g[b])]
                assert (np.array(err) <= 2.0 ** -51 * largest * rows).all(), (k, r, b)


# A kernel's weak boxes with few sources run on the FP64 pipes, those of a crowded
# tile take a second residue part, boxes beyond 2^-60 the pipes again, boxes up to the
# limit neither: over clustered points no group's error exceeds that of the M2L on the
# FP64 pipes (option m2l_fp64), against exact sums as above.
@pytest.mark.parametrize("d", [8, 17, 64])
@pytest.mark.parametrize("points,weak", [("mixture", 1.0), ("corners", 2.0 ** -6), ("corners", 2.0 ** -12),
                                         ("corners", 2.0 ** -70)])
def test_no_less_precise_than_the_fp64_pipes(E, orc, d, points, weak):
    rng = np.random.default_rng(8)
    lv = {}
    for k in range(2, DEPTH + 1):
        p = rng.integers(-128, 128, (2, d, 3)) / 256.0 * 2.0 ** -k
        lv[k] = dict(d=d, X=p[0], Y=p[1], Gamma=np.eye(d), B=np.eye(d), eps_est=1e-6)
    if points == "mixture":
        n = 40000
        x, s = wl.gaussian_mixture(n, 3), wl.sigma_uniform(n, 1, 40)[:, 0]
    else:  # the strong corner, a crowded weak one, single points between
        n = N
        x = np.concatenate([0.25 * wl.uniform_cube(n // 2, 41), 0.75 + 0.25 * wl.uniform_cube(n // 2 - 40, 42),
                            0.3 + 0.4 * wl.uniform_cube(40, 43)])
        s = wl.sigma_uniform(n, 1, 44)[:, 0]
        s[n // 2:] *= weak
    ops = E.eifmm_ops_load("quad", 1.0, DEPTH, lv)
    g = {}
    for fp64 in (True, False):
        tree = E.eifmm_tree_build(dev(x), None, (0, 0, 0), 1.0, DEPTH, True)
        tree.set_option("m2l_fp64", fp64)
        E.eifmm_evaluate(tree, ops, dev(s), torch.zeros(n, dtype=torch.float64, device="cuda"), "fp64")
        W, g[fp64] = (E.eifmm_debug_export(tree, w, DEPTH, d)[:, 0] for w in (0, 2))
    Kd = orc.m2l_operators("quad", 1.0, DEPTH, lv[DEPTH]).astype(np.longdouble)
    err = {}  # binary exponents below the level's largest -> [(pipes, residues)]
    for b in rng.choice(8 ** DEPTH, 400, replace=False):
        total, largest, rows = np.zeros(d, np.longdouble), 0.0, np.zeros(d)
        for J in orc.interaction_list(DEPTH, int(b)):
            if J >= 0 and W[J].any():
                t = [p - q for p, q in zip(coords(int(J), DEPTH), coords(int(b), DEPTH))]
                T = Kd[t[0] + 3 + 7 * (t[1] + 3) + 49 * (t[2] + 3)]
                total += T @ W[J].astype(np.longdouble)
                largest, rows = max(largest, np.abs(W[J]).max()), rows + np.abs(T).sum(1).astype(float)
        if largest > 0.0:
            e = [np.sqrt((((g[f][b] - total) / (largest * rows)).astype(float) ** 2).mean()) for f in (True, False)]
            err.setdefault(int(np.log2(np.abs(W).max() / largest)) // 3, []).append(e)
    assert sum(len(e) for e in err.values()) >= 60
    for below, e in err.items():
        pipes, residues = np.mean(e, axis=0)
        # single boxes scatter by a factor; 20 are a mean.  1.1 where the pipes run
        assert len(e) < 20 or residues <= 1.1 * pipes, (below, len(e), pipes, residues)
