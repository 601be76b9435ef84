"""The FP64 far field on uneven problems: charges of order 1 in one corner of the
cube and 1e-14 in the opposite one, every step compared with the CPU EIFMM box by
box, so that a weak box has to keep its own digits.

exp(-r^2) on a cube of edge 8 leaves the weak corner to its own charges (the strong
ones are at e^-48 there); 1/r carries the strong ones everywhere.

Tolerances: W, l and f are sums of at most 8 d and 189 d products in FP64 on both
sides, each sum with errors of 189 d 2^-53 (8e-12 at d = 340) of its absolute terms;
these exceed the results by 7 (exp) and 19 (1/r) at level 4, positive charges: 1e-9
for a box or a target.  g: 10 * 189 d 2^-53 of the absolute terms, summed here.
FP32 pairs (tier 4): 2^-46 a product instead."""
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
