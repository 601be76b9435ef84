"""The FP64 point kernels of 1/r and of config-3 on integer coordinates (P2M, L2P,
near field) against extended-precision sums over the same points, coefficients and nodes.

Tolerance: a value is within 2 ulp (1/r: 0.5 from its rounding, the rest covers
the rounding of coordinates to 2^-62 L and of the leaf centre; config-3 with its
exponential: 4), a sum of n terms
adds at most n 2^-53 of the sum of magnitudes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1408_0210_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def E():
    from paper_1408_0210_gb300 import eifmm
    eifmm.lib()
    return eifmm


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def kernel(kern, t, s):
    d = [t[:, k:k + 1].astype(LD) - s[None, :, k].astype(LD) for k in range(3)]
    r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    with np.errstate(divide="ignore"):
        K = 1 / np.sqrt(r2)
        if kern == "config3":
            # the library's 0.01 and 1e-3 are the doubles
            K = K * np.exp(-np.sqrt(r2)) + 1 / np.sqrt(d[0] * d[0] + LD(0.01) * d[1] * d[1] + d[2] * d[2] + LD(1e-3))
        return np.where(r2 > 0, K, LD(0))


def points(n, lo, L, tiny, seed):
    """Uniform points and a cluster of size `tiny` at the corner lo, where the
    coordinates have more bits than the integers (and one crowded leaf)."""
    x = wl.uniform_cube(n, seed)
    m = n // 3
    x[:m] = tiny * x[:m]
    return np.array(lo) + L * x


# several passes over targets (more than 128 in a leaf) and sources (more than
# 512 staged); every number of columns per kernel value and remainders; a
# corner and a side that are no powers of two; points too close for integers
CASES = [("inv_r", 1500, (0.0, 0.0, 0.0), 1.0, 2, 1, 0.05, False), ("inv_r", 900, (0.0, 0.0, 0.0), 1.0, 3, 3, 1e-13, False),
         ("inv_r", 700, (-0.3, 10.7, 1e-3), 3.7, 2, 5, 1e-6, True), ("inv_r", 400, (0.0, 0.0, 0.0), 1.0, 4, 9, 0.2, True),
         ("inv_r", 300, (0.0, 0.0, 0.0), 2.0 ** -40, 2, 1, 1e-9, False),
         ("config3", 900, (0.0, 0.0, 0.0), 1.0, 3, 1, 1e-7, False),
         ("config3", 500, (-0.3, 10.7, 1e-3), 3.7, 2, 3, 0.05, True),
         ("config3", 300, (0.0, 0.0, 0.0), 2.0 ** -6, 2, 1, 0.1, False)]  # too small a cube for its integers


@pytest.mark.parametrize("kern,n,lo,L,depth,R,tiny,two", CASES)
def test_point_kernels(E, kern, n, lo, L, depth, R, tiny, two):
    d_max = 67
    x = points(n, lo, L, tiny, 51)
    y = points(n // 2, lo, L, tiny, 52) if two else x
    s = wl.sigma_uniform(n, R, 53)
    levels = {}
    for k in range(2, depth + 1):
        X, Y = E.eifmm_training_sets(k, L)
        levels[k] = E.eifmm_eim_build(kern, X, Y, 1e-9, d_max)
    ops = E.eifmm_ops_load(kern, L, depth, levels)
    src = dev(x)
    tree = E.eifmm_tree_build(src, dev(y) if two else None, lo, L, depth, not two)
    f = torch.zeros(R, len(y), dtype=torch.float64, device="cuda").T
    E.eifmm_evaluate(tree, ops, dev(s.T).T, f, "fp64")
    torch.cuda.synchronize()
    d, X = levels[depth]["d"], levels[depth]["X"]
    W = E.eifmm_debug_export(tree, 0, depth, d, R)
    lh = E.eifmm_debug_export(tree, 4, depth, d, R)
    far, near = E.eifmm_debug_export(tree, 5, 0, 0, R), E.eifmm_debug_export(tree, 6, 0, 0, R)
    w = L * 2.0 ** -depth
    cell = lambda p: np.clip(np.floor((p - np.array(lo)) / w), 0, 2 ** depth - 1).astype(int)  # noqa: E731
    cx, cy = cell(x), cell(y)
    # the library's leaf centre: lo + (2 c + 1) w / 2 in one fused operation
    centre = lambda c: (np.array(lo).astype(LD) + (2 * c + 1).astype(LD) * LD(w / 2)).astype(np.float64)  # noqa: E731
    u = 2.0 ** -53
    ulps = 8 if kern == "config3" else 4  # in units of 2^-53 of a value
    key = lambda c: sum(((int(c[a]) >> b) & 1) << (3 * b + a) for a in range(3) for b in range(depth))  # noqa: E731
    for c in np.unique(cx, axis=0):  # P2M
        i = np.flatnonzero((cx == c).all(1))
        z = x[i] - centre(c)
        K = kernel(kern, X, z)
        ref, mag = K @ s[i].astype(LD), K @ np.abs(s[i]).astype(LD)
        assert (np.abs(W[key(c)].T - ref) <= (len(i) + ulps) * u * mag).all()
    for c in np.unique(cy, axis=0):  # L2P and the near field
        i = np.flatnonzero((cy == c).all(1))
        z = y[i] - centre(c)
        K, v = kernel(kern, z, X), lh[key(c)].T.astype(LD)
        assert (np.abs(far[i] - K @ v) <= (d + ulps) * u * (K @ np.abs(v))).all()
        j = np.flatnonzero((np.abs(cx - c) <= 1).all(1))
        K = kernel(kern, y[i], x[j])
        ref, mag = K @ s[j].astype(LD), K @ np.abs(s[j]).astype(LD)
        assert (np.abs(near[i] - ref) <= (len(j) + ulps) * u * mag).all()


# From depth 7 on the nearest nodes lie closer than the integers of box-relative
# coordinates reach (L / 64 here): one warp takes both forms.
@pytest.mark.parametrize("kern", ["inv_r", "config3"])
def test_point_kernels_on_a_deep_tree(E, kern):
    test_point_kernels(E, kern, 300, (0.0, 0.0, 0.0), 1.0, 7, 1, 0.02, False)
