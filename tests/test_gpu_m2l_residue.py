"""The FP64 products by residues on the tensor cores: the M2L against the one on the
FP64 pipes (option m2l_fp64), at the edges of its tiles.

Tolerance: both sum n = 189 d products.  The FP64 kernel's rounding is at most
n 2^-53 sum |T||W| and the largest entry of g is at least 1/40 of the largest
sum |T||W| for these operators and random charges (measured ratios are below
10), so relative to it the two may differ by 40 * 189 d 2^-53; the residue sum
is exact and its operands' rounding (2^-54 of the largest entry of a row, 2^-59
of the largest W) lies far below."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1408_0210_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    from paper_1408_0210_gb300 import eifmm
    eifmm.lib()
    return eifmm


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# d at the smallest rank that takes the tensor cores, at one and two k-steps,
# around one full tile of columns (256) and beyond it; depth 2 and 3 have class
# grids smaller than a tile; three columns; depth 6 splits its scratch in slabs
CASES = [("inv_r", 2, 1e-12, 8, 1), ("inv_r", 3, 1e-12, 16, 3), ("inv_r", 4, 1e-12, 17, 1),
         ("inv_r", 3, 1e-12, 97, 2), ("inv_r", 4, 1e-12, 128, 1), ("inv_r", 3, 1e-12, 255, 1),
         ("inv_r", 3, 1e-12, 257, 2), ("inv_r", 2, 1e-12, 300, 1), ("exp_r2", 4, 1e-6, 512, 1),
         ("inv_r", 5, 1e-12, 40, 1), ("inv_r", 6, 1e-12, 160, 1)]


@pytest.mark.parametrize("kern,depth,eps,d_max,R", CASES)
def test_residue_m2l_matches_fp64(E, kern, depth, eps, d_max, R):
    n = 4000
    x = np.concatenate([wl.uniform_cube(n - 500, 31), 0.02 * wl.uniform_cube(500, 32)])  # one dense corner
    s = wl.sigma_uniform(n, R, 33) * np.logspace(0, -6, R)  # columns of other magnitudes
    ops = E.eifmm_ops_build(kern, 1.0, depth, eps, d_max)
    tree = E.eifmm_tree_build(dev(x), None, (0, 0, 0), 1.0, depth, True)
    sd = dev(s.T).T if R > 1 else dev(s[:, 0])
    g = {}
    for fp64 in (True, False):
        tree.set_option("m2l_fp64", fp64)
        f = torch.zeros(R, n, dtype=torch.float64, device="cuda").T if R > 1 else torch.zeros(n, dtype=torch.float64, device="cuda")
        E.eifmm_evaluate(tree, ops, sd, f, "fp64")
        torch.cuda.synchronize()
        g[fp64] = {k: E.eifmm_debug_export(tree, 2, k, ops.error_estimate(k)[1], R) for k in range(2, depth + 1)}
    for k in range(2, depth + 1):
        a, b = g[False][k], g[True][k]
        tol = 40 * 189 * ops.error_estimate(k)[1] * 2.0 ** -53
        for r in range(R):
            assert np.abs(a[:, r] - b[:, r]).max() <= tol * np.abs(b[:, r]).max(), (k, r)


def test_residue_m2l_extreme_scales(E):
    """Charges of any finite magnitude, and a column of zeros."""
    n, depth = 3000, 3
    x = wl.uniform_cube(n, 34)
    s = wl.sigma_uniform(n, 1, 35)[:, 0]
    ops = E.eifmm_ops_build("inv_r", 1.0, depth, 1e-6)
    tree = E.eifmm_tree_build(dev(x), None, (0, 0, 0), 1.0, depth, True)
    out = {}
    for scale in (1.0, 2.0 ** 900, 2.0 ** -900, 0.0):
        f = torch.ones(n, dtype=torch.float64, device="cuda")
        E.eifmm_evaluate(tree, ops, dev(s * scale), f, "fp64")
        out[scale] = f.cpu().numpy()
    assert not out[0.0].any()
    for scale in (2.0 ** 900, 2.0 ** -900):  # a power of two changes no mantissa
        assert np.array_equal(out[scale], out[1.0] * scale)


# M2M, L2L and Delta^t by residues: ranks that differ from level to level, with
# remainders of a k-step and of a column tile, one and two column tiles, several
# columns.  Against the CPU EIFMM of the same levels: both carry FP64 rounding
# through the chain (1e-12, as for the whole FP64 path; at eps 1e-8 the sums of
# 189 d products of operators with kappa 7e3 add 189 d 2^-53 10 = 6e-11).
@pytest.mark.parametrize("eps,ranks,R,tol", [(1e-6, (70, 129, 193), 1, 1e-12), (1e-6, (193, 65, 8), 3, 1e-12),
                                             (1e-8, (270, 300, 265), 1, 1e-10)])
def test_residue_transfers_match_the_oracle(E, eps, ranks, R, tol):
    import oracle as orc
    depth, n = 4, 5000
    x = wl.uniform_cube(n, 41)
    s = wl.sigma_uniform(n, R, 42)
    lv = {}
    for k, d in zip(range(2, depth + 1), ranks):
        e = orc.eim("inv_r", orc.train_x(k), orc.train_y(k), eps)
        d = min(d, e["d"])
        lv[k] = dict(d=d, X=e["X"][:d], Y=e["Y"][:d], Gamma=np.ascontiguousarray(e["Gamma"][:d, :d]),
                     B=np.ascontiguousarray(e["B"][:d, :d]), eps_est=eps)
    f2, dm = orc.eifmm("inv_r", 1.0, [0, 0, 0], depth, lv, x, x, s, dump=True)
    ops = E.eifmm_ops_load("inv_r", 1.0, depth, lv)
    tree = E.eifmm_tree_build(dev(x), None, (0, 0, 0), 1.0, depth, True)
    f = torch.zeros(R, n, dtype=torch.float64, device="cuda").T
    E.eifmm_evaluate(tree, ops, dev(s.T).T, f, "fp64")
    torch.cuda.synchronize()
    rel = lambda a, b: float(np.abs(a - np.asarray(b).reshape(a.shape)).max() / np.abs(b).max())  # noqa: E731
    for k in range(2, depth + 1):
        assert rel(E.eifmm_debug_export(tree, 0, k, lv[k]["d"], R), dm["W"][k]) <= tol, k
        assert rel(E.eifmm_debug_export(tree, 3, k, lv[k]["d"], R), dm["l"][k]) <= tol, k
    # Delta^t l: backward error, A^t lhat = l
    A = 1.0 / np.linalg.norm(lv[depth]["X"][:, None] - lv[depth]["Y"][None], axis=-1)
    lh = E.eifmm_debug_export(tree, 4, depth, lv[depth]["d"], R)
    ll = E.eifmm_debug_export(tree, 3, depth, lv[depth]["d"], R)
    assert np.abs(lh @ A - ll).max() <= 1e-12 * (np.abs(lh) @ A).max()
    assert rel(E.eifmm_debug_export(tree, 5, depth, 0, R), dm["f_far"]) <= tol
    assert rel(f.cpu().numpy(), f2) <= tol
