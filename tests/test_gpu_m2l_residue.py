"""The FP64 M2L by residues on the tensor cores against the FP64 M2L on the
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
