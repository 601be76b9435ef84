"""Bin/sort at the edges of its tiles (2,048 keys) and for every number of digit
passes (depths 2 to 9: 6 to 27 key bits in 1 to 4 passes): keys, order and leaf
offsets are whole numbers and equal a stable sort on the host."""
import numpy as np
import pytest

from paper_1408_0210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1408_0210_gb300 import build, eifmm
    build.build()
    eifmm.lib()
    return eifmm


def reference(x, depth, lo=(0.0, 0.0, 0.0), L=1.0):
    side = 1 << depth
    c = np.clip(((x - np.array(lo)) * (side / L)).astype(np.int64), 0, side - 1)
    key = np.zeros(len(x), dtype=np.int64)
    for b in range(depth):
        for a in range(3):
            key |= ((c[:, a] >> b) & 1) << (3 * b + a)
    perm = np.argsort(key, kind="stable")
    return key[perm], perm, np.concatenate([[0], np.cumsum(np.bincount(key, minlength=8 ** depth))])


@pytest.mark.parametrize("n", [1, 31, 2047, 2048, 2049, 6000, 1 << 20])
@pytest.mark.parametrize("depth", [2, 3, 5, 6, 8])
def test_sort(E, n, depth):
    x = wl.gaussian_mixture(n, n + depth) if n % 2 else wl.uniform_cube(n, n + depth)
    if n > 40:
        x[17:40] = x[17]  # ties keep their order
        x[3] = [1.0, 0.0, 1.0]
    keys, perm, off = reference(x, depth)
    xd = torch.from_numpy(x).cuda()
    ks, ps, os_ = (a.cpu().numpy() for a in E.eifmm_tree_sort_static(xd, (0, 0, 0), 1.0, depth))
    tk, tp, to = E.eifmm_tree_build(xd, None, (0, 0, 0), 1.0, depth, True).export(0)
    for got in ((ks.view(np.uint32), ps, os_), (tk, tp, to)):
        np.testing.assert_array_equal(got[0], keys)
        np.testing.assert_array_equal(got[1], perm)
        np.testing.assert_array_equal(got[2], off)


def test_sort_of_four_passes(E):
    """A depth whose leaf offsets are too many to compare at every size: keys and order alone."""
    depth = 9
    x = wl.gaussian_mixture(5001, depth)
    side = 1 << depth
    xd = torch.from_numpy(x).cuda()
    ks, ps, _ = (a.cpu().numpy() for a in E.eifmm_tree_sort_static(xd, (0, 0, 0), 1.0, depth))
    c = np.minimum((x * side).astype(np.int64), side - 1)
    key = sum(((c[:, a] >> b) & 1) << (3 * b + a) for a in range(3) for b in range(depth))
    perm = np.argsort(key, kind="stable")
    np.testing.assert_array_equal(ps, perm)
    np.testing.assert_array_equal(ks.view(np.uint32), key[perm])


@pytest.mark.parametrize("lo,L", [((0.0, 0.0, 0.0), 0.75), ((-0.5, -0.0, 2.0), 4.0), ((-0.3, 10.7, 0.001), 3.7),
                                  ((0.0, 0.0, 0.0), 2.0 ** -700), ((-1.0, -2.0, -3.0), 2.0 ** 20 / 3)])
def test_keys_of_general_cubes(E, lo, L):
    depth, n = 6, 5000
    x = np.array(lo) + L * wl.uniform_cube(n, 9)
    x[:4] = [lo, [a + L for a in lo], [lo[0] + L / 2, lo[1], lo[2] + L / 64], [-0.0 if a == 0 else a for a in lo]]
    x = np.clip(x, np.array(lo), np.array(lo) + L)
    keys, perm, off = reference(x, depth, lo, L)
    ks, ps, os_ = (a.cpu().numpy() for a in E.eifmm_tree_sort_static(torch.from_numpy(x).cuda(), lo, L, depth))
    np.testing.assert_array_equal(ks.view(np.uint32), keys)
    np.testing.assert_array_equal(ps, perm)
    np.testing.assert_array_equal(os_, off)
    for bad in (np.nan, -np.nan, np.inf, -np.inf, np.nextafter(lo[1], -np.inf), np.nextafter(lo[1] + L, np.inf)):
        y = x.copy()
        y[77, 1] = bad
        with pytest.raises(E.EifmmError, match="outside"):
            E.eifmm_tree_sort_static(torch.from_numpy(y).cuda(), lo, L, depth)
