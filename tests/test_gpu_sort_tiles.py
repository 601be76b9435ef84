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


def reference(x, depth):
    side = 1 << depth
    c = np.clip((x * side).astype(np.int64), 0, side - 1)
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
