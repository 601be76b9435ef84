"""Trees most of whose leaves are empty: the sparse P2M, M2L and step 6 of the FP32
tiers against the dense ones (targets in every leaf) for the same sources."""
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


# a surface, a few points in one corner (classes without an active box, tiles
# with one row), and one level below the threshold only; tiers 0 and 1
@pytest.mark.parametrize("kind,n,depth,tier", [("sphere", 20000, 6, 0), ("corner", 37, 5, 0), ("sphere", 3000, 5, 0),
                                               ("sphere", 3000, 5, 1)])
def test_sparse_matches_dense(E, kind, n, depth, tier):
    x = wl.sphere_surface(n, 61) if kind == "sphere" else 0.04 * wl.uniform_cube(n, 61)
    y = np.clip(x + 1e-4 * wl.uniform_cube(n, 62), 0.0, 1.0)
    m = 2 ** depth
    c = (np.arange(m) + 0.5) / m
    fill = np.stack(np.meshgrid(c, c, c, indexing="ij"), -1).reshape(-1, 3)  # a target in every leaf
    s = dev(wl.sigma_uniform(n, 1, 63)[:, 0])
    ops = E.eifmm_ops_build("inv_r", 1.0, depth, 1e-4)
    assert ops.plan(tier) == tier
    out = {}
    for name, t in (("sparse", y), ("dense", np.concatenate([y, fill]))):
        tree = E.eifmm_tree_build(dev(x), dev(t), (0, 0, 0), 1.0, depth, False)
        f = torch.zeros(len(t), dtype=torch.float64, device="cuda")
        for _ in range(2):  # rows left out stay zero from call to call
            E.eifmm_evaluate(tree, ops, s, f, "mixed")
        far = E.eifmm_debug_export(tree, 5, 0, 0)[:n, 0]
        d = ops.error_estimate(depth)[1]
        steps = [E.eifmm_debug_export(tree, w, depth, d) for w in (0, 2, 3, 4)]
        out[name] = (far, steps, f.cpu().numpy()[:n])
    # every box of every exported step, to the bit
    for a, b in zip(out["sparse"][1], out["dense"][1]):
        assert np.array_equal(a, b)
    # the far field at the targets: the FP32 L2P groups its terms by the points
    # of a leaf (FP32 rounding of the whole chain: 2e-5 of the largest value)
    a, b = out["sparse"][0], out["dense"][0]
    assert np.abs(a - b).max() <= 2e-5 * np.abs(b).max()
    assert np.abs(out["sparse"][2] - out["dense"][2]).max() <= 2e-5 * np.abs(out["dense"][2]).max()


# One wave of tiles either way at level 5, seven against two at level 6: the M2L of
# a few occupied boxes takes no longer than that of all of them.
@pytest.mark.parametrize("depth", [5, 6])
def test_sparse_m2l_is_not_slower(E, depth):
    n, m = 20000, 2 ** depth
    x = wl.sphere_surface(n, 64)
    c = (np.arange(m) + 0.5) / m
    fill = np.stack(np.meshgrid(c, c, c, indexing="ij"), -1).reshape(-1, 3)
    s = dev(wl.sigma_uniform(n, 1, 65)[:, 0])
    ops = E.eifmm_ops_build("inv_r", 1.0, depth, 1e-4)
    ops.plan(0)
    ms = {}
    for name, t in (("sparse", x), ("dense", fill)):
        tree = E.eifmm_tree_build(dev(x), dev(t), (0, 0, 0), 1.0, depth, False)
        tree.set_option("single_stream", True)
        f = torch.zeros(len(t), dtype=torch.float64, device="cuda")
        E.eifmm_set_timing(True)
        try:
            runs = []
            for _ in range(6):
                E.eifmm_evaluate(tree, ops, s, f, "mixed")
                runs.append(E.eifmm_last_step_times(tree)[9 + depth])
        finally:
            E.eifmm_set_timing(False)
        ms[name] = min(runs)
    assert ms["sparse"] <= 1.25 * ms["dense"], ms


def test_export_gives_what_the_evaluation_used(E):
    """With another M2L kernel (option m2l_128row) nothing is left out and nothing is
    run again for an export: every box's steps are those of that kernel, as on the
    same sources with a target in every leaf; and so they are again afterwards."""
    n, depth = 20000, 6
    x, m = wl.sphere_surface(n, 66), 2 ** depth
    c = (np.arange(m) + 0.5) / m
    fill = np.stack(np.meshgrid(c, c, c, indexing="ij"), -1).reshape(-1, 3)
    s = dev(wl.sigma_uniform(n, 1, 67)[:, 0])
    ops = E.eifmm_ops_build("inv_r", 1.0, depth, 1e-4)
    ops.plan(0)
    d = ops.error_estimate(depth)[1]
    out = {}
    for name, t in (("sparse", x), ("dense", fill)):
        tree = E.eifmm_tree_build(dev(x), dev(t), (0, 0, 0), 1.0, depth, False)
        f = torch.zeros(len(t), dtype=torch.float64, device="cuda")
        for row in (True, False, True):
            tree.set_option("m2l_128row", row)
            E.eifmm_evaluate(tree, ops, s, f, "mixed")
            for again in range(2):  # an export changes nothing for the next one
                out[name, row, again] = [E.eifmm_debug_export(tree, w, depth, d) for w in (2, 3, 4)]
    for row in (True, False):
        for again in range(2):
            for a, b in zip(out["sparse", row, again], out["dense", row, 0]):
                assert np.array_equal(a, b), (row, again)
    assert not np.array_equal(out["dense", True, 0][0], out["dense", False, 0][0])
