"""The FP64 far field where memory is short: operators whose residue image does not
fit, or steps whose scratch does not, run on the FP64 pipes; what did not fit is
asked for once; nothing is built while a stream is captured."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1408_0210_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu
N, DEPTH, EPS = 3000, 3, 1e-4  # d = 126: an M2L image takes 157 MB, a transfer's 4 MB
MB = 1 << 20


@pytest.fixture(scope="module")
def E():
    from paper_1408_0210_gb300 import eifmm
    eifmm.lib()
    return eifmm


@pytest.fixture
def limit(E):
    yield E.eifmm_debug_alloc_limit
    E.eifmm_debug_alloc_limit(-1)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def setup(E, R=1, option=None):
    x, s = wl.uniform_cube(N, 71), wl.sigma_uniform(N, R, 72)
    ops = E.eifmm_ops_build("inv_r", 1.0, DEPTH, EPS)
    tree = E.eifmm_tree_build(dev(x), None, (0, 0, 0), 1.0, DEPTH, True)
    if option:
        tree.set_option(option, True)
    f = torch.zeros(R, N, dtype=torch.float64, device="cuda")
    return ops, tree, dev(s.T).T if R > 1 else dev(s[:, 0]), f.T if R > 1 else f[0]


def close(a, b):
    """Both carry FP64 rounding through the chain: 1e-12, as for the whole FP64 path."""
    a, b = a.cpu().numpy(), b.cpu().numpy()
    return np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


# 64 MB refuses the images of the M2L; with 64 columns 200 MB let them through
# and refuse the scratch
@pytest.mark.parametrize("R,most", [(1, 64 * MB), (64, 200 * MB)])
def test_what_does_not_fit_is_asked_for_once(E, limit, R, most):
    ops, tree, s, f = setup(E, R)
    limit(most)
    counts, refused = [], []
    for _ in range(3):
        before = E.eifmm_kernel_launches()
        E.eifmm_evaluate(tree, ops, s, f, "fp64")
        counts.append(E.eifmm_kernel_launches() - before)
        refused.append(limit(most))
    assert refused[0] > 0 and refused[1:] == [0, 0]
    assert counts[1] == counts[2]
    limit(-1)
    g = torch.zeros_like(f) if R == 1 else torch.zeros(R, N, dtype=torch.float64, device="cuda").T
    ops2, tree2, _, _ = setup(E, R, "m2l_fp64")
    E.eifmm_evaluate(tree2, ops2, s, g, "fp64")
    assert close(f, g)


def test_batch_without_room_for_the_images(E, limit):
    ops, tree, s, f = setup(E)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    limit(64 * MB)
    for call in range(2):
        f.zero_()
        torch.cuda.synchronize()
        before = E.eifmm_kernel_launches()
        E.eifmm_evaluate_batched([tree], [s], [f], ops, "fp64", stream)
        stream.synchronize()
        assert (E.eifmm_kernel_launches() > before) == (call == 0)
        assert (limit(64 * MB) > 0) == (call == 0)
        if call == 0:
            first = f.clone()
    assert torch.equal(first, f)


def test_nothing_is_built_under_capture(E):
    """The option is taken back while the workspace holds no images: the captured
    call runs without them and the next direct one builds them."""
    ops, tree, s, f = setup(E, option="m2l_fp64")
    E.eifmm_evaluate(tree, ops, s, f, "fp64")
    pipes = f.clone()
    torch.cuda.synchronize()
    tree.set_option("m2l_fp64", False)
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        E.eifmm_evaluate(tree, ops, s, f, "fp64", stream)
    f.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(f, pipes)
    E.eifmm_evaluate(tree, ops, s, f, "fp64")
    assert not torch.equal(f, pipes) and close(f, pipes)
