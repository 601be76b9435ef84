"""Recorded batches: a batch whose trees or operators have changed since it was
recorded is recorded anew (a replay launches nothing from the host, so the host's
launch counter tells the two apart), and its results are those of single calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1408_0210_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu
DEPTH, SIZES = 3, (2500, 4000, 3100)


@pytest.fixture(scope="module")
def E():
    from paper_1408_0210_gb300 import eifmm
    eifmm.lib()
    return eifmm


class Batch:
    def __init__(self, E, ops, prec, m2l_fp64=False):
        self.E, self.ops, self.prec, self.stream = E, ops, prec, torch.cuda.Stream()
        self.x = [torch.from_numpy(wl.uniform_cube(n, 50 + n)).cuda() for n in SIZES]
        self.s = [torch.from_numpy(wl.sigma_uniform(n, 1, 60 + n)[:, 0].copy()).cuda() for n in SIZES]
        self.trees = [E.eifmm_tree_build(x, None, (0, 0, 0), 1.0, DEPTH, True) for x in self.x]
        for t in self.trees:
            t.set_option("m2l_fp64", m2l_fp64)
        self.f = [torch.zeros(n, dtype=torch.float64, device="cuda") for n in SIZES]
        torch.cuda.synchronize()

    def call(self):
        """Launches from the host, and the results."""
        before = self.E.eifmm_kernel_launches()
        self.E.eifmm_evaluate_batched(self.trees, self.s, self.f, self.ops, self.prec, self.stream)
        self.stream.synchronize()
        return self.E.eifmm_kernel_launches() - before, [f.cpu().numpy() for f in self.f]

    def record(self):
        n, f = self.call()
        assert n > 0
        n, g = self.call()
        assert n == 0 and all(np.array_equal(a, b) for a, b in zip(f, g))
        return f

    def single(self, option=None):
        """The same on trees of their own."""
        out = []
        for x, s in zip(self.x, self.s):
            t = self.E.eifmm_tree_build(x, None, (0, 0, 0), 1.0, DEPTH, True)
            if option:
                t.set_option(option, True)
            f = torch.zeros(len(x), dtype=torch.float64, device="cuda")
            self.E.eifmm_evaluate(t, self.ops, s, f, self.prec)
            out.append(f.cpu().numpy())
        return out


def same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


def test_calibration_leaves_the_operands_in_place(E):
    """A calibration builds nothing into a set whose tier needs no FP64 operands and
    frees none that the set holds: the next FP64 call launches what a warm call does."""
    ops = E.eifmm_ops_build("inv_r", 1.0, DEPTH, 1e-4)
    assert ops.plan() < 3
    b = Batch(E, ops, "fp64")
    f = b.record()
    out = torch.zeros(SIZES[0], dtype=torch.float64, device="cuda")
    counts = []
    for recalibrate in (False, False, True):
        if recalibrate:
            ops.calibrate(1e-4)
        before = E.eifmm_kernel_launches()
        E.eifmm_evaluate(b.trees[0], ops, b.s[0], out, "fp64")
        counts.append(E.eifmm_kernel_launches() - before)
    assert counts[1] == counts[2]
    assert np.array_equal(out.cpu().numpy(), f[0])
    assert same(b.call()[1], f)


@pytest.mark.parametrize("change", ["option", "columns", "compress", "plan", "autotune"])
def test_changed_batch_is_recorded_anew(E, change):
    prec = "mixed" if change in ("plan", "autotune") else "fp64"
    ops = E.eifmm_ops_build("inv_r", 1.0, DEPTH, 1e-4)
    b = Batch(E, ops, prec, m2l_fp64=change == "option")
    b.record()
    if change == "option":  # the residue products: one tree's scratch grows in a call of its own
        for t in b.trees:
            t.set_option("m2l_fp64", False)
        E.eifmm_evaluate(b.trees[1], ops, b.s[1], torch.zeros(SIZES[1], dtype=torch.float64, device="cuda"), prec)
    elif change == "columns":  # a call with other columns sizes the workspace anew
        s = torch.stack([b.s[2], b.s[2]]).T
        E.eifmm_evaluate(b.trees[2], ops, s, torch.zeros(2, SIZES[2], dtype=torch.float64, device="cuda").T, prec)
    elif change == "compress":
        ops.compress(1e-6)
    elif change == "plan":  # other operand planes and back
        ops.plan(1)
        ops.plan(0)
    else:
        E.eifmm_autotune(b.trees[0], ops, 1, prec)
    torch.cuda.synchronize()
    n, f = b.call()
    assert n > 0
    if change != "autotune":  # the tuned kernels group their sums differently
        assert same(f, b.single())
    n, g = b.call()
    assert n == 0 and same(f, g)
