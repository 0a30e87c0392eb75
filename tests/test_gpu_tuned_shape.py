"""The launch shape that asm_tune keeps serves the calls it was timed for: the same
precision and number of chains.  The kernels of several chains per warp end at
different block widths in the two precisions (FP32: 1024 points with four chains, 2048
with two; FP64: 256 and 1024), and the best shape of many chains is a slow one for
few, so that a handle tuned in one precision for one number of chains must sample in
the other precision, and with any other number, as an untuned handle does: accepted,
with the same shape and the same chains bit for bit."""
import os

import numpy as np
import pytest

from paper_1912_01379_gb300 import asm
from paper_1912_01379_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    torch.cuda.synchronize()


def _run(gp, chains, precision):
    gp.sample(chains, 0, 2, 17, precision=precision)
    f, chi2 = gp.chain_state()
    st = gp.status()
    return (st["team_lanes"], st["consumers_per_cta"]), f, chi2


def _same(x, y):
    assert x[0] == y[0]
    assert np.array_equal(x[1], y[1]) and np.array_equal(x[2], y[2])


# one block whose FP32 kernels run up to four (600) or two (1100) chains per warp and whose
# FP64 kernels two or one; enough chains that several per warp are the fastest in FP32
@pytest.mark.parametrize("N", [600, 1100])
def test_tuned_in_one_precision(N):
    p = W.small_problem(12, N, seed=9)
    gp = asm.Problem(p.K, p.G, p.C, p.levels, w=p.w)
    few = [_run(gp, n, prec) for n, prec in ((13, asm.ASM_MIXED), (13, asm.ASM_FP64), (8191, asm.ASM_FP64))]
    many = _run(gp, 8192, asm.ASM_MIXED)
    team, cons, _ = gp.tune(8192, precision=asm.ASM_MIXED)
    tuned = _run(gp, 8192, asm.ASM_MIXED)
    assert tuned[0][0] == team and (cons == 0 or tuned[0][1] == cons)
    assert np.array_equal(tuned[1], many[1]) and np.array_equal(tuned[2], many[2])
    _same(_run(gp, 13, asm.ASM_FP64), few[1])
    _same(_run(gp, 8191, asm.ASM_FP64), few[2])
    _same(_run(gp, 13, asm.ASM_MIXED), few[0])
    # a choice in the other precision leaves this one in place
    gp.tune(13, precision=asm.ASM_FP64)
    _same(_run(gp, 8192, asm.ASM_MIXED), tuned)


@pytest.mark.parametrize("M,N,precision", [(12, 600, asm.ASM_FP64), (12, 1100, asm.ASM_MIXED), (12, 1100, asm.ASM_FP64),
                                           (7000, 24, asm.ASM_FP64)])
def test_lanes_without_a_kernel_or_room(M, N, precision):
    """ASM_TEAM_LANES=8 where no kernel runs four chains per warp on such blocks, or where their
    residuals do not fit shared memory: the handle runs as without it."""
    p = W.small_problem(M, N, seed=9)
    first = _run(asm.Problem(p.K, p.G, p.C, p.levels, w=p.w), 13, precision)
    old = os.environ.get("ASM_TEAM_LANES")
    os.environ["ASM_TEAM_LANES"] = "8"
    try:
        gp = asm.Problem(p.K, p.G, p.C, p.levels, w=p.w)
    finally:
        if old is None:
            os.environ.pop("ASM_TEAM_LANES")
        else:
            os.environ["ASM_TEAM_LANES"] = old
    _same(_run(gp, 13, precision), first)
