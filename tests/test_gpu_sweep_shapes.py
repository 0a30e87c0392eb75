"""The sweep kernel's branches on block width and launch shape: half and whole
vectors, whole and partly filled register tiles, blocks of at most eight modes
(partial sums over lanes), the null-space tail of a block's moves, one, two and
four chains per warp, U in the visit packet or in global memory, shallow rings.

FP64: one sweep from the oracle's factors and random numbers within 1e-9 of the
oracle's states (the tolerance of the step parity: the window over which the
oracle's own one-ulp divergence stays below 1e-11).  Every shape must then give
the first shape's states and counters bit for bit, in both precisions."""
import os

import numpy as np
import pytest

from oracle import oracle as O
from paper_1912_01379_gb300 import asm
from paper_1912_01379_gb300 import workloads as W

pytestmark = pytest.mark.gpu

COUNTS = ("degenerate_moves", "zero_mode_moves", "tail_capped", "nonfinite_moves", "timeouts")
SHAPES = [{}, {"ASM_TEAM_LANES": "16"}, {"ASM_TEAM_LANES": "8"}, {"ASM_NO_U_STAGE": "1", "ASM_TEAM_LANES": "16"},
          {"ASM_NO_U_STAGE": "1", "ASM_RING_DEPTH": "2", "ASM_RECORDS_PER_STAGE": "1", "ASM_CONSUMERS_PER_CTA": "2",
           "ASM_TEAM_LANES": "32"}]


@pytest.fixture(autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    torch.cuda.synchronize()


def _states(p, factors, shape, precision, sweeps, chains=13):
    old = {k: os.environ.get(k) for k in shape}
    os.environ.update(shape)
    try:
        gp = asm.Problem(p.K, p.G, p.C, p.levels, w=p.w, factors=factors)
        gp.sample(chains, 0, sweeps, 17, precision=precision)
        f, chi2 = gp.chain_state()
        st = gp.status()
        return f, chi2, [st[k] for k in COUNTS], gp.average()["mean_fbar"]
    finally:
        for k, v in old.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v


# widths around the half vector (32 / 64 elements), the vector (64 / 128), the next tiles, and tiny blocks
@pytest.mark.parametrize("M,N,levels", [
    (10, 32, [[0]]), (10, 33, [[0]]), (70, 64, [[0]]), (9, 65, [[0]]), (40, 128, [[0]]), (16, 129, [[0]]),
    (33, 257, [[0], [0, 129]]), (21, 400, [[0, 130, 260, 380]]), (12, 20, [[0, 1, 3, 6, 10, 15]]),
    (7, 40, [[0, 8, 17, 26, 33]])])
def test_block_widths_and_shapes(M, N, levels):
    p = W.small_problem(M, N, seed=100 + N, levels=levels)
    op = O.OracleProblem(p.K, p.G, p.C, p.levels)
    dec = op.decomposition()
    ref = op.run(13, 0, 1, seed=17)["f_final"]
    first = _states(p, dec, {}, asm.ASM_FP64, 1)
    err = np.abs(first[0] - ref) / np.abs(ref).max(axis=1, keepdims=True)
    assert err.max() <= 1e-9, err.max()
    for precision in (asm.ASM_FP64, asm.ASM_MIXED):
        first = _states(p, dec, SHAPES[0], precision, 66)
        assert first[2][-1] == 0
        for shape in SHAPES[1:]:
            other = _states(p, dec, shape, precision, 66)
            for a, b in zip(first, other):
                assert np.array_equal(a, b), (shape, precision)


def test_long_residuals():
    """Thousands of data points leave shared memory for a few chains only, down to one warp of
    one chain on an SM: every chain count is taken and gives the few chains' states."""
    p = W.small_problem(7000, 24, seed=77, levels=[[0], [0, 12]])
    for precision, chains in ((asm.ASM_FP64, (13, 500, 2300)), (asm.ASM_MIXED, (13, 2300))):
        gp = asm.Problem(p.K, p.G, p.C, p.levels, w=p.w)
        states = []
        for n in chains:
            gp.sample(n, 0, 2, 17, precision=precision)
            states.append([x[:13].copy() for x in gp.chain_state()])
            assert gp.status()["timeouts"] == 0
        for f, chi2 in states[1:]:
            assert np.array_equal(f, states[0][0]) and np.array_equal(chi2, states[0][1])
