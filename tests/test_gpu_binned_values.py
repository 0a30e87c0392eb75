"""asm_mc_error's binned variances against numpy, from bins read one at a time: chain q
alone (chain offset q, the same problem id, so the same moves bit for bit) run in steps of
64 sweeps gives each of its bin means as a difference of the kept sweeps' totals.

FP64.  A total of at most 256 sweeps carries 256 2^-53 = 3e-14 relative, a difference of two
totals four times that relative to a bin's mean, and the variance of at most 160 bin means is
formed as a difference of sums of squares, 160 2^-53 of the squared mean: 1e-12 of the squared
mean and the variance together bounds all of them."""
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


# columns one beyond a tile of 8, one tile, several; fewer chains than the 32 row groups, as many, more
@pytest.mark.parametrize("N,chains,n_bins", [(9, 3, 1), (8, 32, 2), (33, 40, 4), (17, 1, 4)])
def test_levels_equal_numpy(N, chains, n_bins):
    p = W.small_problem(8, N, seed=2, noise=1e-2)
    gp = asm.Problem(p.K, p.G, p.C, p.levels, w=p.w)
    gp.sample(chains, 0, 64 * n_bins, 5, precision=asm.ASM_FP64)
    e = gp.mc_error()
    assert list(e["bins_per_chain"]) == [n_bins >> l for l in range(8)]
    bins = np.zeros((chains, n_bins, N))
    one = asm.Problem(p.K, p.G, p.C, p.levels, w=p.w)
    for q in range(chains):
        one.set_stream_ids(0, q)
        last = np.zeros(N)
        for k in range(n_bins):
            one.sample(1, 0, 64, 5, precision=asm.ASM_FP64, cont=k > 0)
            total = one.average()["mean_fbar"] * (64 * (k + 1))
            bins[q, k] = (total - last) / 64
            last = total
    for l in range(8):
        c = n_bins >> l
        got = e["sigma2_levels"][l]
        if c * chains < 2:
            assert np.all(np.isnan(got)), l
            continue
        b = bins[:, :c << l].reshape(chains, c, 1 << l, N).mean(axis=2).reshape(chains * c, N)
        var, tol = b.var(axis=0, ddof=1), 1e-12 * (b ** 2).mean(axis=0)
        assert np.all(np.abs(got * (chains * c) - var) <= tol), l
        assert np.median(tol / var) < 1e-6, l   # the spread stands far above the tolerance
        if c == 1:   # one bin per chain: its mean is the mean over the chain's binned sweeps
            sem2 = gp.average()["sem_fbar"] ** 2
            assert np.all(np.abs(got - sem2) * chains <= tol), l
