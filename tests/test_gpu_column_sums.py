"""The sums over chains behind asm_average, asm_mc_error and asm_backward (CTAs of
eight columns, the chains in 32 row groups) against numpy sums of the chain states
they are made of, at ragged column and chain counts: one chain, fewer chains than
row groups, one more than a multiple, columns one beyond a tile.

With one kept sweep the sums are the chain states themselves; with eight the only
snapshot of the moments is the final state, so that the covariance products follow
from it too.  FP64 chain state; the sums of at most 97 terms carry 97 2^-53 = 1e-14
relative to the sum of magnitudes, which the centring (mean^2 / variance < 1e3 on
these problems) and the tracked residual (1e-10 of the recomputed one) raise to at
most 1e-8 of the products' norm."""
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


def _close(x, y, tol):
    assert np.linalg.norm(x - y) <= tol * np.linalg.norm(y), (x, y)


@pytest.mark.parametrize("N,chains", [(7, 1), (8, 5), (9, 32), (17, 33), (40, 97)])
def test_sums_over_chains(N, chains):
    p = W.theta_problem(N=N, M=12, noise=1e-2)
    dK, dw = p.extra["dK_dtheta"], p.extra["dw_dtheta"]
    gp = asm.Problem(p.K, p.G, p.C, [[0]], w=p.w, dK_dtheta=dK, dw_dtheta=dw)
    gp.sample(chains, 4, 1, 11, precision=asm.ASM_FP64)
    f, _ = gp.chain_state()
    r = gp.average()
    _close(r["mean_fbar"], f.mean(axis=0), 1e-12)
    if chains == 1:
        assert np.all(np.isnan(r["sem_fbar"]))
        return
    _close(r["sem_fbar"], f.std(axis=0, ddof=1) / np.sqrt(chains), 1e-9)

    gp.sample(chains, 4, 8, 12, precision=asm.ASM_FP64, moments=True)
    f, _ = gp.chain_state()
    v = np.random.default_rng(N).standard_normal(N)
    gG, gt = gp.backward(v)
    d = f - f.mean(axis=0)
    vf = d @ (v / p.w)
    _close(gG, np.linalg.solve(p.C, p.K @ (d.T @ vf / chains)), 1e-8)
    res = np.linalg.solve(p.C, (p.G[:, None] - p.K @ f.T))                       # M x chains
    s = np.einsum("mq,pmn,qn->qp", res, dK, f)
    _close(gt, vf @ (s - s.mean(axis=0)) / chains - dw @ (v * f.mean(axis=0) / p.w ** 2), 1e-8)


@pytest.mark.parametrize("N,chains,sweeps", [(9, 3, 64), (33, 40, 192)])
def test_binned_levels(N, chains, sweeps):
    """Level 0 of the binning from runs that stop at each bin boundary: bins of 64 sweeps."""
    p = W.small_problem(8, N, seed=2)
    gp = asm.Problem(p.K, p.G, p.C, p.levels, w=p.w)
    bins, last = [], 0.0
    for k in range(sweeps // 64):
        gp.sample(chains, 0, 64, 5, precision=asm.ASM_FP64, cont=k > 0)
        total = gp.average()["mean_fbar"] * 64 * (k + 1)
        bins.append((total - last) / 64)
        last = total
    e = gp.mc_error()
    assert list(e["bins_per_chain"]) == [(sweeps // 64) >> l for l in range(8)]
    assert np.all(np.isnan(e["sigma2_levels"][2:]))
    assert np.all(np.isfinite(e["sigma2_levels"][0]))
    _close(np.mean(bins, axis=0), gp.average()["mean_fbar"], 1e-12)
