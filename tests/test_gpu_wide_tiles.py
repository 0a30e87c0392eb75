"""The widest register tiles, the gamma prior's two forms and the tightest shared memory.

* Blocks of 513 to 2048 points: the states and counters of one chain per warp, bit for
  bit, from the kernels of two and four (where one exists for the width).
* The prior's kernel keeps a - 1 and the logarithms of a block's points in registers
  (up to 1024 points in FP32, 512 in FP64), a - 1 alone (2048, 1024) or neither.  The
  tile follows the handle's largest block, so that a problem takes the one form alone
  and another in a batch with a wider problem: the same states bit for bit.
* The most data points that one warp of one chain leaves room for (a single packet slot,
  a ring of two stages, U streamed), and one more.  Rows of zeros add nothing to a
  chain's sums, so that the same problem without them, which has packets with U and a deep
  ring, gives the same states bit for bit."""
import os
from types import SimpleNamespace

import numpy as np
import pytest

from paper_1912_01379_gb300 import asm
from paper_1912_01379_gb300 import workloads as W

pytestmark = pytest.mark.gpu

COUNTS = ("degenerate_moves", "zero_mode_moves", "tail_capped", "nonfinite_moves", "timeouts", "prior_rejections")


@pytest.fixture(autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    torch.cuda.synchronize()


def _with_lanes(lanes, make):
    old = os.environ.get("ASM_TEAM_LANES")
    os.environ["ASM_TEAM_LANES"] = str(lanes)
    try:
        return make()
    finally:
        if old is None:
            os.environ.pop("ASM_TEAM_LANES")
        else:
            os.environ["ASM_TEAM_LANES"] = old


def _states(gp, chains, sweeps, precision):
    gp.sample(chains, 0, sweeps, 17, precision=precision)
    f, chi2 = gp.chain_state()
    st = gp.status()
    assert st["timeouts"] == 0
    return f, chi2, np.array([st[k] for k in COUNTS]), gp.average()["mean_fbar"]


def _given(Kt, gt, levels):
    """The blocks' factors of a whitened kernel, in the layout of asm_desc."""
    M, N = Kt.shape
    d, V, U = [], [], []
    for lv in levels:
        for s0, s1 in zip(lv, list(lv[1:]) + [N]):
            n = s1 - s0
            u, s, vt = np.linalg.svd(Kt[:, s0:s1], full_matrices=n > M)
            d.append(np.concatenate([s, np.zeros(n - s.size)]))
            V.append(vt.ravel())
            U.append(np.ascontiguousarray(u.T[:min(M, n)]).ravel())
    return SimpleNamespace(Kt=Kt, gt=gt, d=np.concatenate(d), V=np.concatenate(V), U=np.concatenate(U))


def _handle(fac, levels):
    """A handle from given factors, without a covariance."""
    desc, keep, shape = asm._make_desc(fac.Kt, fac.gt, np.eye(1), levels, factors=fac)
    desc.C = None
    gp = asm.Problem.__new__(asm.Problem)
    gp._h, gp._ws, gp.chains = None, None, 0
    gp.M, gp.N, gp.w, gp.levels, gp.P = shape
    h = asm.ct.c_void_p()
    asm._check(asm.load().asm_setup(asm.ct.byref(desc), asm.ct.byref(h)), "asm_setup")
    gp._h = h
    return gp


@pytest.mark.parametrize("N", [520, 1024, 1040, 2048])
def test_wide_blocks(N):
    levels = [[0], [0, N // 2 + 3]]
    p = W.small_problem(9, N, seed=N, levels=levels)
    fac = _given(p.K / 1e-3, p.G / 1e-3, levels)   # the problem's noise is 1e-3
    handles = {s: _with_lanes(s, lambda: _handle(fac, levels)) for s in (32, 16, 8)}
    for precision, widest in ((asm.ASM_MIXED, {16: 2048, 8: 1024}), (asm.ASM_FP64, {16: 1024, 8: 256})):
        first = _states(handles[32], 13, 3, precision)
        assert np.all(first[0] >= 0) and first[2][3] == 0
        for lanes, most in widest.items():
            if N > most:
                continue
            other = _states(handles[lanes], 13, 3, precision)
            assert handles[lanes].status()["team_lanes"] == lanes
            for a, b in zip(first, other):
                assert np.array_equal(a, b), (lanes, precision)


# the narrow problem's blocks fill its own tile wholly or in part; the wide one raises the tile
@pytest.mark.parametrize("precision,levels,N,wide", [
    (asm.ASM_MIXED, [[0], [0, 300]], 500, 520), (asm.ASM_MIXED, [[0, 200]], 340, 600),
    (asm.ASM_FP64, [[0], [0, 150]], 250, 260), (asm.ASM_FP64, [[0, 100]], 170, 300),
    (asm.ASM_MIXED, [[0], [0, 300]], 500, 1100), (asm.ASM_MIXED, [[0], [0, 560]], 900, 1030),
    (asm.ASM_FP64, [[0], [0, 150]], 250, 520), (asm.ASM_FP64, [[0, 300]], 500, 1030),
    (asm.ASM_FP64, [[0], [0, 300]], 600, 1030)])
def test_prior_in_registers_and_from_memory(precision, levels, N, wide):
    def spec(n, lv, seed):
        p = W.small_problem(12, n, seed=seed, levels=lv, noise=3e-3)
        return dict(K=p.K, G=p.G, C=p.C, levels=p.levels, w=p.w, prior_shape=1.0 + 0.75 * (np.arange(n) % 3))

    alone = asm.Problem(**spec(N, levels, 4))
    alone.sample(13, 0, 20, 17, precision=precision)
    both = asm.Batch([spec(N, levels, 4), spec(wide, [[0]], 5)])
    both.sample(13, 0, 20, 17, precision=precision)
    assert alone.status()["prior_rejections"] > 0 and both.status()["timeouts"] == 0
    x, y = alone.average(), both.average(0)
    for k in ("mean_fbar", "sem_fbar", "ess"):
        assert np.array_equal(x[k], y[k]), k


@pytest.mark.parametrize("precision,most", [(asm.ASM_FP64, 28064), (asm.ASM_MIXED, 56928)])
def test_single_packet_slot(precision, most):
    """227 KB less 512 bytes hold, per element of T: c / w (32), r~ (M to a multiple of 32) and
    128 uniforms; 896 + 256 bytes of barriers and padding; one packet without U (32 + 64
    elements) and two stages of 256 elements.  A second packet does not fit at `most`."""
    N, M0, levels = 24, 40, [[0], [0, 11]]
    es = 8 if precision == asm.ASM_FP64 else 4
    room = 227 * 1024 - 512 - 896 - 256 - 2 * 256 * es - 160 * es
    packet = 96 * es
    assert most % 32 == 0 and es * most + packet <= room < es * most + 2 * packet and es * (most + 32) + packet > room
    rng = np.random.default_rng(6)
    small = _given(rng.standard_normal((M0, N)) + 2.0, 20.0 + rng.standard_normal(M0), levels)
    f0, chi0, n0, mean0 = _states(_handle(small, levels), 5, 3, precision)
    for M in (most, most + 1):
        pad = lambda a: np.concatenate([a, np.zeros((M - M0,) + a.shape[1:])])
        U = small.U.reshape(-1, M0)
        big = SimpleNamespace(Kt=pad(small.Kt), gt=pad(small.gt), d=small.d, V=small.V,
                              U=np.concatenate([U, np.zeros((U.shape[0], M - M0))], axis=1).ravel())
        gp = _handle(big, levels)
        if M > most:
            with pytest.raises(asm.ASMError) as e:
                gp.sample(5, 0, 3, 17, precision=precision)
            assert e.value.code == -9
            continue
        f, chi2, n, mean = _states(gp, 5, 3, precision)
        assert gp.status()["consumers_per_cta"] == 1
        assert np.array_equal(f, f0) and np.array_equal(n, n0) and np.array_equal(mean, mean0)
        assert np.array_equal(chi2, chi0)
