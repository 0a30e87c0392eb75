"""Cases of the average-spectrum sampler whose speed is measured.

Every case goes through the calls that a user's program makes: a problem (or a
batch of problems) is set up once from host arrays, and a pass samples its
chains afresh and reads the averages, the Monte Carlo error or the gradients.
The workloads are those of paper_1912_01379_gb300.workloads: the paper's own
test case, plain modes, blocked modes, the grid-size sweep, the batch of uneven
problems and the differentiation workload, with run lengths of a few refresh
periods (64 sweeps) each, so that a pass stays below a second; the cost of
longer runs is proportional to their sweeps.

Keys of a case:
  workload   "modes" (M x N, one level), "blocked" (one level and equal blocks),
             "paper" (60 Matsubara frequencies, full hierarchy), "grid" (400
             times, 16 blocks), "batch" (uneven problems), "theta" (grid
             parameters, gradients)
  call       "sample" (sample, averages, binned error), "first_sweep" (one sweep
             with given factors, chain states read back), "gradient" (sample
             with moments, averages, both vector-Jacobian products), "noalloc"
             (device outputs, nothing allocated), "fresh" (set-up in the pass)
  mixed      FP32 chain state with FP64 sums, or plain FP64
"""
import math

import numpy as np
import torch

from paper_1912_01379_gb300 import asm
from paper_1912_01379_gb300 import workloads as W


def listed():
    return [
        # the smallest call: the first sweep of a few chains with the user's own factors,
        # its states read back (how another implementation's modes are checked or traced)
        {"name": "first_sweep_f64", "workload": "modes", "call": "first_sweep", "mixed": False,
         "M": 20, "N": 50, "blocks": 1, "chains": 16, "burn": 0, "sweeps": 1},
        # plain modes sampling of one spectrum with few chains in plain FP64
        {"name": "plain_f64", "workload": "modes", "call": "sample", "mixed": False,
         "M": 20, "N": 50, "blocks": 1, "chains": 16, "burn": 64, "sweeps": 128},
        # the same in a host program that owns all device memory: results stay on the device
        {"name": "plain_noalloc", "workload": "modes", "call": "noalloc", "mixed": True,
         "M": 20, "N": 50, "blocks": 1, "chains": 16, "burn": 64, "sweeps": 192},
        # the paper's own test case on a non-uniform grid over the whole block hierarchy
        {"name": "paper_hierarchy", "workload": "paper", "call": "sample", "mixed": True,
         "grid": "gaussian", "N": 64, "chains": 1024, "burn": 128, "sweeps": 384},
        # blocked modes, the benchmark's workload: 1024 chains of one problem
        {"name": "blocked", "workload": "blocked", "call": "sample", "mixed": True,
         "M": 100, "N": 400, "blocks": 8, "chains": 1024, "burn": 128, "sweeps": 256},
        # the same in plain FP64, the reference precision
        {"name": "blocked_f64", "workload": "blocked", "call": "sample", "mixed": False,
         "M": 100, "N": 400, "blocks": 8, "chains": 1024, "burn": 16, "sweeps": 64},
        # odd sizes and a gamma prior (one grid's measure simulated on another)
        {"name": "prior_ragged", "workload": "blocked", "call": "sample", "mixed": True, "prior": True,
         "M": 37, "N": 101, "blocks": 5, "chains": 250, "burn": 64, "sweeps": 192},
        # new data from a measurement: set-up, a short run and the averages, as one call
        {"name": "fresh_blocked", "workload": "blocked", "call": "fresh", "mixed": True,
         "M": 100, "N": 400, "blocks": 8, "chains": 1024, "burn": 64, "sweeps": 192},
        # many independent uneven problems in one handle (a momentum-resolved run)
        {"name": "batch", "workload": "batch", "call": "sample", "mixed": True,
         "problems": 24, "chains": 64, "burn": 64, "sweeps": 192},
        # gradients of the average: 4096 chains with snapshots, both products
        {"name": "gradient", "workload": "theta", "call": "gradient", "mixed": True,
         "M": 64, "N": 200, "chains": 4096, "burn": 64, "sweeps": 192},
        # the grid-size sweep at its small end
        {"name": "grid_250", "workload": "grid", "call": "sample", "mixed": True,
         "density": "uniform", "N": 250, "chains": 8192, "burn": 64, "sweeps": 128},
        # and at its large end: the largest grid
        {"name": "grid_2000", "workload": "grid", "call": "sample", "mixed": True,
         "density": "gaussian", "N": 2000, "chains": 2048, "burn": 8, "sweeps": 56},
    ]


def _seconds(c):
    """Rough time of a pass, from a move's latency and the chains that run side by side."""
    n = c.get("N", 550) * (c["burn"] + c["sweeps"])
    chains = c["chains"] * c.get("problems", 1)
    if c["mixed"]:
        return n * 5e-7 * (1 + c.get("N", 550) / 300) * max(1.0, chains / 1000)
    return n * 8e-6 * max(1.0, chains / 1000)


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["modes", "blocked", "blocked", "paper", "grid", "batch", "theta"])
        c = {"workload": kind, "call": "sample", "mixed": rng.random() < 0.7, "chains": log(1, 4096),
             "burn": rng.choice([0, 16, 64, 100]), "sweeps": log(8, 400)}
        if kind in ("modes", "blocked"):
            c["M"], c["N"] = log(10, 200), log(24, 800)
            c["blocks"] = 1 if kind == "modes" else rng.randint(2, max(2, min(16, c["N"] // 12)))
            if rng.random() < 0.2:
                c["call"] = rng.choice(["first_sweep", "noalloc", "fresh"])
            elif kind == "blocked" and rng.random() < 0.2:
                c["prior"] = True
            if c["call"] == "first_sweep":
                c.update(burn=0, sweeps=1, M=min(c["M"], 100), N=min(c["N"], 200), chains=min(c["chains"], 512))
                c["blocks"] = min(c["blocks"], c["N"] // 12)
            if c["call"] == "noalloc":   # its scratch is bounded: 64 MiB
                c["chains"] = max(1, min(c["chains"], (40 << 20) // (280 * (c["N"] + c["M"]))))
        elif kind == "paper":
            c["grid"], c["N"] = rng.choice(["uniform", "gaussian", "exponential", "lorentzian"]), log(32, 256)
        elif kind == "grid":
            c["density"], c["N"], c["chains"] = rng.choice(["uniform", "gaussian"]), log(250, 2000), log(512, 8192)
        elif kind == "batch":
            c["problems"], c["chains"] = rng.randint(2, 24), log(16, 256)
        else:
            c.update(call="gradient", M=log(24, 96), N=log(60, 300), chains=log(128, 4096))
            c["sweeps"] = max(c["sweeps"], 32)
        if _seconds(c) <= 0.6:
            return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _problem(c, seed):
    kind = c["workload"]
    if kind == "paper":
        p = W.paper_problem(grid=c["grid"], N=c["N"], seed=2000 + seed)
        p.levels = asm.partition_hierarchy(c["N"])
        return p
    if kind == "grid":
        return W.grid_sweep_problem(c["N"], c["density"], seed=3000 + seed)
    if kind == "theta":
        return W.theta_problem(N=c["N"], M=c["M"], seed=4000 + seed)
    levels = [[0]] if c["blocks"] == 1 else [[0], W.equal_blocks(c["N"], c["blocks"])]
    if (c["M"], c["N"], c["blocks"]) == (100, 400, 8):
        return W.blocked_modes_problem(seed=5000 + seed)
    if (c["M"], c["N"], c["blocks"]) == (20, 50, 1):
        return W.plain_modes_problem(seed=6000 + seed)
    return W.small_problem(c["M"], c["N"], 7000 + seed, levels=levels, beta=16.0, bosonic=bool(c["N"] % 2))


def _fields(p):
    return dict(K=p.K, G=p.G, C=p.C, levels=p.levels, w=p.w)


def _prior_shape(N):
    return 1.0 + 0.5 * (np.arange(N) % 3)


class _Factors:
    """Whitened kernel and data and the singular vectors of every block of every
    level, zero modes marked by d = 0, in the layout that the library takes."""

    def __init__(self, p):
        L = np.linalg.cholesky(p.C)
        self.Kt, self.gt = np.linalg.solve(L, p.K), np.linalg.solve(L, p.G)
        M, N = p.K.shape
        self.blocks = []   # (level, start, end, d, V, U)
        for level, starts in enumerate(p.levels):
            for a, b in zip(starts, list(starts[1:]) + [N]):
                U, d, V = np.linalg.svd(self.Kt[:, a:b], full_matrices=True)
                n, k = b - a, min(M, b - a)
                d = np.concatenate([d, np.zeros(n - k)])
                U = np.ascontiguousarray(U[:, :k].T)
                signs = (V.max(axis=1) > 0) & (V.min(axis=1) < 0)
                d[(d <= d[0] * max(M, n) * 2.0 ** -52) | ((d <= d[0] * max(M, n) * 2.0 ** -40) & signs)] = 0.0
                self.blocks.append((level, int(a), int(b), d, V, U))
        self.d, self.V, self.U = (np.concatenate([x[i].ravel() for x in self.blocks]) for i in (3, 4, 5))


def prepare(case, seed):
    c, kind = case, case["workload"]
    s = {"case": c, "seed": int(seed)}
    if kind == "batch":
        problems = W.batch_problems(seed=8000 + c["problems"], n_problems=c["problems"])   # sizes by the case
        rng = np.random.default_rng(seed)
        for p in problems:
            p.G = p.K @ p.fbar_true + np.linalg.cholesky(p.C) @ rng.standard_normal(p.M)
        s["handle"] = asm.Batch([_fields(p) for p in problems])
        return s
    p = _problem(c, seed)
    args = _fields(p)
    if c.get("prior"):
        args["prior_shape"] = _prior_shape(p.N)
    if c["call"] == "first_sweep":
        args["factors"] = _Factors(p)
    if c["call"] == "gradient":
        args.update(dK_dtheta=p.extra["dK_dtheta"], dw_dtheta=p.extra["dw_dtheta"])
        s["v"] = np.random.default_rng(seed).standard_normal(p.N)
    if c["call"] == "fresh":
        s["args"] = args
        return s
    s["handle"] = asm.Problem(**args)
    if c["call"] == "noalloc":
        s["out"] = [torch.empty(p.N, dtype=torch.float64, device="cuda") for _ in range(3)]
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def run(state):
    c = state["case"]
    h = state.get("handle") or asm.Problem(**state["args"])
    precision = asm.ASM_MIXED if c["mixed"] else asm.ASM_FP64
    if c["call"] == "noalloc":
        h.sample_noalloc(c["chains"], c["burn"], c["sweeps"], state["seed"], precision, *state["out"])
        return state["out"]
    h.sample(c["chains"], c["burn"], c["sweeps"], state["seed"], precision=precision,
             moments=c["call"] == "gradient")
    if c["workload"] == "batch":
        each = [h.average(k) for k in range(len(h))]
        return {key: np.concatenate([r[key] for r in each]) for key in each[0]}
    out = h.average()
    if c["call"] == "gradient":
        out["grad_G"], out["grad_theta"] = h.backward(state["v"])
    elif c["call"] == "first_sweep":
        out["f"], out["chi2"] = h.chain_state()
    else:
        out["sem_binned"] = h.mc_error()["sem_fbar"]
    return out


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def _levels(c):
    """[(M, N, [blocks of each level])] of the problems of a case."""
    kind = c["workload"]
    if kind == "batch":   # the ranges' means: 100-1000 grid points, 50-200 times, blocks of 25-100
        return [(125, 550, [[550], [55] * 10])] * c["problems"]
    N = c["N"]
    if kind == "paper":
        parts = [list(l) + [N] for l in asm.partition_hierarchy(N)]
        return [(60, N, [np.diff(l).tolist() for l in parts])]
    if kind == "modes":
        return [(c["M"], N, [[N]])]
    k = {"grid": 16, "theta": 8}.get(kind) or c["blocks"]
    M = 400 if kind == "grid" else c["M"]
    return [(M, N, [[N]] if k == 1 else [[N], [N / k] * k])]


def work(case):
    """Per move of a block of n points: the step along the mode (2 n), the clamp,
    the ratio and the two bounds (4 n); per visit the projections of the residual
    on entry and exit (4 M min(M, n)).  Bytes: the factors once, the states, sums
    and results once."""
    c = case
    size = 4 if c["mixed"] else 8
    flops = nbytes = 0.0
    for M, N, levels in _levels(c):
        sweep = [sum(6 * n * n + 4 * M * min(M, n) for n in blocks) for blocks in levels]
        flops += c["chains"] * (c["burn"] + c["sweeps"]) * sum(sweep) / len(sweep)
        nbytes += sum(n * n + M * min(M, n) for blocks in levels for n in blocks) * size
        nbytes += c["chains"] * ((N + M) * size + 2 * N * 8) + 5 * N * 8
        if c["call"] == "gradient":   # snapshots every eight kept sweeps: f f^T, scores of 8 parameters
            flops += c["sweeps"] // 8 * c["chains"] * (N * N + 2.0 * 8 * M * N)
            nbytes += 8 * M * N * 8 + N * N * 8
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------
# the first sweep in 64 bits: numpy and torch alone
# --------------------------------------------------------------------------

def _philox(c0, c1, c2, c3, key):
    """Philox4x64-10 (Salmon et al. 2011) of one counter: four 64-bit words."""
    mask, k0, k1 = (1 << 64) - 1, key, 0
    for _ in range(10):
        a, b = 0xD2E7470EE14C6C93 * c0, 0xCA5A826395121157 * c2
        c0, c1, c2, c3 = (b >> 64) ^ c1 ^ k0, b & mask, (a >> 64) ^ c3 ^ k1, a & mask
        k0, k1 = (k0 + 0x9E3779B97F4A7C15) & mask, (k1 + 0xBB67AE8584CAA73B) & mask
    return c0, c1, c2, c3


def _truncated(mu, sd, lo, hi, u):
    """Inverse CDF at u of N(mu, sd^2) on [lo, hi]: the normal quantile where the
    centre lies well inside, else by bisection of the offset from the end nearer
    the centre, on log Q(a + y) / Q(a) through erfcx."""
    a, b = (lo - mu) / sd, (hi - mu) / sd
    q = torch.special.ndtr
    left, right = (1 - u) * q(a) + u * q(b), (1 - u) * q(-a) + u * q(-b)
    centre = torch.where(left <= 0.5, torch.special.ndtri(left), -torch.special.ndtri(right))
    inside = (a < -3.0) & (b > 3.0)
    a, b, w = torch.where(inside, 0.0, a), torch.where(inside, 1.0, b), torch.where(inside, 1.0, (hi - lo) / sd)
    flip = a + b < 0
    a, u = torch.where(flip, -b, a), torch.where(flip, 1 - u, u)

    def log_q(y):
        e = torch.special.erfcx
        return torch.log(e((a + y) / math.sqrt(2.0)) / e(a / math.sqrt(2.0))) - y * (a + 0.5 * y)

    mass = u * -torch.expm1(log_q(w))
    left, right = torch.zeros_like(w), w
    for _ in range(64):
        mid = 0.5 * (left + right)
        above = -torch.expm1(log_q(mid)) > mass
        left, right = torch.where(above, left, mid), torch.where(above, mid, right)
    y = 0.5 * (left + right) * sd
    return torch.where(inside, mu + sd * centre, torch.where(flip, hi - y, lo + y))


def exact(case, seed):
    if case["call"] != "first_sweep":
        return None   # the moves amplify a rounding a hundredfold per sweep: no value to compare with
    p = _problem(case, seed)
    F = _Factors(p)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    t = lambda x: torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device=dev)  # noqa: E731
    Q, (M, N) = case["chains"], p.K.shape
    Kt, gt = t(F.Kt), t(F.gt)
    k1 = Kt.sum(dim=1)
    f = torch.full((Q, N), float((k1 @ gt) / (k1 @ k1)), dtype=torch.float64, device=dev)
    word = _philox((1 << 64) - 1, 0, 0, 0, seed)[0]
    level = min(int(((word >> 12) + 0.5) * 2.0 ** -52 * len(p.levels)), len(p.levels) - 1)
    words = np.array([[x for i in range((N + 3) // 4) for x in _philox(i, 0, q, 0, seed)] for q in range(Q)], dtype=np.uint64)
    uniforms = t(((words >> np.uint64(12)).astype(np.float64) + 0.5) * 2.0 ** -52) if not case["mixed"] else \
        t(((words >> np.uint64(41)).astype(np.float64) + 0.5) * 2.0 ** -23)
    for lv, a, b, d, V, U in F.blocks:
        if lv != level:
            continue
        c, V = (gt - f @ Kt.T) @ t(U).T, t(V)
        x = f[:, a:b].clone()
        for j in range(b - a):
            v = V[j]
            use = v.abs() >= 2.0 ** -40 * v.abs().max()
            r = -x / v
            inf = torch.full_like(x, math.inf)
            lo = torch.where(use & (v > 0), r, -inf).amax(dim=1)
            hi = torch.where(use & (v < 0), r, inf).amin(dim=1)
            u = uniforms[:, a + j]
            if d[j] > 0.0:
                s = torch.full_like(u, 1.0 / d[j])
                mu = c[:, j] * s
                delta = _truncated(mu, s, torch.maximum(lo, torch.minimum(mu, hi) - 40.0 * s),   # no mass beyond
                                   torch.minimum(hi, torch.maximum(mu, lo) + 40.0 * s), u)
            else:
                delta = lo + u * (hi - lo)
            delta = torch.where(hi > lo, delta, torch.zeros_like(delta))
            x = (x + delta[:, None] * v).clamp(min=0.0)
        f[:, a:b] = x
    chi2 = ((gt - f @ Kt.T) ** 2).sum(dim=1)
    mean, w = f.mean(dim=0), t(p.w)
    sem = f.std(dim=0) / math.sqrt(Q) if Q > 1 else torch.full_like(mean, math.nan)
    var = (f ** 2).mean(dim=0) - mean ** 2
    out = {"mean_A": mean / w, "sem_A": sem / w, "ess": var.clamp(min=0.0) / sem ** 2, "mean_fbar": mean,
           "sem_fbar": sem, "f": f, "chi2": chi2}
    return {k: x.cpu().numpy() for k, x in out.items()}

