"""The FP32 draw's divisions by a value whose correctly rounded reciprocal is at hand
(div_by) against the correctly rounded quotient, bit for bit, over the ranges of the
three places that use it, and the narrow draw's start, which divides by a slope of any
size, against the same start with a plain division."""
import ctypes as ct
import subprocess

import numpy as np
import pytest

from paper_1912_01379_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "asm_sweep.cuh"
using namespace asmgb;
__global__ void quotients(const float *n, const float *d, float *got, float *want, int count)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    got[i] = div_by(n[i], d[i], __frcp_rn(d[i]));
    want[i] = __fdiv_rn(n[i], d[i]);
}
__global__ void starts(const float *a, const float *w, const float *u, float *got, float *want, int count)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    int capped = 0;
    got[i] = narrow_offset(a[i], w[i], u[i], capped);
    const float lam = a[i] + 0.5f * w[i], x = lam * w[i];
    const float t = __fdiv_rn(-m_log1p(u[i] * m_expm1(-x)), lam);
    want[i] = m_min(m_max(t, 0.0f), w[i]);
}
extern "C" int run(int kind, const float *x, const float *y, const float *z, float *got, float *want, int count)
{
    const int blocks = (count + 255) / 256;
    if (kind == 0) quotients<<<blocks, 256>>>(x, y, got, want, count);
    else starts<<<blocks, 256>>>(x, y, z, got, want, count);
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : -1;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("div")
    (d / "div.cu").write_text(SOURCE)
    subprocess.run([build.NVCC, *build.FLAGS, "-I", build.CSRC, "-shared", "-o", str(d / "div.so"), str(d / "div.cu")],
                   check=True)
    return ct.CDLL(str(d / "div.so"))


def _run(lib, kind, *arrays):
    import torch
    n = arrays[0].size
    t = [torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda() for a in arrays]
    out = torch.empty(2, n, dtype=torch.float32, device="cuda")
    ptr = [ct.c_void_p(x.data_ptr()) for x in (*t, *([t[0]] * (3 - len(t))), out[0], out[1])]
    torch.cuda.synchronize()
    assert lib.run(kind, *ptr, n) == 0
    got, want = out.cpu().numpy()
    assert np.all(np.isfinite(want))
    bad = got.view(np.int32) != want.view(np.int32)
    assert not bad.any(), (int(bad.sum()), [a[bad][:3] for a in arrays], got[bad][:3], want[bad][:3])


COUNT = 1 << 22


def test_quotients_over_the_ranges_in_use(lib):
    r = np.random.default_rng(1)
    sign = r.choice([-1.0, 1.0], COUNT)
    # the start: n = -log1p(u expm1(-x)), 2^-34 <= |n| < 1, over 1.4e-3 <= |lam| < 1e27
    _run(lib, 0, sign * np.exp2(r.uniform(-34, 0, COUNT)), sign * np.exp2(r.uniform(np.log2(1.4e-3), np.log2(1e27), COUNT)))
    # a Newton step: a small difference over a density in [e^-1/2, e^1/2]
    _run(lib, 0, sign * np.exp2(r.uniform(-83, 1, COUNT)), np.exp(r.uniform(-0.5, 0.5, COUNT)))
    # a ratio of erfcx values: the divisor down to 1e-25, the quotient near 1 or well below
    d = np.exp2(r.uniform(np.log2(1.0001e-25), -2, COUNT)).astype(np.float32)
    _run(lib, 0, d * np.exp2(r.uniform(-12, 2, COUNT)).astype(np.float32), d)


@pytest.mark.parametrize("lo,hi", [(1.4e-3, 1e3), (1e3, 1e26), (1e26, 1e28), (1e28, 1e30), (1e30, 1e34)])
def test_start_of_the_narrow_draw(lib, lo, hi):
    """Intervals so narrow that the start is the answer (w^2 <= 4e-7), slopes lam of few
    significant bits (quotients halfway between two subnormal numbers are then common)."""
    r = np.random.default_rng(2)
    a = np.exp2(np.floor(r.uniform(np.log2(lo), np.log2(hi) - 1, COUNT))) * (1 + 0.125 * r.integers(0, 8, COUNT))
    x = np.exp2(r.uniform(np.log2(1.1e-3), -1, COUNT)) * r.choice([1.0, 0.25, 1.0 / 64], COUNT)
    x = np.maximum(x, 1.1e-3)
    w = np.minimum(x / a, 6.3e-4)
    keep = a * w >= 1.1e-3
    u = (r.integers(0, 1 << 23, COUNT) + 0.5) * 2.0 ** -23
    u = np.where(r.random(COUNT) < 0.5, u * 2.0 ** -r.integers(0, 16, COUNT), u)
    u = (np.floor(u * 2 ** 23) + 0.5) * 2.0 ** -23
    sign = r.choice([-1.0, 1.0], COUNT)
    if keep.sum() == 0:
        pytest.fail("no draw of this range")
    _run(lib, 1, (sign * a)[keep], w[keep], u[keep])
