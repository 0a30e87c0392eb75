// asm_sweep.cuh -- the chain kernel of blocked modes sampling (Ghanem & Koch,
// arXiv:1912.01379, Sec. IV.B-C) for sm_103a.
//
// Layout.  A warp runs C chains (1, 2 or 4) of one problem.  While a block is
// visited, the block's part of each chain's state f is in registers, spread over
// the 32 lanes in 16-byte vectors (8-byte ones for small blocks).  Mode rows (V,
// and the masked reciprocals R = -1/V that give the bounds of Eq. modeLimits) are
// read as vectors from a CTA-shared ring of move records, once for the warp's C
// chains; every chain of the same problem reads the same rows at the same time.
// A block visit starts from its packet in shared memory (block descriptor, bounds
// row of the first mode, U_b).  The tracked residual r~ = g~ - K~ f and the
// block's projections c_j = U_j^T r~ live in shared memory, the chain state too
// where it fits.
//
// One move of mode j (Sec. IV.B, "sample e_i' from a univariate Gaussian ...
// truncated to the interval for which f' >= 0"):
//   [lo, hi]  = interval of delta from the previous pass (warp minima of the
//               bound keys, see BoundKey)
//   delta     ~ N(c_j/d_j, 1/d_j^2) on [lo, hi] by the inverse CDF (flat if d_j = 0)
//   pass      f += delta V_j, clamp at 0, and the bounds of mode j+1 in the same
//             sweep over the registers
//   w_j       = dres_j delta  (the residual moves by -w_j U_j, dres_j = |K~_b V_j|;
//               c_j is not needed again)
// Block entry computes c = U_b^T r~, block exit applies r~ -= U_b w.
#pragma once

#include <cuda_runtime.h>
#include <type_traits>
#include <math_constants.h>

#include "asm_internal.h"

namespace asmgb {

// --------------------------------------------------------------------------
// Philox4x64-10 (Salmon et al., SC'11): counter-based, so every move's uniform
// is a pure function of (seed, move, sweep, chain, problem).
// --------------------------------------------------------------------------
__device__ __forceinline__ void philox4x64_10(unsigned long long &c0, unsigned long long &c1,
                                              unsigned long long &c2, unsigned long long &c3,
                                              unsigned long long k0, unsigned long long k1)
{
    const unsigned long long M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
    const unsigned long long W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) { k0 += W0; k1 += W1; }
        const unsigned long long hi0 = __umul64hi(M0, c0), lo0 = M0 * c0;
        const unsigned long long hi1 = __umul64hi(M1, c2), lo1 = M1 * c2;
        const unsigned long long y0 = hi1 ^ c1 ^ k0, y2 = hi0 ^ c3 ^ k1;
        c0 = y0; c1 = lo1; c2 = y2; c3 = lo0;
    }
}

// u in (0,1) on the grid (k + 1/2) 2^-52 (FP64) or (k + 1/2) 2^-23 (FP32, the
// top 23 bits of the same word); 1 - u is exact in both.
template <class T> __device__ __forceinline__ T uniform_from(unsigned long long w);
template <> __device__ __forceinline__ double uniform_from<double>(unsigned long long w)
{
    return ((double)(w >> 12) + 0.5) * 0x1p-52;
}
template <> __device__ __forceinline__ float uniform_from<float>(unsigned long long w)
{
    return ((float)(unsigned)(w >> 41) + 0.5f) * 0x1p-23f;
}

// --------------------------------------------------------------------------
// math by precision (CUDA math library calls)
// --------------------------------------------------------------------------
__device__ __forceinline__ double m_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float m_fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double m_max(double a, double b) { return fmax(a, b); }
__device__ __forceinline__ float m_max(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ float m_min(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ float m_phi(float x) { return normcdff(x); }
__device__ __forceinline__ float m_phiinv(float p) { return normcdfinvf(p); }
__device__ __forceinline__ float m_erfcx(float x) { return erfcxf(x); }
__device__ __forceinline__ double m_log(double x) { return log(x); }
__device__ __forceinline__ float m_log(float x) { return logf(x); }
__device__ __forceinline__ float m_log1p(float x) { return log1pf(x); }
__device__ __forceinline__ float m_exp(float x) { return expf(x); }
__device__ __forceinline__ float m_expm1(float x) { return expm1f(x); }
__device__ __forceinline__ float m_abs(float x) { return fabsf(x); }

template <class T> struct TailTraits;
// far: with both standardized bounds beyond +-far, Phi(a) and 1 - Phi(b) are
// below half an ulp of the smallest uniform (2^-53 resp. 2^-24), so
// (1-u) Phi(a) + u Phi(b) rounds to u: Phi(-12) = 1.8e-33 < 2^-107 and
// Phi(-10) = 7.6e-24 < 2^-49.
template <> struct TailTraits<double> {
    static constexpr double tol = 1e-14;
    static constexpr int nmax = 40;
    static constexpr double far = 12.0;
};
template <> struct TailTraits<float> {
    static constexpr float tol = 2e-6f;
    static constexpr int nmax = 16;
    static constexpr float far = 10.0f;
};

// Gauss-Legendre rule on [-1, 1] (symmetric half: nodes x > 0 and weights;
// values of numpy.polynomial.legendre.leggauss).  8 points for FP64 (relative
// error ~2e-16 on the narrow intervals below), 4 points for FP32 (~2e-10).
template <class T> struct GaussLegendre;
template <> struct GaussLegendre<double> {
    static constexpr int half = 4;
    __device__ static constexpr double x(int i)
    {
        return i == 0 ? 0.18343464249564978 : i == 1 ? 0.525532409916329 : i == 2 ? 0.7966664774136267
                                                                                 : 0.9602898564975362;
    }
    __device__ static constexpr double w(int i)
    {
        return i == 0 ? 0.36268378337836166 : i == 1 ? 0.3137066458778869 : i == 2 ? 0.22238103445337443
                                                                                  : 0.10122853629037706;
    }
    static constexpr double tol = 4e-16;
    static constexpr int nmax = 40;
};
template <> struct GaussLegendre<float> {
    static constexpr int half = 2;
    __device__ static constexpr float x(int i) { return i == 0 ? 0.33998104358485626f : 0.8611363115940526f; }
    __device__ static constexpr float w(int i) { return i == 0 ? 0.6521451548625464f : 0.34785484513745357f; }
    static constexpr float tol = 4e-7f;
    static constexpr int nmax = 12;
};

// elements of a 16-byte vector
template <class T> struct VecOf;
template <> struct VecOf<float> { static constexpr int n = 4; };
template <> struct VecOf<double> { static constexpr int n = 2; };

// Bound keys.  With x >= +0 and R = -1/V (NaN where V is left out of the
// bounds), t = x R is <= -0 exactly when V > 0 (a lower-bound candidate for
// the step) and >= +0 when V < 0 (an upper-bound candidate).  Read as integers
// of the same width, the largest lower candidate is the SIGNED minimum of the
// bit patterns of all t (negative floats order by magnitude, above every
// negative the -inf of the initial key) and the smallest upper candidate the
// UNSIGNED minimum (negative floats and NaN lie above +inf).  One multiply and
// two integer minima per element, one R row instead of two.
template <class T> struct BoundKey;
template <> struct BoundKey<float> {
    using S = int;
    using U = unsigned;
    static constexpr S lo0 = (S)0xff800000;   // -inf
    static constexpr U hi0 = 0x7f800000u;     // +inf
    static __device__ __forceinline__ S bits(float x) { return __float_as_int(x); }
};
template <> struct BoundKey<double> {
    using S = long long;
    using U = unsigned long long;
    static constexpr S lo0 = (S)0xfff0000000000000ull;
    static constexpr U hi0 = 0x7ff0000000000000ull;
    static __device__ __forceinline__ S bits(double x) { return __double_as_longlong(x); }
};
// max(x, +0) (NaN gives +0).  FP64 as an integer test of the high word: a DSETP
// would occupy the FP64 pipe, which issues one warp instruction per 64 cycles and
// sub-partition, for as long as the fused multiply-add itself.
__device__ __forceinline__ float clamp0(float x) { return fmaxf(x, 0.0f); }
__device__ __forceinline__ double clamp0(double x)
{
    return (unsigned)__double2hiint(x) <= 0x7ff00000u ? x : 0.0;
}

// One vector of the pass: x = max(f + delta V, +0), f = x, and the keys of t = x R.
// The minima are exact, so the keys do not depend on the grouping.  FP32: the
// products and the fused multiply-adds in packed pairs (one instruction per two
// elements, each element rounded as by the scalar instruction), and three-way
// minima (0.63 issue slots of an SM per warp instruction against 0.41 for a
// two-way one that takes half as many elements).
template <class T>
struct Keys {
    typename BoundKey<T>::S l;
    typename BoundKey<T>::U h;
    __device__ __forceinline__ void reset()
    {
        l = BoundKey<T>::lo0;
        h = BoundKey<T>::hi0;
    }
    __device__ __forceinline__ void fold(typename BoundKey<T>::S &lk, typename BoundKey<T>::U &hk) const
    {
        lk = l;
        hk = h;
    }
    __device__ __forceinline__ void take(T t)
    {
        const typename BoundKey<T>::S k = BoundKey<T>::bits(t);
        const typename BoundKey<T>::U u = (typename BoundKey<T>::U)k;
        l = k < l ? k : l;
        h = u < h ? u : h;
    }
};
__device__ __forceinline__ void take2(Keys<float> &kk, float2 t)
{
    const int a = __float_as_int(t.x), b = __float_as_int(t.y);
    kk.l = __vimin3_s32(kk.l, a, b);
    kk.h = __vimin3_u32(kk.h, (unsigned)a, (unsigned)b);
}
template <int VE>
__device__ __forceinline__ void pass_chunk(float (&f)[VE], float delta, const float (&vv)[VE], const float (&rr)[VE],
                                           Keys<float> &kk)
{
    const float2 d2 = make_float2(delta, delta);
#pragma unroll
    for (int v = 0; v < VE; v += 2) {
        float2 a = __ffma2_rn(d2, make_float2(vv[v], vv[v + 1]), make_float2(f[v], f[v + 1]));
        a.x = clamp0(a.x);
        a.y = clamp0(a.y);
        f[v] = a.x;
        f[v + 1] = a.y;
        take2(kk, __fmul2_rn(a, make_float2(rr[v], rr[v + 1])));
    }
}
template <int VE>
__device__ __forceinline__ void pass_chunk(double (&f)[VE], double delta, const double (&vv)[VE], const double (&rr)[VE],
                                           Keys<double> &kk)
{
#pragma unroll
    for (int v = 0; v < VE; ++v) {
        f[v] = clamp0(fma(delta, vv[v], f[v]));
        kk.take(f[v] * rr[v]);
    }
}
// Keys alone (the first mode of a block: f is unchanged, t = f R).
template <int VE>
__device__ __forceinline__ void key_chunk(const float (&f)[VE], const float (&rr)[VE], Keys<float> &kk)
{
#pragma unroll
    for (int v = 0; v < VE; v += 2)
        take2(kk, __fmul2_rn(make_float2(f[v], f[v + 1]), make_float2(rr[v], rr[v + 1])));
}
template <int VE>
__device__ __forceinline__ void key_chunk(const double (&f)[VE], const double (&rr)[VE], Keys<double> &kk)
{
#pragma unroll
    for (int v = 0; v < VE; ++v) kk.take(f[v] * rr[v]);
}

// --------------------------------------------------------------------------
// bulk copies (TMA engine) and mbarriers, inline PTX
// --------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_addr(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_test_wait(unsigned long long *bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after `limit` polls (each poll may suspend briefly).
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity, int limit)
{
    for (int i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, unsigned long long *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// The warp's bounds from the lanes' keys: signed and unsigned integer minima,
// one redux instruction each (24 cycles, 26 for a pair in flight; with half-warp
// masks 168, which is why a chain always spans the warp).  FP64: the minimum of
// the high words, then of the low words of the lanes that hold it (a butterfly
// of 64-bit shuffles took five dependent steps of ~45 cycles).
template <int C>
__device__ __forceinline__ void warp_bounds(const int (&lk)[C], const unsigned (&hk)[C], float (&lo)[C], float (&hi)[C])
{
#pragma unroll
    for (int c = 0; c < C; ++c) {
        lo[c] = __int_as_float(__reduce_min_sync(0xffffffffu, lk[c]));
        hi[c] = __uint_as_float(__reduce_min_sync(0xffffffffu, hk[c]));
    }
}
template <int C>
__device__ __forceinline__ void warp_bounds(const long long (&lk)[C], const unsigned long long (&hk)[C], double (&lo)[C],
                                            double (&hi)[C])
{
    int lh[C];
    unsigned hh[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        lh[c] = __reduce_min_sync(0xffffffffu, (int)(lk[c] >> 32));
        hh[c] = __reduce_min_sync(0xffffffffu, (unsigned)(hk[c] >> 32));
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const unsigned ll = __reduce_min_sync(0xffffffffu, (int)(lk[c] >> 32) == lh[c] ? (unsigned)lk[c] : 0xffffffffu);
        const unsigned hl =
            __reduce_min_sync(0xffffffffu, (unsigned)(hk[c] >> 32) == hh[c] ? (unsigned)hk[c] : 0xffffffffu);
        lo[c] = __hiloint2double(lh[c], (int)ll);
        hi[c] = __hiloint2double((int)hh[c], (int)hl);
    }
}

// A value that is the same in all lanes, broadcast so that the compiler knows it too.
// Loop bounds and branch conditions read from shared memory count as divergent
// otherwise: every loop then carries reconvergence and every redux or shuffle a
// warp synchronisation.
template <class I>
__device__ __forceinline__ I uni(I x) { return __shfl_sync(0xffffffffu, x, 0); }

// lo < hi for bounds that come from keys: lo is -0 or below, hi +0 or above, neither
// is NaN, so they differ unless both are zeros.  FP64 as an integer test: a DSETP would
// occupy the FP64 pipe for 64 cycles.
__device__ __forceinline__ bool open_interval(float lo, float hi) { return hi > lo; }
__device__ __forceinline__ bool open_interval(double lo, double hi)
{
    return ((__double_as_longlong(lo) | __double_as_longlong(hi)) << 1) != 0;
}
__device__ __forceinline__ bool is_zero(float x) { return x == 0.0f; }
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ bool is_finite(float x) { return isfinite(x); }
__device__ __forceinline__ bool is_finite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// vector loads from shared memory: VE elements, naturally aligned
__device__ __forceinline__ void lds_v(const float *p, float (&o)[4])
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void lds_v(const float *p, float (&o)[2])
{
    const float2 v = *reinterpret_cast<const float2 *>(p);
    o[0] = v.x; o[1] = v.y;
}
__device__ __forceinline__ void lds_v(const double *p, double (&o)[2])
{
    const double2 v = *reinterpret_cast<const double2 *>(p);
    o[0] = v.x; o[1] = v.y;
}
__device__ __forceinline__ void lds_v(const double *p, double (&o)[1]) { o[0] = *p; }

// The mode data of a record: d_j, 1/d_j, dres_j.
__device__ __forceinline__ void lds_mode(const float *p, float &d, float &invd, float &dres)
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    d = v.x; invd = v.y; dres = v.z;
}
__device__ __forceinline__ void lds_mode(const double *p, double &d, double &invd, double &dres)
{
    const double2 v = *reinterpret_cast<const double2 *>(p);
    d = v.x; invd = v.y;
    dres = p[2];
}

// --------------------------------------------------------------------------
// The draw: delta ~ N(c/d, 1/d^2) restricted to [lo, hi] (lo < hi), by the inverse
// CDF at u.  In standard units x = d delta - c the interval is [a, b] =
// [d lo - c, d hi - c].  Each branch returns delta in the form that keeps delta - lo
// (or hi - delta) accurate relative to hi - lo.
//
// Narrow interval, w (|a| + w) <= 1/2 with w = b - a (the Gaussian nearly flat across
// it): the offset t from a solves I(t) = u I(w), I(t) = int_0^t exp(-a s - s^2/2) ds by
// Gauss-Legendre (accurate while t (|a| + t) <= 1/2), by Newton's method.  The start is
// the inverse CDF of the exponential law whose rate is the log-density's slope at the
// interval's midpoint, lam = a + w/2: the neglected curvature changes the log-density by
// at most w^2/8 across the interval, so one or two steps converge where the flat start
// t = u w needed four.  The offset keeps its relative accuracy however narrow the
// interval is.  In FP32 the start is the answer when w^2 / 8, the curvature's bound on
// the relative error of the exponential law's CDF, lies below 5e-8 (w <= 6e-4: the weak
// modes whose intervals are a tiny fraction of their Gaussian's width); with the series
// that stands for the exponential law below |lam w| = 1e-3 and leaves out terms of up to
// (lam w)^2 / 6 = 1.7e-7, the start is within 2.2e-7 relative (2.0e-7 measured at 2 million
// (a, w, u), 3.3e-8 beyond the series), half the FP32 tolerance.  One Newton
// step is the answer when w <= 0.2: Newton's error is quadratic in the start's, which is below
// w^2/12 relative, and one step leaves at most 1.5e-7 relative over the narrow regime
// with w <= 0.2 (measured against the root of a 64-point rule at 4 million (a, w, u)),
// below the FP32 tolerance.
//
// Tail, x in [a, a + w], a >= 0, 0 < w <= inf, by Q(x) = (1-u)Q(a) + uQ(b), b = a + w.
// The width comes in as w, formed from the interval's ends before they are
// standardised: b - a of two standardised ends far in the tail cancels (a = 35 and
// w = 0.03 leave w with a relative error of 2^-24 a / w = 7e-5 in FP32).  The equation
// in the offset y = x - a,
//   log Q(a + y) - log Q(a) = dt,  dt = log((1-u) + u Q(b)/Q(a)),
// is solved by Newton's method on log Q (concave, so the iterates are monotone after the
// first step), with Q(b)/Q(a) formed through erfcx to keep narrow intervals accurate.
// The start is the exponential tail's inverse for a >= 5 and, below,
// y = -Phi^{-1}(q) - a with q = (1-u)Q(a) + uQ(b): accurate to a few ulp of a, which
// FP32 keeps; in FP64 the offset form refines it so that y keeps its relative accuracy
// however small it is.  Otherwise x is the normal quantile of (1-u) Phi(a) + u Phi(b),
// taken from the side with the smaller mass.
//
// A warp holds C chains; every lane of the G = 32/C lanes of a chain's team has the same
// arguments, so the C draws of a move cost one.  The draw's independent function values
// go to different lanes: the pairs Phi(a), Phi(b) and erfcx(a), erfcx(b) are one call
// each, and in FP64 the exponentials of the quadratures at t and at w and of the density
// that Newton's step divides by are one exponential.  A warp instruction of the FP64 pipe
// takes 64 cycles of a sub-partition whether one lane is active or all are, so that is a
// quarter of the time of the scalar form (plain modes FP64, 50 points, 16 chains: 0.403
// -> 0.168 ms a sweep); in FP32 it shortens the instruction stream (the hierarchy of 64
// points, 1024 chains: 0.092 -> 0.071 ms a sweep).  Sums are formed from
// the lanes' values in one order for every team width, and products that could be fused
// either way are written out, so that a draw does not depend on C.
// --------------------------------------------------------------------------
template <int G>
struct TeamLanes {
    unsigned mask;   // lanes of the warp that run this path (whole teams)
    int base, gl;    // first lane of the team, lane within the team
    template <class T>
    __device__ __forceinline__ T from(T v, int l) const { return __shfl_sync(mask, v, base + l); }
};

// f(x0) and f(x1) from one call: the even lanes take x0, the odd ones x1.
template <int G, class T, class F>
__device__ __forceinline__ void pair_of(F f, T x0, T x1, const TeamLanes<G> &tl, T &y0, T &y1)
{
    const T y = f((tl.gl & 1) ? x1 : x0);
    y0 = tl.from(y, 0);
    y1 = tl.from(y, 1);
}

// ---- FP32 ----------------------------------------------------------------

// n / d, correctly rounded, from r = the correctly rounded 1 / d (Markstein 1990: the
// remainder is exact in a fused multiply-add; the second step makes it correct where the
// first product was off by more than an ulp).  For normal d, r and n / d, with |n| >= 2^-100,
// so that the remainder, a multiple of 2^-48 |n|, is a number too; or n = +0.  A subnormal
// quotient can lie halfway between two numbers, and then it came out an ulp off.
__device__ __forceinline__ float div_by(float n, float d, float r)
{
    const float q0 = __fmul_rn(n, r);
    const float q1 = __fmaf_rn(__fmaf_rn(-q0, d, n), r, q0);
    return __fmaf_rn(__fmaf_rn(-q1, d, n), r, q1);
}

// I(t) / (t/2) by the quadrature.
__device__ __forceinline__ float narrow_sum(float a, float t)
{
    using GL = GaussLegendre<float>;
    const float h = 0.5f * t;
    float acc = 0.0f;
#pragma unroll
    for (int i = 0; i < GL::half; ++i) {
        const float s1 = h * (1.0f - GL::x(i)), s2 = h * (1.0f + GL::x(i));
        acc = fmaf(GL::w(i), m_exp(-s1 * (a + 0.5f * s1)) + m_exp(-s2 * (a + 0.5f * s2)), acc);
    }
    return acc;
}

// The offset in a narrow interval.  Every lane evaluates the whole quadrature: four
// exponentials in flight together are no slower than one and the shuffles that would
// spread and collect them, and those of the target do not wait for the start.
__device__ __forceinline__ float narrow_offset(float a, float w, float u, int &capped)
{
    using GL = GaussLegendre<float>;
    const float lam = a + 0.5f * w;
    const float x = lam * w;
    // beyond the series the dividend is at least 2^-34 (u >= 2^-24, |x| >= 1e-3) and |lam| >= 1.4e-3
    // (w < 0.71): a normal quotient up to lam = 1e27
    float t = m_abs(x) < 1e-3f ? u * w * (1.0f - 0.5f * x * (1.0f - u))   // the series for small lam w
                               : m_abs(lam) < 1e27f ? div_by(-m_log1p(u * m_expm1(-x)), lam, __frcp_rn(lam))
                                                    : -m_log1p(u * m_expm1(-x)) / lam;
    t = m_min(m_max(t, 0.0f), w);
    if (w * w <= 4e-7f) return t;
    const float target = __fmul_rn(u, __fmul_rn(0.5f * w, narrow_sum(a, w)));
    int it = 0;
    for (; it < GL::nmax; ++it) {
        const float den = m_exp(-t * (a + 0.5f * t));   // in [e^-1/2, e^1/2]
        const float step = div_by(fmaf(0.5f * t, narrow_sum(a, t), -target), den, __frcp_rn(den));
        t = m_min(m_max(t - step, 0.0f), w);
        if (w <= 0.2f || m_abs(step) <= GL::tol * t || t == 0.0f) break;
    }
    if (it == GL::nmax) ++capped;
    return t;
}

// The offset in a tail beyond a = 5.
template <int G>
__device__ __forceinline__ float far_tail_team(float a, float w, float u, const TeamLanes<G> &tl, int &capped)
{
    const float b = a + w;
    const float kRsqrt2 = 0.70710678118654752440f;
    const float kSqrtPiOver2 = 1.25331413731550025121f;
    float exa, exb;
    pair_of<G>([](float z) { return m_erfcx(z); }, a * kRsqrt2, b * kRsqrt2, tl, exa, exb);
    float r = 0.0f, lr = 0.0f;
    if (!isinf(b)) {
        lr = m_log(exb / exa) - 0.5f * w * (a + b);
        r = m_exp(lr);
    }
    const float dt = r < 0.5f ? m_log((1.0f - u) + u * r) : m_log1p(u * m_expm1(lr));
    float y = -dt / a;
    const float inva = 1.0f / a, invx = __frcp_rn(exa);
    const bool plain = exa > 1e-25f;
    int it = 0;
    for (; it < TailTraits<float>::nmax; ++it) {
        const float exy = m_erfcx((a + y) * kRsqrt2);
        const float ratio = plain ? div_by(exy, exa, invx) : exy / exa;
        const float g = m_log(ratio) - y * (a + 0.5f * y) - dt;
        const float step = -g * exy * kSqrtPiOver2;   // g / g', g' = -sqrt(2/pi)/erfcx
        y -= step;
        if (m_abs(step) <= TailTraits<float>::tol * (y + inva)) break;
    }
    if (it == TailTraits<float>::nmax) ++capped;
    return m_min(m_max(y, 0.0f), w);
}

// The draw for the chains of a warp, FP32 (called by the whole warp; teams whose
// interval is not open return 0).  The branches that go through the normal quantile
// (the centre, tails nearer than 5, the interval that does not truncate) share one call
// of Phi for both ends and one quantile: the draw is most of the instructions of a
// workload with many Gaussian modes, and inlined per branch it overran the
// instruction cache.
template <int G>
__device__ __forceinline__ float draw_team(float c, float d, float invd, float lo, float hi, float u, bool open,
                                              int lane, int &capped)
{
    TeamLanes<G> tl;
    tl.base = lane & ~(G - 1);
    tl.gl = lane & (G - 1);
    const float a = m_fma(lo, d, -c);
    const float b = m_fma(hi, d, -c);
    const float wid = (hi - lo) * d;
    const bool narrow = open && isfinite(wid) && wid * (m_abs(a) + wid) <= 0.5f;
    const bool right = !narrow && a >= 0.0f, left = !narrow && !right && b <= 0.0f, tail = right || left;
    const float ta = right ? a : -b, tu = right ? u : 1.0f - u;   // the tail's near end and uniform
    const bool far = open && tail && ta >= 5.0f, quantile = open && !narrow && !far;
    const unsigned mn = __ballot_sync(0xffffffffu, narrow), mf = __ballot_sync(0xffffffffu, far),
                   mq = __ballot_sync(0xffffffffu, quantile);
    float delta = 0.0f;
    if (G == 32 ? mn != 0u : narrow) {   // one chain: uniform branches
        delta = lo + invd * narrow_offset(a, wid, u, capped);
    } else if (G == 32 ? mf != 0u : far) {
        tl.mask = mf;
        const float y = far_tail_team<G>(ta, wid, tu, tl, capped);
        delta = right ? lo + invd * y : hi - invd * y;
    } else if (G == 32 ? mq != 0u : quantile) {
        // both ends beyond: the truncation is below the resolution of u
        const bool untruncated = !tail && a < -TailTraits<float>::far && b > TailTraits<float>::far;
        float q = u <= 0.5f ? u : 1.0f - u;
        bool neg = u > 0.5f;
        tl.mask = __ballot_sync(mq, !untruncated);
        if (!untruncated) {
            const float tb = ta + wid;
            float A = tail ? -ta : a, B = tail ? -tb : b;
            const float v = tail ? tu : u;
            neg = tail;
            for (;;) {
                float pa, pb;
                pair_of<G>([](float z) { return m_phi(z); }, A, B, tl, pa, pb);
                if (tail && isinf(tb)) pb = 0.0f;
                // the larger half of the centre is taken from the other side: q and its mirror image
                // (1-v) pa + v pb; the mirror image rounds the other product first
                const bool mirror = neg && !tail;
                q = fmaf(mirror ? v : 1.0f - v, mirror ? pb : pa, __fmul_rn(mirror ? 1.0f - v : v, mirror ? pa : pb));
                const bool again = !neg && q > 0.5f;
                tl.mask = __ballot_sync(tl.mask, again);
                if (!again) break;
                A = -a;
                B = -b;
                neg = true;
            }
        }
        const float z = m_phiinv(q), x = neg ? -z : z;
        if (tail) {
            const float y = m_min(m_max(x - ta, 0.0f), wid);
            delta = right ? lo + invd * y : hi - invd * y;
        } else {
            delta = (x + c) * invd;
        }
    }
    return open ? m_min(m_max(delta, lo), hi) : 0.0f;
}

// ---- FP64 ----------------------------------------------------------------

// 1 - x or 1 + x of the quadrature node of a lane: lanes 2i, 2i + 1 of eight take node i.
__device__ __forceinline__ double gl_node(int lane)
{
    using GL = GaussLegendre<double>;
    const int i = (lane >> 1) & 3;
    const double lo = i == 0 ? 1.0 - GL::x(0) : i == 1 ? 1.0 - GL::x(1) : i == 2 ? 1.0 - GL::x(2) : 1.0 - GL::x(3);
    const double hi = i == 0 ? 1.0 + GL::x(0) : i == 1 ? 1.0 + GL::x(1) : i == 2 ? 1.0 + GL::x(2) : 1.0 + GL::x(3);
    return (lane & 1) ? hi : lo;
}

// sum_i w_i (e_{2i} + e_{2i+1}) from the exponentials held by lanes first .. first + 7 of the team.
template <int G>
__device__ __forceinline__ double gl_sum(const TeamLanes<G> &tl, double e, int first)
{
    using GL = GaussLegendre<double>;
    const double pair = e + __shfl_xor_sync(tl.mask, e, 1);
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < GL::half; ++i) acc = fma(GL::w(i), tl.from(pair, first + 2 * i), acc);
    return acc;
}

template <int G>
__device__ __forceinline__ double narrow_offset_team(double a, double w, double u, const TeamLanes<G> &tl, int &capped)
{
    using GL = GaussLegendre<double>;
    const double lam = a + 0.5 * w;
    const double x = lam * w;
    double t = fabs(x) < 1e-3 ? u * w * (1.0 - 0.5 * x * (1.0 - u)) : -log1p(u * expm1(-x)) / lam;
    t = fmin(fmax(t, 0.0), w);
    const double node = gl_node(tl.gl);
    double target = 0.0;
    bool live = true;
    for (int it = 0; it < GL::nmax; ++it) {
        // lanes 0-7: the nodes of I(t); lane 8 (teams of 16 and 32): the density at t;
        // the first time also I(w) for the target, on lanes 16-23 of a team of 32
        double acc, den;   // I(t) = t/2 acc
        if (G == 32) {
            const bool at_w = it == 0 && (tl.gl & 16);
            const double h = 0.5 * (at_w ? w : t);
            const double s = tl.gl == 8 ? t : h * node;
            const double e = exp(-s * fma(0.5, s, a));
            if (it == 0) target = __dmul_rn(u, __dmul_rn(0.5 * w, gl_sum<G>(tl, e, 16)));
            den = tl.from(e, 8);
            acc = gl_sum<G>(tl, e, 0);
        } else {
            if (it == 0) {
                const double s = 0.5 * w * node;
                target = __dmul_rn(u, __dmul_rn(0.5 * w, gl_sum<G>(tl, exp(-s * fma(0.5, s, a)), 0)));
            }
            const double s = G > 8 && tl.gl == 8 ? t : 0.5 * t * node;
            const double e = exp(-s * fma(0.5, s, a));
            den = G > 8 ? tl.from(e, G > 8 ? 8 : 0) : exp(-t * fma(0.5, t, a));
            acc = gl_sum<G>(tl, e, 0);
        }
        if (live) {
            const double step = (__dmul_rn(0.5 * t, acc) - target) / den;
            t = fmin(fmax(t - step, 0.0), w);
            if (fabs(step) <= GL::tol * t || t == 0.0) live = false;
        }
        if (!__any_sync(tl.mask, live)) break;
    }
    if (live) ++capped;
    return t;
}

template <int G>
__device__ __forceinline__ double right_tail_team(double a, double w, double u, TeamLanes<G> tl, int &capped)
{
    const double b = a + w;
    const double kRsqrt2 = 0.70710678118654752440;
    const double kSqrtPiOver2 = 1.25331413731550025121;
    double y = 0.0;
    const unsigned all = tl.mask, near = __ballot_sync(all, a < 5.0), refine = __ballot_sync(all, a > 0.0);
    if (a < 5.0) {
        double qa, qb;
        tl.mask = near;
        pair_of<G>([](double z) { return normcdf(z); }, -a, -b, tl, qa, qb);
        if (isinf(b)) qb = 0.0;
        const double q = (1.0 - u) * qa + u * qb;
        y = -normcdfinv(q) - a;
    }
    if (a > 0.0) {
        double exa, exb;
        tl.mask = refine;
        pair_of<G>([](double z) { return erfcx(z); }, a * kRsqrt2, b * kRsqrt2, tl, exa, exb);
        double r = 0.0, lr = 0.0;
        if (!isinf(b)) {
            lr = log(exb / exa) - 0.5 * w * (a + b);
            r = exp(lr);
        }
        const double dt = r < 0.5 ? log((1.0 - u) + u * r) : log1p(u * expm1(lr));
        if (a >= 5.0) y = -dt / a;
        int it = 0;
        for (; it < TailTraits<double>::nmax; ++it) {
            const double exy = erfcx((a + y) * kRsqrt2);
            const double g = log(exy / exa) - y * (a + 0.5 * y) - dt;
            const double step = -g * exy * kSqrtPiOver2;   // g / g', g' = -sqrt(2/pi)/erfcx
            y -= step;
            if (fabs(step) <= TailTraits<double>::tol * (y + 1.0 / a)) break;
        }
        if (it == TailTraits<double>::nmax) ++capped;
    }
    y = fmax(y, 0.0);
    y = fmin(y, w);
    return y;
}

// The draw for the chains of a warp, FP64 (called by the whole warp; teams whose
// interval is not open return 0).
template <int G>
__device__ __forceinline__ double draw_team(double c, double d, double invd, double lo, double hi, double u, bool open,
                                               int lane, int &capped)
{
    TeamLanes<G> tl;
    tl.base = lane & ~(G - 1);
    tl.gl = lane & (G - 1);
    const double a = fma(lo, d, -c);
    const double b = fma(hi, d, -c);
    const double wid = (hi - lo) * d;
    const bool narrow = open && is_finite(wid) && wid * (fabs(a) + wid) <= 0.5;
    const bool right = open && !narrow && a >= 0.0;
    const bool left = open && !narrow && !right && b <= 0.0;
    const bool middle = open && !narrow && !right && !left;
    const bool untruncated = middle && a < -TailTraits<double>::far && b > TailTraits<double>::far;
    double delta = 0.0;
    const unsigned mn = __ballot_sync(0xffffffffu, narrow), mt = __ballot_sync(0xffffffffu, right || left),
                   mc = __ballot_sync(0xffffffffu, middle && !untruncated);
    if (narrow) {
        tl.mask = mn;
        delta = lo + invd * narrow_offset_team<G>(a, wid, u, tl, capped);
    } else if (right || left) {
        tl.mask = mt;
        const double y = right_tail_team<G>(right ? a : -b, wid, right ? u : 1.0 - u, tl, capped);
        delta = right ? lo + invd * y : hi - invd * y;
    } else if (untruncated) {
        // the truncation is below the resolution of u: the untruncated inverse CDF
        const double x = u <= 0.5 ? normcdfinv(u) : -normcdfinv(1.0 - u);
        delta = (x + c) * invd;
    } else if (middle) {
        double pa, pb, x;
        tl.mask = mc;
        pair_of<G>([](double z) { return normcdf(z); }, a, b, tl, pa, pb);
        const double p = fma(1.0 - u, pa, __dmul_rn(u, pb));
        tl.mask = __ballot_sync(mc, p > 0.5);
        if (p > 0.5) {
            double na, nb;
            pair_of<G>([](double z) { return normcdf(z); }, -a, -b, tl, na, nb);
            x = -normcdfinv(fma(u, nb, __dmul_rn(1.0 - u, na)));
        } else {
            x = normcdfinv(p);
        }
        delta = (x + c) * invd;
    }
    return open ? fmin(fmax(delta, lo), hi) : 0.0;
}

// The launch's sweep range, read from the device control block.
struct SweepRange {
    long long sweep0, nsweeps, burn_in;
};

// A warp's position in the record ring and in the ring of visit packets (kept
// incrementally: no division per move).
struct RingPos {
    unsigned g;             // record stages so far in this launch
    int slot;
    unsigned phase;
    unsigned pg;            // visit packets so far
    int pslot;
    unsigned pphase;
};

__device__ __forceinline__ void ring_next(RingPos &r, int depth)
{
    ++r.g;
    if (++r.slot == depth) {
        r.slot = 0;
        r.phase ^= 1u;
    }
}
__device__ __forceinline__ void packet_next(RingPos &r, int slots)
{
    ++r.pg;
    if (++r.pslot == slots) {
        r.pslot = 0;
        r.pphase ^= 1u;
    }
}

// Whether a block's U comes with its visit packet, and the packet's bytes.
template <class T>
__device__ __forceinline__ bool u_staged(const LaunchShape &sh, int pkn)
{
    return pkn <= sh.pbytes / (int)sizeof(T);
}
template <class T>
__device__ __forceinline__ unsigned packet_bytes(const LaunchShape &sh, int pkn, int rs)
{
    return u_staged<T>(sh, pkn) ? (unsigned)(pkn * sizeof(T) + 15) & ~15u : (unsigned)((kPacketHeader + rs) * sizeof(T));
}
// Streamed U: columns of an entry tile (modes; 32, or fewer for small blocks) and rows per ring stage.
__device__ __forceinline__ int entry_width(int np) { return np > 16 ? 32 : np > 8 ? 16 : np > 4 ? 8 : 4; }
template <class T>
__device__ __forceinline__ int stream_rows(int stage_bytes, int width)
{
    return (stage_bytes / (int)(width * sizeof(T))) & ~7;
}
// Records of a block per ring stage: floor(stage / record) by the block's reciprocal (an
// integer division costs each visit of a small block about as much as a flat move).  The
// product is off by less than 64 2^-23, and a quotient that is not whole stays 1/4100 (the
// longest record) away from the next whole number, so 1e-4 makes the floor exact.
template <class T>
__device__ __forceinline__ int records_per_stage(const LaunchShape &sh, float inv_rec)
{
    return min(kMaxRecordsPerStage, (int)((float)(sh.stage_bytes / (int)sizeof(T)) * inv_rec + 1e-4f));
}

__device__ __forceinline__ int level_of_sweep(long long s, unsigned long long seed, unsigned long long pid,
                                              int n_levels)
{
    unsigned long long l0 = ~0ull, l1 = (unsigned long long)s, l2 = 0ull, l3 = pid;
    philox4x64_10(l0, l1, l2, l3, seed, 0ull);
    int level = (int)(uniform_from<double>(l0) * n_levels);
    return level >= n_levels ? n_levels - 1 : level;
}

// Arrival by lane 0 of the warp only, as a predicated instruction (no branch).
__device__ __forceinline__ void mbar_arrive_lane0(unsigned long long *bar, int lane)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.eq.s32 p, %1, 0;\n\t"
        "@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(smem_addr(bar)),
        "r"(lane)
        : "memory");
}
// Wait of a whole warp: true once the phase has completed, decided warp-wide.
__device__ __forceinline__ bool warp_wait(unsigned long long *bar, unsigned parity, int limit)
{
    bool ok = mbar_test_wait(bar, parity);
    if (__any_sync(0xffffffffu, !ok)) {
        ok = ok || mbar_wait(bar, parity, limit);
        if (__any_sync(0xffffffffu, !ok)) return false;
    }
    return true;
}

// Shared-memory regions of a CTA.
struct Regions {
    unsigned long long *full, *empty, *pfull, *pempty;
    unsigned char *stages, *packets;
};

// --------------------------------------------------------------------------
// The producer warp.  Per block visit one bulk copy of the visit packet (block
// descriptor, bounds row of the first mode, U where it fits) into the next
// packet slot, then the block's move records, as many to a ring stage as fit,
// one bulk copy per stage, before and after them the tiles of U for the
// projections where it did not fit; each copy after every consumer warp has
// released the slot's previous contents.  Lane 0 issues; the lanes hold the
// descriptors of the next 32 blocks of the level, read while the copies before
// them are issued (a descriptor read from global memory per visit made the
// producer the slowest warp of a level of one-point blocks).  The ring positions
// run on across the CTA's items.
// --------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ void produce(const SweepParams<T> &p, const LaunchShape &sh, const SweepRange &rg,
                                        const Regions &R, RingPos &rp, bool &failed)
{
    const long long nsweeps = uni(rg.nsweeps), sweep0 = uni(rg.sweep0);
    if (nsweeps <= 0 || failed || sh.stall) return;
    const int lane = threadIdx.x & 31;
    const int D = sh.depth, P = sh.pslots, M = uni(p.M);
    const unsigned g0 = rp.g, pg0 = rp.pg;
    // the blocks [base, base + 32) of sweep s, lane i's in B
    struct Batch {
        long long s;
        int base, nb, first;
        BlockDesc B;
    };
    auto load = [&](Batch &b) {   // the batch's descriptors (read-only data)
        const int i = min(b.base + lane, b.nb - 1);
        b.B = p.blocks[b.first + i];
    };
    auto start = [&](Batch &b, long long s) {
        const int level = level_of_sweep(s, p.seed, p.problem_id, p.n_levels);
        b.s = s;
        b.base = 0;
        b.nb = uni(p.level_nblocks[level]);
        b.first = uni(p.level_first[level]);
        load(b);
    };
    auto advance = [&](Batch &b) {
        b.base += 32;
        if (b.base < b.nb) load(b);
        else if (b.s + 1 < sweep0 + nsweeps) start(b, b.s + 1);
        else b.s = -1;
    };
    // one bulk copy into the next ring stage (lane 0)
    auto stage = [&](const T *src, unsigned bytes) {
        if (failed || (rp.g >= (unsigned)D && !mbar_wait(R.empty + rp.slot, rp.phase ^ 1u, sh.wait_limit))) {
            failed = true;
            return;
        }
        mbar_expect_tx(R.full + rp.slot, bytes);
        bulk_g2s(R.stages + (size_t)rp.slot * sh.stage_bytes, src, bytes, R.full + rp.slot);
        ring_next(rp, D);
    };
    // tiles of a streamed projection: columns [32 t, 32 t + width) x K rows, tile after tile
    auto stream = [&](const T *src, int K, int cols, int width) {
        const int rows = stream_rows<T>(sh.stage_bytes, width);
        for (int col0 = 0; col0 < cols && !failed; col0 += 32)
            for (int k = 0; k < K && !failed; k += rows) {
                const int n = min(rows, K - k);
                stage(src, (unsigned)(n * width * sizeof(T)));
                src += (size_t)n * width;
            }
    };
    Batch cur;
    start(cur, sweep0);
    while (cur.s >= 0 && !failed) {
        // this batch's blocks: what lane 0 needs of each, from its lane
        const int count = min(32, cur.nb - cur.base);
        const int n_ = cur.B.n, np_ = cur.B.np, rb_ = cur.B.recstride * (int)sizeof(T);
        const int rps_ = records_per_stage<T>(sh, cur.B.inv_rec);
        const unsigned pb_ = packet_bytes<T>(sh, cur.B.pkn, cur.B.rs);
        const int staged_ = u_staged<T>(sh, cur.B.pkn);
        const long long pk_ = cur.B.offPk, rec_ = cur.B.offRec, ue_ = cur.B.offUe, ux_ = cur.B.offUx;
        advance(cur);   // in flight while the copies of this batch are issued
        for (int i = 0; i < count && !failed; ++i) {
            const int n = __shfl_sync(0xffffffffu, n_, i), rps = __shfl_sync(0xffffffffu, rps_, i),
                      rb = __shfl_sync(0xffffffffu, rb_, i), staged = __shfl_sync(0xffffffffu, staged_, i);
            const unsigned pb = __shfl_sync(0xffffffffu, pb_, i);
            const long long pk = __shfl_sync(0xffffffffu, pk_, i), rec = __shfl_sync(0xffffffffu, rec_, i);
            int np = 0;
            long long ue = 0, ux = 0;
            if (!staged) {
                np = __shfl_sync(0xffffffffu, np_, i);
                ue = __shfl_sync(0xffffffffu, ue_, i);
                ux = __shfl_sync(0xffffffffu, ux_, i);
            }
            if (lane == 0) {
                if (rp.pg >= (unsigned)P && !mbar_wait(R.pempty + rp.pslot, rp.pphase ^ 1u, sh.wait_limit)) {
                    failed = true;
                } else {
                    mbar_expect_tx(R.pfull + rp.pslot, pb);
                    bulk_g2s(R.packets + (size_t)rp.pslot * sh.pbytes, p.pd.pk + pk, pb, R.pfull + rp.pslot);
                    packet_next(rp, P);
                }
                if (!staged) stream(p.pd.Ue + ue, M, np, entry_width(np));
                const char *src = reinterpret_cast<const char *>(p.pd.rec + rec);
                for (int j = 0; j < n && !failed; j += rps) {
                    const unsigned bytes = (unsigned)(min(rps, n - j) * rb);
                    stage(reinterpret_cast<const T *>(src), bytes);
                    src += bytes;
                }
                if (!staged) stream(p.pd.Ux + ux, np, M, 32);
            }
            failed = uni((int)failed) != 0;
        }
    }
    if (failed && lane == 0) {
        // the copies already issued must land before the CTA may exit
        const unsigned from = rp.g > g0 + (unsigned)D ? rp.g - D : g0;
        for (unsigned k = from; k < rp.g; ++k)
            mbar_wait(R.full + (k % (unsigned)D), (k / (unsigned)D) & 1u, sh.wait_limit);
        const unsigned pfrom = rp.pg > pg0 + (unsigned)P ? rp.pg - P : pg0;
        for (unsigned k = pfrom; k < rp.pg; ++k)
            mbar_wait(R.pfull + (k % (unsigned)P), (k / (unsigned)P) & 1u, sh.wait_limit);
        atomicAdd(&p.counters->timeouts, 1ull);
    }
    __syncwarp();
}

// The C chains of a consumer warp: shared memory and state of each.
template <class T, int C>
struct WarpChains {
    long long q[C];        // local chain (idle ones shadow the last chain and write nothing)
    bool active[C];
    T *sm;                 // chain 0's shared memory; chain c at sm + c * team_words
    int tw;
    int off_r, off_u, off_f, off_p;   // words: c and w at 0, r~, uniforms, f, sums
    __device__ __forceinline__ T *c_(int c) const { return sm + (size_t)c * tw; }
    __device__ __forceinline__ T *w_(int c) const { return c_(c); }
    __device__ __forceinline__ T *r_(int c) const { return c_(c) + off_r; }
    __device__ __forceinline__ T *u_(int c) const { return c_(c) + off_u; }
};

// Move counts of a warp's chains in one launch (at most 64 sweeps): degenerate Gaussian
// moves, flat moves made, non-finite steps, rejections; and the flat moves in all.
template <int C>
struct MoveCounts {
    unsigned deg[C], zero[C], bad[C], rej[C], flat;
    int capped;
};

// c = U_b^T r~ for the warp's chains: partial sum i of eight takes the terms m = i mod 8
// in increasing m, the rest goes to sum 0, then a fixed tree; so the sums are the same for
// any C, from a packet or streamed.  Blocks of up to eight modes spread the eight
// partial sums over lanes (four modes at a time): with a lane per mode most lanes idle.
// FP32: U's rows in the packet are 4 x odd elements apart, so that 16-byte loads of a row per
// lane meet no bank conflict (hierarchy of 64 points, 1024 chains: 0.0693 -> 0.0650 ms a sweep).
template <class T, int C>
__device__ __forceinline__ void project_entry(const WarpChains<T, C> &wc, const T *Us, int np, int usr, int M, int lane)
{
    constexpr int VEC = VecOf<T>::n;
    if (np <= 8) {
        const int i = lane & 7, m8 = M & ~7;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const T *r = wc.r_(c);
            for (int j0 = 0; j0 < np; j0 += 4) {
                const int j = j0 + (lane >> 3);
                const T *u = Us + (size_t)min(j, np - 1) * usr;
                T tu[7], tr[7];   // the last M mod 8 terms, loaded ahead
#pragma unroll
                for (int k = 0; k < 7; ++k) {
                    const bool in = i == 0 && m8 + k < M;
                    tu[k] = in ? u[m8 + k] : T(0);
                    tr[k] = in ? r[m8 + k] : T(0);
                }
                T a = T(0);
#pragma unroll 8
                for (int m = i; m < m8; m += 8) a = m_fma(u[m], r[m], a);
#pragma unroll
                for (int k = 0; k < 7; ++k)
                    if (i == 0 && m8 + k < M) a = m_fma(tu[k], tr[k], a);
                a += __shfl_xor_sync(0xffffffffu, a, 1);
                a += __shfl_xor_sync(0xffffffffu, a, 2);
                a += __shfl_xor_sync(0xffffffffu, a, 4);
                if (i == 0 && j < np) wc.c_(c)[j] = a;
            }
        }
        return;
    }
    constexpr int JJ = C == 1 ? 2 : 1;   // modes of a lane at a time
    for (int j = lane; j < np; j += 32 * JJ) {
        T a[C * JJ][8];
#pragma unroll
        for (int x = 0; x < C * JJ; ++x)
#pragma unroll
            for (int i = 0; i < 8; ++i) a[x][i] = T(0);
        const T *u[JJ];
#pragma unroll
        for (int x = 0; x < JJ; ++x) u[x] = Us + (size_t)(j + 32 * x < np ? j + 32 * x : j) * usr;
        int m = 0;
        for (; m + 7 < M; m += 8) {
#pragma unroll
            for (int v = 0; v < 8; v += VEC) {
                T r[C][VEC];
#pragma unroll
                for (int c = 0; c < C; ++c) lds_v(wc.r_(c) + m + v, r[c]);
#pragma unroll
                for (int x = 0; x < JJ; ++x) {
                    T uu[VEC];
                    if constexpr (sizeof(T) == 4) {
                        lds_v(u[x] + m + v, uu);
                    } else {   // rows of an odd stride
#pragma unroll
                        for (int k = 0; k < VEC; ++k) uu[k] = u[x][m + v + k];
                    }
#pragma unroll
                    for (int k = 0; k < VEC; ++k)
#pragma unroll
                        for (int c = 0; c < C; ++c) a[c * JJ + x][v + k] = m_fma(uu[k], r[c][k], a[c * JJ + x][v + k]);
                }
            }
        }
        for (; m < M; ++m)
#pragma unroll
            for (int c = 0; c < C; ++c)
#pragma unroll
                for (int x = 0; x < JJ; ++x) a[c * JJ + x][0] = m_fma(u[x][m], wc.r_(c)[m], a[c * JJ + x][0]);
#pragma unroll
        for (int c = 0; c < C; ++c)
#pragma unroll
            for (int x = 0; x < JJ; ++x) {
                const T(&b)[8] = a[c * JJ + x];
                if (x == 0 || j + 32 * x < np)
                    wc.c_(c)[j + 32 * x] = ((b[0] + b[1]) + (b[2] + b[3])) + ((b[4] + b[5]) + (b[6] + b[7]));
            }
    }
}

// r~ -= U_b w for the warp's chains (lanes split the data points; partial sum i of eight
// takes the modes j = i mod 8 as at entry).
template <class T, int C>
__device__ __forceinline__ void project_exit(const WarpChains<T, C> &wc, const T *Us, int np, int usr, int M, int lane)
{
    constexpr int VEC = VecOf<T>::n;
    constexpr int MM = C == 1 ? 2 : 1;   // data points of a lane at a time
    for (int m = lane; m < M; m += 32 * MM) {
        T a[C * MM][8];
#pragma unroll
        for (int x = 0; x < C * MM; ++x)
#pragma unroll
            for (int i = 0; i < 8; ++i) a[x][i] = T(0);
        int mm[MM];
#pragma unroll
        for (int x = 0; x < MM; ++x) mm[x] = m + 32 * x < M ? m + 32 * x : m;
        int j = 0;
        for (; j + 7 < np; j += 8) {
            const T *u = Us + (size_t)j * usr;
#pragma unroll
            for (int v = 0; v < 8; v += VEC) {
                T w[C][VEC];
#pragma unroll
                for (int c = 0; c < C; ++c) lds_v(wc.w_(c) + j + v, w[c]);
#pragma unroll
                for (int k = 0; k < VEC; ++k)
#pragma unroll
                    for (int x = 0; x < MM; ++x) {
                        const T uu = u[(v + k) * usr + mm[x]];
#pragma unroll
                        for (int c = 0; c < C; ++c) a[c * MM + x][v + k] = m_fma(uu, w[c][k], a[c * MM + x][v + k]);
                    }
            }
        }
        for (; j < np; ++j)
#pragma unroll
            for (int c = 0; c < C; ++c)
#pragma unroll
                for (int x = 0; x < MM; ++x)
                    a[c * MM + x][0] = m_fma(Us[(size_t)j * usr + mm[x]], wc.w_(c)[j], a[c * MM + x][0]);
#pragma unroll
        for (int c = 0; c < C; ++c)
#pragma unroll
            for (int x = 0; x < MM; ++x) {
                const T(&b)[8] = a[c * MM + x];
                if (x == 0 || m + 32 * x < M)
                    wc.r_(c)[m + 32 * x] -= ((b[0] + b[1]) + (b[2] + b[3])) + ((b[4] + b[5]) + (b[6] + b[7]));
            }
    }
}

// The columns of a projection whose U does not fit a packet, streamed through the record
// ring in tiles of 32 columns (lane = column): sum over the K rows k of U[k][col] vec[k],
// partial sum i of eight taking the rows k = i mod 8, the rest to sum 0, as above; stored
// to out (entry) or subtracted from it (exit).  vec and out are chain 0's, chain c's lie
// c tw elements on.  Every warp of the CTA reads the same stage; reads of U from global
// memory by each warp were bound by their latency with eight loads in flight per lane
// (N = 2000, M = 400, 2048 chains, U of 0.2 MB for a block of 125 points and 0.64 MB for
// the whole grid: 2.39 ms a sweep, 1.35 streamed; 24 problems of 100 to 1000 points: 0.382,
// 0.313).  Not inlined, so that kernels whose blocks bring U with their packets keep
// their instruction cache.  In and out: the ring position (stage, phase); ok: no bounded
// wait gave up.
struct StreamPos {
    int slot;
    unsigned phase;
    bool ok;
};
template <class T, int C>
__device__ __noinline__ StreamPos project_stream(const T *vec, T *out, int tw, bool subtract, unsigned long long *full,
                                                 unsigned long long *empty, const unsigned char *stages, int stage_bytes,
                                                 int depth, int wait_limit, int K, int cols, int width, StreamPos at)
{
    constexpr int VEC = VecOf<T>::n;
    const int lane = threadIdx.x & 31;
    const int rows = stream_rows<T>(stage_bytes, width);
    for (int col0 = 0; col0 < cols; col0 += 32) {
        T a[C][8];
#pragma unroll
        for (int c = 0; c < C; ++c)
#pragma unroll
            for (int i = 0; i < 8; ++i) a[c][i] = T(0);
        for (int k = 0; k < K;) {
            if (!warp_wait(full + at.slot, at.phase, wait_limit)) {
                at.ok = false;
                return at;
            }
            const T *u = reinterpret_cast<const T *>(stages + (size_t)at.slot * stage_bytes) + (lane < width ? lane : 0);
            const int kend = min(K, k + rows);
#pragma unroll 2
            for (; k + 7 < kend; k += 8, u += 8 * width) {
#pragma unroll
                for (int v = 0; v < 8; v += VEC) {
                    T x[C][VEC];
#pragma unroll
                    for (int c = 0; c < C; ++c) lds_v(vec + c * tw + k + v, x[c]);
#pragma unroll
                    for (int i = 0; i < VEC; ++i) {
                        const T uu = u[(v + i) * width];
#pragma unroll
                        for (int c = 0; c < C; ++c) a[c][v + i] = m_fma(uu, x[c][i], a[c][v + i]);
                    }
                }
            }
            for (; k < kend; ++k, u += width)
#pragma unroll
                for (int c = 0; c < C; ++c) a[c][0] = m_fma(u[0], vec[c * tw + k], a[c][0]);
            __syncwarp();
            mbar_arrive_lane0(empty + at.slot, lane);
            if (++at.slot == depth) {
                at.slot = 0;
                at.phase ^= 1u;
            }
        }
        const int col = col0 + lane;
        if (col < cols) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const T x = ((a[c][0] + a[c][1]) + (a[c][2] + a[c][3])) + ((a[c][4] + a[c][5]) + (a[c][6] + a[c][7]));
                if (subtract) out[c * tw + col] -= x;
                else out[c * tw + col] = x;
            }
        }
    }
    return at;
}

// --------------------------------------------------------------------------
// The moves of one block visit.  Lane l holds the elements VE (32 k + l) + v of
// the block, k < KK, v < VE, of each of the warp's C chains.  VE = VEC (16-byte
// vectors), or half of that for blocks of at most 16 VEC points, whose rows
// would fill only half the lanes.  KC = KK chunks known to be present, or 0: each
// of KV is tested (uniformly) against kcnt.
// --------------------------------------------------------------------------
template <class T, int KV, int C, bool PRIOR, int KC, int VE>
struct Visit {
    static constexpr int KK = KC ? KC : KV;
    static constexpr bool CHK = KC == 0;
    using KS = typename BoundKey<T>::S;
    using KU = typename BoundKey<T>::U;

    static __device__ __forceinline__ void pass(T (&f)[C][KK][VE], const T (&delta)[C], const T (&v0)[VE], const T (&r0)[VE],
                                                const T *st, int rs, int kcnt, int lane, KS (&lk)[C], KU (&hk)[C])
    {
        Keys<T> kk[C];
#pragma unroll
        for (int c = 0; c < C; ++c) kk[c].reset();
#pragma unroll
        for (int k = 0; k < KK; ++k) {
            if (!CHK || k < kcnt) {
                T vv[VE], rr[VE];
                if (k) {
                    lds_v(st + VE * (32 * k + lane), vv);
                    lds_v(st + rs + VE * (32 * k + lane), rr);
                }
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    if (k) pass_chunk(f[c][k], delta[c], vv, rr, kk[c]);
                    else pass_chunk(f[c][0], delta[c], v0, r0, kk[c]);
                }
            }
        }
#pragma unroll
        for (int c = 0; c < C; ++c) kk[c].fold(lk[c], hk[c]);
    }

    // The residual moves by K~_b V_j delta = dres_j delta U_j (dres = d for a Gaussian mode,
    // |K~_b V_j| for one sampled flat); all lanes store the same.
    static __device__ __forceinline__ void store_w(const WarpChains<T, C> &wc, int j, int np, T dres, const T (&delta)[C])
    {
        if (j < np) {
#pragma unroll
            for (int c = 0; c < C; ++c) wc.w_(c)[j] = dres * delta[c];
        }
    }

    // Gamma prior (Eq. compat): the draw is a proposal, accepted with probability
    // min(1, prod ((f + delta V)_+ / f)^(a - 1)) over the block.  Where the tile leaves registers
    // a visit keeps a - 1 there (kKeepShape), and the logarithms of its points too (kKeepLogs): an
    // accepted proposal's logarithms are the next move's current ones, so a move takes one logarithm
    // per point instead of two and reads nothing from global memory (250 chains, ms a sweep: ragged
    // blocks of 20 points and a level of 101, FP32, 0.100 -> 0.066; one of 520, 2.07 -> 1.18; of 100 to 300, FP64,
    // 6.8 -> 4.2; with a - 1 alone: one of 1100, FP32, 8.4 -> 5.6; one of 600, FP64, both 23.1).
    static constexpr bool kKeepLogs = PRIOR && KK * VE * sizeof(T) <= 128;
    static constexpr bool kKeepShape = PRIOR && KK * VE * sizeof(T) <= 256;
    struct PriorState {
        T am1[kKeepShape ? KK : 1][kKeepShape ? VE : 1], lg[kKeepLogs ? KK : 1][kKeepLogs ? VE : 1];
    };
    static __device__ __forceinline__ void prior_start(const SweepParams<T> &p, const T (&f)[C][KK][VE], int bn, int bstart,
                                                       int lane, PriorState &ps)
    {
        if constexpr (kKeepShape) {
#pragma unroll
            for (int k = 0; k < KK; ++k)
#pragma unroll
                for (int v = 0; v < VE; ++v) {
                    const int nl = VE * (32 * k + lane) + v;
                    ps.am1[k][v] = nl < bn ? __ldg(p.prior_am1 + bstart + nl) : T(0);
                    if constexpr (kKeepLogs) ps.lg[k][v] = ps.am1[k][v] != T(0) ? m_log(f[0][k][v]) : T(0);
                }
        }
    }
    static __device__ __forceinline__ void prior_step(const SweepParams<T> &p, const T (&f)[C][KK][VE], T (&delta)[C],
                                                      const T (&v0)[VE], const T *st, T ua, int bn, int bstart, int kcnt,
                                                      int lane, PriorState &ps, unsigned (&rej)[C])
    {
        if (delta[0] == T(0)) return;
        const T log_ua = m_log(ua);
        T lsum = T(0);
        T l1[kKeepLogs ? KK : 1][kKeepLogs ? VE : 1];
        unsigned zflags = 0u;   // 1: a proposed value is 0, 2: a current value is 0
#pragma unroll
        for (int k = 0; k < KK; ++k) {
            if (!CHK || k < kcnt) {
                T vv[VE];
                if (k == 0) {
#pragma unroll
                    for (int v = 0; v < VE; ++v) vv[v] = v0[v];
                } else {
                    lds_v(st + VE * (32 * k + lane), vv);
                }
#pragma unroll
                for (int v = 0; v < VE; ++v) {
                    const int nl = VE * (32 * k + lane) + v;
                    T am1;
                    if constexpr (kKeepShape) am1 = ps.am1[k][v];
                    else am1 = nl < bn ? __ldg(p.prior_am1 + bstart + nl) : T(0);
                    const T x0 = f[0][k][v];
                    const T x1 = m_max(m_fma(delta[0], vv[v], x0), T(0));
                    if constexpr (kKeepLogs) l1[k][v] = T(0);
                    if (am1 != T(0)) {
                        if constexpr (kKeepLogs) l1[k][v] = m_log(x1);
                        if (x1 == T(0)) zflags |= 1u;
                        else if (x0 == T(0)) zflags |= 2u;
                        else if constexpr (kKeepLogs) lsum += am1 * (l1[k][v] - ps.lg[k][v]);
                        else lsum += am1 * (m_log(x1) - m_log(x0));
                    }
                }
            } else if constexpr (kKeepLogs) {
#pragma unroll
                for (int v = 0; v < VE; ++v) l1[k][v] = T(0);
            }
        }
        for (int off = 1; off < 32; off <<= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
        zflags = __reduce_or_sync(0xffffffffu, zflags);
        const T lr = (zflags & 1u) ? -CUDART_INF_F : (zflags & 2u) ? CUDART_INF_F : lsum;
        if (!(log_ua < lr)) {
            delta[0] = T(0);
            ++rej[0];
        } else if constexpr (kKeepLogs) {
#pragma unroll
            for (int k = 0; k < KK; ++k)
#pragma unroll
                for (int v = 0; v < VE; ++v) ps.lg[k][v] = l1[k][v];
        }
    }

    // false: a bounded wait gave up
    static __device__ __forceinline__ bool run(const SweepParams<T> &p, const LaunchShape &sh, const Regions &R, RingPos &rp,
                                               const WarpChains<T, C> &wc, MoveCounts<C> &n, const BlockDesc &B,
                                               const T *pk, long long s, bool keep, bool trace, int &win, int &win_end,
                                               int lane, T (&sd2)[C], T (&sf2)[C])
    {
        const int bn = uni(B.n), bstart = uni(B.start), rs = uni(B.rs), np = uni(B.np), recstride = 2 * rs + 4;
        const int kcnt = (bn + 32 * VE - 1) / (32 * VE);
        T f[C][KK][VE];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const T *Fq = sh.fpad ? wc.c_(c) + wc.off_f : p.F + (size_t)wc.q[c] * p.ldF;
#pragma unroll
            for (int k = 0; k < KK; ++k)
#pragma unroll
                for (int v = 0; v < VE; ++v) {
                    const int nl = VE * (32 * k + lane) + v;
                    f[c][k][v] = nl < bn ? Fq[bstart + nl] : T(0);
                }
        }
        PriorState ps;
        if constexpr (PRIOR) prior_start(p, f, bn, bstart, lane, ps);
        // keys of the block's first mode: f >= +0, so that the pass reduces to the products
        KS lk[C];
        KU hk[C];
        {
            Keys<T> kk[C];
#pragma unroll
            for (int c = 0; c < C; ++c) kk[c].reset();
#pragma unroll
            for (int k = 0; k < KK; ++k) {
                if (!CHK || k < kcnt) {
                    T rr[VE];
                    lds_v(pk + kPacketHeader + VE * (32 * k + lane), rr);
#pragma unroll
                    for (int c = 0; c < C; ++c) key_chunk(f[c][k], rr, kk[c]);
                }
            }
#pragma unroll
            for (int c = 0; c < C; ++c) kk[c].fold(lk[c], hk[c]);
        }
        const int rps = records_per_stage<T>(sh, uni(B.inv_rec));
        // modes j < ng are Gaussian, those from nz on flat; in between both occur (never, when
        // the singular values are sorted)
        const int ng = uni(B.ng), nz = uni(B.nz);
        // flat moves are unrolled where one chain's latency is the limit and runs are long
        // (blocked modes, 1024 chains: 0.0850 -> 0.0808 ms a sweep); not in the kernels for blocks
        // of one vector, whose time is draws and whose code has to stay small (hierarchy: 0.0688 by
        // 1, 0.0744 by 4), nor with several chains, which fill the pipes (4096 chains: 0.1125, 0.1173)
        constexpr int kUnroll = PRIOR || C > 1 || KV == 1 ? 1 : KK <= 2 ? 4 : KK <= 4 ? 2 : 1;
        for (int j = 0; j < bn;) {
            // one ring stage of moves [j, jstage)
            const int t0 = bstart + j, jstage = min(j + rps, bn);
            // uniform of move t: word t%4 of Philox(ctr = {t/4, s, q, problem}); 128 of them, from
            // the stage's first move on, come from one Philox call per lane and chain
            if (bstart + jstage > win_end) {
                win = t0 & ~3;
                win_end = win + 128;
                __syncwarp();   // the previous window is read by every lane
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    unsigned long long c0 = (unsigned long long)(win >> 2) + (unsigned long long)lane;
                    unsigned long long c1 = (unsigned long long)s, c2 = (unsigned long long)wc.q[c] + p.chain_offset,
                                       c3 = p.problem_id;
                    philox4x64_10(c0, c1, c2, c3, p.seed, 0ull);
                    T *usm = wc.u_(c);
                    usm[4 * lane] = uniform_from<T>(c0);
                    usm[4 * lane + 1] = uniform_from<T>(c1);
                    usm[4 * lane + 2] = uniform_from<T>(c2);
                    usm[4 * lane + 3] = uniform_from<T>(c3);
                    if constexpr (PRIOR) {   // acceptance uniforms: ctr {t/4, s, q, problem xor 2^63}
                        c0 = (unsigned long long)(win >> 2) + (unsigned long long)lane;
                        c1 = (unsigned long long)s;
                        c2 = (unsigned long long)wc.q[c] + p.chain_offset;
                        c3 = p.problem_id ^ (1ull << 63);
                        philox4x64_10(c0, c1, c2, c3, p.seed, 0ull);
                        usm[128 + 4 * lane] = uniform_from<T>(c0);
                        usm[128 + 4 * lane + 1] = uniform_from<T>(c1);
                        usm[128 + 4 * lane + 2] = uniform_from<T>(c2);
                        usm[128 + 4 * lane + 3] = uniform_from<T>(c3);
                    }
                }
                __syncwarp();
            }
            const T *up = wc.u_(0) + (bstart - win);
            // the stage has usually landed long ago
            if (!warp_wait(R.full + rp.slot, rp.phase, sh.wait_limit)) return false;
            const T *st = reinterpret_cast<const T *>(R.stages + (size_t)rp.slot * sh.stage_bytes);
            while (j < jstage) {
                // moves of one kind
                const int jbeg = j;
                int jend = jstage;
                bool flat = j >= nz;
                if (j < ng) {
                    jend = min(jstage, ng);
                } else if (!flat) {   // a mode between: one move, by its own d
                    jend = j + 1;
                    flat = uni((int)is_zero(st[2 * rs])) != 0;
                }
                if (flat) {
#pragma unroll kUnroll
                    for (; j < jend; ++j, st += recstride) {
                        T u[C], v0[VE], r0[VE], lo[C], hi[C], delta[C];
                        // chunk 0 of the pass and the mode's data do not depend on the bounds: loaded first
                        const T dres = st[2 * rs + 2];
#pragma unroll
                        for (int c = 0; c < C; ++c) u[c] = up[j + c * wc.tw];
                        lds_v(st + VE * lane, v0);
                        lds_v(st + rs + VE * lane, r0);
                        warp_bounds<C>(lk, hk, lo, hi);
                        // degenerate interval: no move; else flat on [lo, hi] (both bounds finite:
                        // set-up rejects zero modes that do not change sign)
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            const bool open = open_interval(lo[c], hi[c]);
                            delta[c] = open ? m_fma(u[c], hi[c] - lo[c], lo[c]) : T(0);
                            n.zero[c] += open ? 1u : 0u;
                        }
                        if constexpr (PRIOR) prior_step(p, f, delta, v0, st, up[128 + j], bn, bstart, kcnt, lane, ps, n.rej);
                        pass(f, delta, v0, r0, st, rs, kcnt, lane, lk, hk);
                        store_w(wc, j, np, dres, delta);
                    }
                    n.flat += (unsigned)(j - jbeg);
                } else {
#pragma unroll 1
                    for (; j < jend; ++j, st += recstride) {
                        T u[C], v0[VE], r0[VE], lo[C], hi[C], delta[C], dj, ij, dres;
                        lds_mode(st + 2 * rs, dj, ij, dres);
#pragma unroll
                        for (int c = 0; c < C; ++c) u[c] = up[j + c * wc.tw];
                        lds_v(st + VE * lane, v0);
                        lds_v(st + rs + VE * lane, r0);
                        warp_bounds<C>(lk, hk, lo, hi);
                        // degenerate interval: no move; else the truncated Gaussian
                        constexpr int G = 32 / C;
                        T l = lo[0], h = hi[0], uu = u[0];
                        const T *cs = wc.c_(0);
#pragma unroll
                        for (int c = 1; c < C; ++c) {
                            const bool mine = lane / G == c;
                            l = mine ? lo[c] : l;
                            h = mine ? hi[c] : h;
                            uu = mine ? u[c] : uu;
                            cs = mine ? wc.c_(c) : cs;
                        }
                        const T cj = j < np ? cs[j] : T(0);
                        const T dl = draw_team<G>(cj, dj, ij, l, h, uu, open_interval(l, h), lane, n.capped);
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            const T x = C == 1 ? dl : __shfl_sync(0xffffffffu, dl, c * G);
                            const bool fin = is_finite(x);
                            n.bad[c] += fin ? 0u : 1u;
                            n.deg[c] += open_interval(lo[c], hi[c]) ? 0u : 1u;
                            delta[c] = fin ? x : T(0);
                        }
                        if constexpr (PRIOR) prior_step(p, f, delta, v0, st, up[128 + j], bn, bstart, kcnt, lane, ps, n.rej);
                        pass(f, delta, v0, r0, st, rs, kcnt, lane, lk, hk);
                        store_w(wc, j, np, dres, delta);
                    }
                }
            }
            // release the stage to the producer (one arrival per warp)
            __syncwarp();
            mbar_arrive_lane0(R.empty + rp.slot, lane);
            ring_next(rp, sh.depth);
        }
        // write the block back and accumulate the kept sweep
        constexpr bool psums = sizeof(T) == 4;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            T *Fq = sh.fpad ? wc.c_(c) + wc.off_f : p.F + (size_t)wc.q[c] * p.ldF;
            const bool write = wc.active[c];
#pragma unroll
            for (int k = 0; k < KK; ++k)
#pragma unroll
                for (int v = 0; v < VE; ++v) {
                    const int nl = VE * (32 * k + lane) + v;
                    if (write && nl < bn) {
                        const int i = bstart + nl;
                        if (trace) {
                            const T old = Fq[i], dlt = f[c][k][v] - old;
                            sd2[c] = m_fma(dlt, dlt, sd2[c]);
                            sf2[c] = m_fma(old, old, sf2[c]);
                        }
                        Fq[i] = f[c][k][v];
                        if (keep) {
                            if constexpr (psums) {
                                T *p1 = sh.npad ? wc.c_(c) + wc.off_p : reinterpret_cast<T *>(p.P1) + (size_t)wc.q[c] * p.ldF;
                                T *p2 = sh.npad ? p1 + sh.npad : reinterpret_cast<T *>(p.P2) + (size_t)wc.q[c] * p.ldF;
                                p1[i] += f[c][k][v];
                                p2[i] = m_fma(f[c][k][v], f[c][k][v], p2[i]);
                            } else {
                                const double x = (double)f[c][k][v];
                                p.S1[(size_t)wc.q[c] * p.N + i] += x;
                                p.S2[(size_t)wc.q[c] * p.N + i] += x * x;
                            }
                        }
                    }
                    // one chunk's sums at a time: keeps the compiler from holding every
                    // chunk's loaded sums in registers at once (the widest tiles spilled)
                    if (v + 1 == VE) asm volatile("" ::: "memory");
                }
        }
        return true;
    }
};

// --------------------------------------------------------------------------
// A consumer warp: its C chains of chain group `group` (consumers x C chains) of
// problem p for the launch's sweeps.
// --------------------------------------------------------------------------
template <class T, int KV, int C, bool PRIOR>
__device__ __forceinline__ void consume(const SweepParams<T> &p, const LaunchShape &sh, const SweepRange &rg, int group,
                                        unsigned char *smem_raw, const Regions &R, RingPos &rp, bool &failed)
{
    constexpr int VEC = VecOf<T>::n;
    if (failed) return;
    const int lane = threadIdx.x & 31;
    const int wcta = uni((int)(threadIdx.x >> 5));
    WarpChains<T, C> wc;
    // per chain in shared memory: c and w (cpad: w_j takes c_j's place, which move j has
    // read), r~ (mpad), the uniforms of the current window of 128 moves (with a prior 128
    // more) and, where they fit, the chain state (fpad) and the sums of f and f^2 over this
    // launch's kept sweeps (FP32, npad each)
    wc.tw = sh.team_words;
    wc.sm = reinterpret_cast<T *>(smem_raw) + (size_t)(wcta * C) * sh.team_words;
    wc.off_r = sh.cpad;
    wc.off_u = sh.cpad + sh.mpad;
    wc.off_f = wc.off_u + (PRIOR ? 256 : 128);
    wc.off_p = wc.off_f + sh.fpad;
    // FP32 chain state: the kept-sweep sums of the current kBinSweeps-sweep block (aligned
    // to absolute sweep indices) in FP32, added to the FP64 sums when the block closes.
    // Between launches they wait in the workspace (P1, P2); during one they live in shared
    // memory where they fit, else in the workspace -- the same arithmetic in the same order
    // either way, so results do not depend on where a run is split into calls.
    // FP64 chain state: straight into the FP64 sums.
    constexpr bool psums = sizeof(T) == 4;
    const bool kept_here = psums && rg.burn_in < rg.sweep0 + rg.nsweeps;
    MoveCounts<C> n;
    n.capped = 0;
    n.flat = 0u;
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const long long q_raw = ((long long)group * sh.consumers + wcta) * C + c;
        wc.active[c] = q_raw < p.chains;
        wc.q[c] = wc.active[c] ? q_raw : (long long)p.chains - 1;   // idle chains shadow a real one, write nothing
        n.deg[c] = n.zero[c] = n.bad[c] = n.rej[c] = 0u;
        const T *Rq = p.R + (size_t)wc.q[c] * p.ldR;
        for (int m = lane; m < p.M; m += 32) wc.r_(c)[m] = Rq[m];
        if (sh.fpad) {
            const T *Fq = p.F + (size_t)wc.q[c] * p.ldF;
            T *fs = wc.c_(c) + wc.off_f;
            for (int i = lane; i < p.N; i += 32) fs[i] = Fq[i];
        }
        if (kept_here && sh.npad) {
            const T *P1q = reinterpret_cast<const T *>(p.P1) + (size_t)wc.q[c] * p.ldF;
            const T *P2q = reinterpret_cast<const T *>(p.P2) + (size_t)wc.q[c] * p.ldF;
            T *p1 = wc.c_(c) + wc.off_p;
            for (int i = lane; i < p.N; i += 32) {
                p1[i] = P1q[i];
                p1[sh.npad + i] = P2q[i];
            }
        }
    }
    __syncwarp();

    const bool trace = p.steptrace != nullptr;   // step-size trace of Fig. MCsteps (diagnostic)
    const long long s_begin = uni(rg.sweep0), s_end = s_begin + uni(rg.nsweeps), burn_in = uni(rg.burn_in);
    const int M = uni(p.M);
    for (long long s = s_begin; s < s_end && !failed; ++s) {
        const bool keep = s >= burn_in;
        int win = 0, win_end = -1;  // window [win, win_end) of moves whose uniforms are in shared memory
        T sd2[C], sf2[C];           // this lane's |f(s+1) - f(s)|^2 and |f(s)|^2 (trace only)
#pragma unroll
        for (int c = 0; c < C; ++c) sd2[c] = sf2[c] = T(0);
        // the sweep's blocks, as the packets bring them: the producer draws the level, the same
        // for every chain of the problem (Sec. IV.C), and the last block of a level says so
        for (bool last = false; !last;) {
            if (!warp_wait(R.pfull + rp.pslot, rp.pphase, sh.wait_limit)) {
                failed = true;
                break;
            }
            const T *pk = reinterpret_cast<const T *>(R.packets + (size_t)rp.pslot * sh.pbytes);
            const BlockDesc &B = *reinterpret_cast<const BlockDesc *>(pk);
            last = uni(B.last) != 0;
            const int bn = uni(B.n), np = uni(B.np), usr = packet_row<T>(M);
            const T *Us = u_staged<T>(sh, uni(B.pkn)) ? pk + kPacketHeader + uni(B.rs) : nullptr;
            // a projection through the record ring, from vec to out
            auto streamed = [&](int vec, int out, bool subtract, int K, int cols, int width) {
                const StreamPos at = project_stream<T, C>(wc.sm + vec, wc.sm + out, wc.tw, subtract, R.full, R.empty, R.stages,
                                                          sh.stage_bytes, sh.depth, sh.wait_limit, K, cols, width,
                                                          StreamPos{rp.slot, rp.phase, true});
                rp.slot = uni(at.slot);
                rp.phase = uni(at.phase);
                return uni((int)at.ok) != 0;
            };
            bool ok = true;
            if (Us)
                project_entry<T, C>(wc, Us, np, usr, M, lane);
            else
                ok = streamed(wc.off_r, 0, false, M, np, entry_width(np));
            if (!ok) {
                failed = true;
                break;
            }
            __syncwarp();
            if (bn <= 16 * VEC)
                ok = Visit<T, KV, C, PRIOR, 1, VEC / 2>::run(p, sh, R, rp, wc, n, B, pk, s, keep, trace, win, win_end,
                                                             lane, sd2, sf2);
            else if (KV == 1 || bn <= 32 * VEC)
                ok = Visit<T, KV, C, PRIOR, 1, VEC>::run(p, sh, R, rp, wc, n, B, pk, s, keep, trace, win, win_end, lane,
                                                         sd2, sf2);
            else if (KV == 2 || bn > 32 * VEC * (KV - 1))
                ok = Visit<T, KV, C, PRIOR, KV, VEC>::run(p, sh, R, rp, wc, n, B, pk, s, keep, trace, win, win_end, lane,
                                                          sd2, sf2);
            else
                ok = Visit<T, KV, C, PRIOR, 0, VEC>::run(p, sh, R, rp, wc, n, B, pk, s, keep, trace, win, win_end, lane,
                                                         sd2, sf2);
            if (!ok) {
                failed = true;
                break;
            }
            __syncwarp();
            if (Us)
                project_exit<T, C>(wc, Us, np, usr, M, lane);
            else if (!streamed(0, wc.off_r, true, np, M, 32)) {
                failed = true;
                break;
            }
            // release the packet to the producer (one arrival per warp)
            __syncwarp();
            mbar_arrive_lane0(R.pempty + rp.pslot, lane);
            packet_next(rp, sh.pslots);
        }
        if (trace && !failed) {   // Delta_s = |f(s+1) - f(s)| / |f(s)| of this chain, summed over chains
#pragma unroll
            for (int c = 0; c < C; ++c) {
                T a = sd2[c], b = sf2[c];
                for (int off = 1; off < 32; off <<= 1) {
                    a += __shfl_xor_sync(0xffffffffu, a, off);
                    b += __shfl_xor_sync(0xffffffffu, b, off);
                }
                if (wc.active[c] && lane == 0 && s < p.trace_cap && b > T(0))
                    atomicAdd(p.steptrace + s, sqrt((double)a / (double)b));
            }
        }
    }
    if (failed) {
        if (lane == 0) atomicAdd(&p.counters->timeouts, 1ull);
        return;
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < C; ++c) {
        if (wc.active[c]) {
            T *Rq = p.R + (size_t)wc.q[c] * p.ldR;
            for (int m = lane; m < p.M; m += 32) Rq[m] = wc.r_(c)[m];
            if (sh.fpad) {
                T *Fq = p.F + (size_t)wc.q[c] * p.ldF;
                const T *fs = wc.c_(c) + wc.off_f;
                for (int i = lane; i < p.N; i += 32) Fq[i] = fs[i];
            }
            if (kept_here) {
                T *P1q = reinterpret_cast<T *>(p.P1) + (size_t)wc.q[c] * p.ldF;
                T *P2q = reinterpret_cast<T *>(p.P2) + (size_t)wc.q[c] * p.ldF;
                const T *p1 = sh.npad ? wc.c_(c) + wc.off_p : P1q;
                const T *p2 = sh.npad ? p1 + sh.npad : P2q;
                if (s_end % kBinSweeps == 0) {   // the block closes: into the FP64 sums
                    for (int i = lane; i < p.N; i += 32) {
                        p.S1[(size_t)wc.q[c] * p.N + i] += (double)p1[i];
                        p.S2[(size_t)wc.q[c] * p.N + i] += (double)p2[i];
                        P1q[i] = P2q[i] = T(0);
                    }
                } else if (sh.npad) {   // the block continues in a later launch
                    for (int i = lane; i < p.N; i += 32) {
                        P1q[i] = p1[i];
                        P2q[i] = p2[i];
                    }
                }
            }
        }
        // counters: the solver's cap is counted by the lanes of a chain's team alike
        const int capped = __shfl_sync(0xffffffffu, n.capped, c * (32 / C));
        if (wc.active[c] && lane == 0) {
            const unsigned deg = n.deg[c] + (n.flat - n.zero[c]);
            if (deg) atomicAdd(&p.counters->degenerate, (unsigned long long)deg);
            if (n.zero[c]) atomicAdd(&p.counters->zero_mode, (unsigned long long)n.zero[c]);
            if (n.bad[c]) atomicAdd(&p.counters->nonfinite, (unsigned long long)n.bad[c]);
            if (n.rej[c]) atomicAdd(&p.counters->prior_rejections, (unsigned long long)n.rej[c]);
            if (capped) atomicAdd(&p.counters->tail_capped, (unsigned long long)capped);
        }
    }
}

// --------------------------------------------------------------------------
// the persistent sweep kernel: the sweeps [ctrl->sweep0, + ctrl->nsweeps) of
// every work item (problem, chain group).  Warps 0 .. consumers-1 run chains;
// warp `consumers` produces visit packets and move records.  CTAs pull items
// from ctrl->queue; an item's parameters are copied from probs into shared memory.
// --------------------------------------------------------------------------
template <class T, int KV, int C, bool PRIOR>
__global__ void __launch_bounds__(32 * (kMaxConsumers + 1), 1)
sweep_kernel(const SweepParams<T> *__restrict__ probs, const WorkItem *__restrict__ items, RunCtrl *ctrl,
             const __grid_constant__ LaunchShape shape)
{
    __shared__ SweepParams<T> sp;
    __shared__ SweepRange rg;
    __shared__ int s_item;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Regions R;
    R.full = reinterpret_cast<unsigned long long *>(smem_raw + shape.off_bars);
    R.empty = R.full + kMaxRingDepth;
    R.pfull = R.empty + kMaxRingDepth;
    R.pempty = R.pfull + kMaxPacketSlots;
    R.packets = smem_raw + shape.off_packets;
    R.stages = smem_raw + shape.off_stages;
    const int wcta = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int i = 0; i < shape.depth; ++i) {
            mbar_init(R.full + i, 1);
            mbar_init(R.empty + i, (unsigned)shape.consumers);
        }
        for (int i = 0; i < shape.pslots; ++i) {
            mbar_init(R.pfull + i, 1);
            mbar_init(R.pempty + i, (unsigned)shape.consumers);
        }
        fence_mbar_init();
        fence_proxy_async_smem();
        rg.sweep0 = ctrl->sweep0;
        rg.nsweeps = ctrl->nsweeps;
        rg.burn_in = ctrl->burn_in;
    }
    RingPos rp{0u, 0, 0u, 0u, 0, 0u};
    bool failed = false;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(&ctrl->queue, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= shape.n_items) break;
        const WorkItem w = items[it];
        static_assert(sizeof(SweepParams<T>) % 8 == 0, "copied in 8-byte words");
        for (int i = threadIdx.x; i < (int)(sizeof(SweepParams<T>) / 8); i += blockDim.x)
            reinterpret_cast<unsigned long long *>(&sp)[i] =
                reinterpret_cast<const unsigned long long *>(probs + w.problem)[i];
        __syncthreads();
        if (wcta == shape.consumers)
            produce(sp, shape, rg, R, rp, failed);
        else
            consume<T, KV, C, PRIOR>(sp, shape, rg, w.group, smem_raw, R, rp, failed);
        __syncthreads();   // the item is finished before sp and s_item change
    }
}

template <class T, int KV, int C, bool PRIOR>
struct SweepKernel {
    static size_t smem(const LaunchShape &sh) { return (size_t)sh.off_stages + (size_t)sh.depth * sh.stage_bytes; }
    static cudaError_t launch(const SweepParams<T> *probs, const WorkItem *items, RunCtrl *ctrl, const LaunchShape &sh,
                              int ctas, cudaStream_t stream)
    {
        const cudaError_t e = cudaFuncSetAttribute(sweep_kernel<T, KV, C, PRIOR>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem(sh));
        if (e != cudaSuccess) return e;
        sweep_kernel<T, KV, C, PRIOR>
            <<<(unsigned)ctas, 32 * (sh.consumers + 1), smem(sh), stream>>>(probs, items, ctrl, sh);
        return cudaGetLastError();
    }
    static int per_sm(const LaunchShape &sh)
    {
        int n = 0;
        if (cudaFuncSetAttribute(sweep_kernel<T, KV, C, PRIOR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem(sh)) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sweep_kernel<T, KV, C, PRIOR>,
                                                          32 * (sh.consumers + 1), smem(sh)) != cudaSuccess)
            return 0;
        return n;
    }
};

// dispatch over the register tile (kv) for one chain count per warp and prior flag
template <class T, int C, bool PRIOR, int... KVs>
struct SweepDispatch {
    static cudaError_t launch(const SweepParams<T> *probs, const WorkItem *items, RunCtrl *ctrl, const LaunchShape &sh,
                              int kv, int ctas, cudaStream_t s)
    {
        cudaError_t e = cudaErrorInvalidValue;
        ((kv == KVs ? (e = SweepKernel<T, KVs, C, PRIOR>::launch(probs, items, ctrl, sh, ctas, s), 0) : 0), ...);
        return e;
    }
    static int per_sm(const LaunchShape &sh, int kv)
    {
        int n = 0;
        ((kv == KVs ? (n = SweepKernel<T, KVs, C, PRIOR>::per_sm(sh), 0) : 0), ...);
        return n;
    }
};

}  // namespace asmgb
