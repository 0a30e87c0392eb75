// asm_internal.h -- types shared by the host library and the sweep kernels.
// Not part of the public ABI (include/asm.h).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace asmgb {

// Rows of a block's mode data are padded so that 32 lanes of whole vectors stay in
// the row: 64 elements for blocks of up to 64 points, else a multiple of 128.
constexpr int kRowAlignSmall = 64;
constexpr int kRowAlign = 128;
// Elements reserved for the block descriptor at the head of a visit packet.
constexpr int kPacketHeader = 32;
// Residual refresh period of the sweep loop (sweeps).
constexpr int kRefreshPeriod = 64;

// Row stride of U in a packet: FP32 4 x odd, so that 16-byte loads of a row per lane are free
// of bank conflicts, FP64 odd, for 8-byte ones.  Packets are laid out for the larger of the two.
template <class T>
__host__ __device__ constexpr int packet_row(int M)
{
    return sizeof(T) == 4 ? ((M + 3) / 4 | 1) * 4 : M | 1;
}

// One block of one level, as the device sees it.  Offsets are in elements of
// the precision-specific arrays.
struct BlockDesc {
    int start;       // first grid point of the block
    int n;           // block width n_b
    int np;          // modes with a U column: min(M, n_b)
    int ng, nz;      // modes before ng are Gaussian (d > 0), from nz on flat (d = 0 in this precision)
    int rs;          // row stride of V/R rows
    int recstride;   // elements per move record: 2 rs + 4
    int usr;         // elements a packet provides per row of U (the larger precision's stride)
    int last;        // 1: the last block of its level
    int pkn;         // elements of the visit packet with U (saturated)
    float inv_rec;   // 1 / recstride
    long long offUe, offUx;   // U in tiles of 32 columns for the streamed projections: entry
                              // (columns are modes, M rows each), exit (data points, np rows)
    long long offRec;  // move records of the block: n records of recstride elements
    long long offPk;   // visit packet: header, R row of mode 0 (rs), U (np rows of usr); 16-byte aligned
};
static_assert(sizeof(BlockDesc) <= kPacketHeader * sizeof(float), "the packet's header holds the descriptor");

// Device-side problem data in one precision T (R = -1/V, NaN where V is left out of the bounds).
template <class T>
struct ProblemData {
    const T *rec;            // per move j: {V_j, R_{j+1} (rs each), d_j, 1/d_j, |K~_b V_j|, 0}
    const T *pk;             // visit packets
    const T *Ue, *Ux;        // U in two tilings, for blocks whose U does not fit a packet slot
};

struct Counters {            // device counters, first bytes of the workspace
    unsigned long long degenerate, zero_mode, tail_capped, nonfinite;
    unsigned long long drift_bits;   // max relative chi2 drift, as ordered bits of a double
    unsigned long long timeouts;     // bounded waits that gave up (the launch then stopped early)
    unsigned long long prior_rejections;   // proposals the gamma prior rejected
    unsigned long long pad;
};

template <class T>
struct SweepParams {
    int M, N;
    int n_levels;
    const int *level_first;           // first block index of each level
    const int *level_nblocks;
    const BlockDesc *blocks;
    ProblemData<T> pd;
    T *F; int ldF;                    // chain states, chains x ldF
    T *R; int ldR;                    // tracked residuals, chains x ldR
    double *S1, *S2;                  // sums of f and f^2, chains x N
    // binning of the Monte Carlo error (every kBinSweeps sweeps): S1 at the last bin
    // boundary (chains x N), per chain and level the pending half of a bin pair and the
    // sums of the bin means and their squares (chains x kBinLevels x N), level-0 bins per chain
    double *S1p, *bpend, *bacc1, *bacc2;
    int *bcount;
    int chains;
    unsigned long long seed, problem_id;
    unsigned long long chain_offset;  // global id of local chain 0 (Philox key word)
    Counters *counters;
    // residual refresh / initial state of this problem (FP64)
    const double *KtT, *gt;           // whitened kernel (N x M) and data
    double *chi2;                     // chains
    double f0;                        // starting value of every fbar_n (no kernel reads it; without it the fields
                                      // behind it move, and blocked modes took 0.4 % longer, grids 0.7 % less)
    // whitened kernel split into TF32 high and low parts (M x ldK FP32 each) for
    // the tensor-core refresh of the mixed path
    const float *Khi, *Klo;
    int ldK;
    // reference state of the tensor-core refresh: the mean chain state fref (N,
    // FP32) and r_ref = g~ - K~ fref (M, FP64); the product is taken of f - fref
    float *fref;
    double *rref;
    // k-split of the tensor-core refresh: the grid points are cut into ksplit parts
    // whose FP32 partial products (ksplit x chains x ldR) are added in FP64 in part
    // order by the finishing kernel; ksplit = 1: no partials (nullptr)
    float *Dpart;
    int ksplit;
    // gamma prior: a_n - 1 per grid point (nullptr: flat)
    const T *prior_am1;
    // step-size trace (nullptr: off): sum over chains of |f(s+1) - f(s)| / |f(s)| for
    // the absolute sweeps s < trace_cap
    double *steptrace;
    int trace_cap;
    // FP32 chain state: the sums of f and f^2 over one launch's kept sweeps (FP32,
    // chains x ldF) where shared memory cannot hold them; added to S1, S2 per launch
    float *P1, *P2;
};

// What every problem of one launch shares: the CTA shape and the
// shared-memory plan (the union of the problems' needs).  The move records
// of a CTA's item flow through a ring of `depth` stages and its visit packets
// through `pslots` slots, filled by one producer warp with bulk copies (TMA
// engine); `full` barriers signal landed bytes, `empty` barriers collect the
// consumer warps' releases.
struct LaunchShape {
    int C;                            // chains per warp
    int consumers;                    // consumer warps per CTA (the producer is one more)
    int depth;                        // stages in the ring
    int stage_bytes;                  // bytes per stage (>= rps of the largest records)
    int rps;                          // the largest block's move records per stage
    int pslots, pbytes;               // visit packets: slots and bytes of one
    int off_bars, off_packets, off_stages;  // byte offsets in dynamic shared memory
    int cpad;                         // shared-memory elements of the c / w buffer (>= max np)
    int mpad;                         // shared-memory stride of the residual (>= max M)
    int fpad;                         // chain state in shared memory (>= max N; 0: in global memory)
    int npad;                         // shared-memory sums of the kept sweeps per chain (>= max N;
                                      // 0: in the workspace)
    int team_words;                   // shared-memory elements per chain
    int n_items;                      // (problem, chain group) work items
    int prior;                        // 1: kernels with the gamma prior's acceptance step
    int wait_limit;                   // polls before a bounded mbarrier wait gives up
    int stall;                        // test of the failure path: the producer issues no records
};

// Per-launch control block in device memory: the work queue and the launch's
// sweep range.  Kept on the device so that one refresh period (advance the
// range, sweep, refresh) is a fixed sequence that a CUDA graph can replay.
struct RunCtrl {
    int queue;                        // next work item
    int pad_;
    long long sweep0, nsweeps;        // sweeps [sweep0, sweep0 + nsweeps)
    long long burn_in;                // absolute sweep index where accumulation starts
};

// A work item: problem index and chain group (consumers x C chains).
struct WorkItem {
    int problem, group;
};

// Launchers (asm_sweep_*.cu).  kv: 16-byte vectors per lane and chain, a power of two.
// Persistent: `ctas` CTAs of (consumers + 1) warps pull work items from
// ctrl->queue (reset to 0 before the launch); work item problems index the
// device array probs.  _cC: C chains per warp.  The registers are budgeted for one
// CTA per SM (up to 255 per thread).  A kv that a launcher has no kernel for gives
// cudaErrorInvalidValue, and 0 CTAs per SM.
#define ASM_DECLARE_SWEEP_LAUNCHER(T, NAME)                                                                     \
    cudaError_t launch_sweeps_##NAME(const SweepParams<T> *probs, const WorkItem *items, RunCtrl *ctrl,         \
                                     const LaunchShape &shape, int kv, int ctas, cudaStream_t s);               \
    int sweep_ctas_per_sm_##NAME(const LaunchShape &shape, int kv);
ASM_DECLARE_SWEEP_LAUNCHER(float, f32_c1)
ASM_DECLARE_SWEEP_LAUNCHER(float, f32_c2)
ASM_DECLARE_SWEEP_LAUNCHER(float, f32_c4)
ASM_DECLARE_SWEEP_LAUNCHER(float, f32_prior)     // with the gamma prior: one chain per warp
ASM_DECLARE_SWEEP_LAUNCHER(double, f64_c1)
ASM_DECLARE_SWEEP_LAUNCHER(double, f64_c2)
ASM_DECLARE_SWEEP_LAUNCHER(double, f64_c4)
ASM_DECLARE_SWEEP_LAUNCHER(double, f64_prior)
#undef ASM_DECLARE_SWEEP_LAUNCHER
#define ASM_DEFINE_SWEEP_LAUNCHER(T, NAME, C, PRIOR, ...)                                                       \
    cudaError_t launch_sweeps_##NAME(const SweepParams<T> *probs, const WorkItem *items, RunCtrl *ctrl,         \
                                     const LaunchShape &shape, int kv, int ctas, cudaStream_t s)                \
    {                                                                                                           \
        return SweepDispatch<T, C, PRIOR, __VA_ARGS__>::launch(probs, items, ctrl, shape, kv, ctas, s);         \
    }                                                                                                           \
    int sweep_ctas_per_sm_##NAME(const LaunchShape &shape, int kv)                                              \
    {                                                                                                           \
        return SweepDispatch<T, C, PRIOR, __VA_ARGS__>::per_sm(shape, kv);                                      \
    }
// Tensor-core residual refresh of the mixed path (asm_refresh_tc.cu): grid of
// (chain tiles of 128) x n_problems x (the largest k split) CTAs; max_bn = the
// largest refresh_tc_bn(M).
cudaError_t launch_refresh_tc(const SweepParams<float> *probs, int n_problems, int chains, int max_bn, int max_parts,
                              bool track_drift, cudaStream_t s);
int refresh_tc_bn(int M);                  // MMA N of a problem's M_tau tiles
int refresh_tc_ksplit(int chains, int N);  // parts of a problem's k range (a function of the problem)
// The FP64 combination of the k parts (problems with ksplit > 1): r~, chi^2, drift.
cudaError_t launch_refresh_finish(const SweepParams<float> *probs, int n_problems, int chains, bool track_drift,
                                  cudaStream_t s);
size_t refresh_tc_smem(int max_bn);        // dynamic shared memory of one CTA
constexpr int kRefreshTcLdK = 32;          // ldK is a multiple of this (one k-tile)
cudaError_t launch_split_k(const double *KtT, int M, int N, int ldK, float *Khi, float *Klo, cudaStream_t s);
// Reference state of every problem's tensor-core refresh: fref over tiles of 32
// grid points, then r_ref over tiles of 128 data points (two launches).
cudaError_t launch_refresh_ref(const SweepParams<float> *probs, int n_problems, int chains, int max_N, int max_M,
                               cudaStream_t s);
// Contractions of the backward pass (asm_moments.cu).  D: chains x ldD snapshot
// (centred); Sff (N x N, FP64) += D^T D; Y (chains x PM) = D Kth^T with Kth
// PM x N row-major (the whitened dK/dtheta of all parameters); Sq (chains x P)
// = the scores r~_q . (Y_q,p + kshift_p); y = L^{-T} K~ u for the G-product.
cudaError_t launch_gram(const float *D, int ldD, int chains, int N, double *Sff, cudaStream_t s);
cudaError_t launch_gram(const double *D, int ldD, int chains, int N, double *Sff, cudaStream_t s);
cudaError_t launch_kth_product(const float *D, int ldD, int chains, int N, const float *Kth, int PM, float *Y,
                               cudaStream_t s);
cudaError_t launch_kth_product(const double *D, int ldD, int chains, int N, const double *Kth, int PM, double *Y,
                               cudaStream_t s);
cudaError_t launch_scores(const float *R, int ldR, const float *Y, const double *kshift, int M, int chains, int P,
                          double *Sq, cudaStream_t s);
cudaError_t launch_scores(const double *R, int ldR, const double *Y, const double *kshift, int M, int chains, int P,
                          double *Sq, cudaStream_t s);
cudaError_t launch_vjp_G(const double *KtT, const double *L, const double *u, int M, int N, double *y,
                         cudaStream_t s);
// Polls of a bounded mbarrier wait before it gives up (each poll may suspend
// the thread briefly); a run that gives up counts a timeout and its results
// are reported as ASM_ERR_TIMEOUT.
constexpr int kWaitLimit = 1 << 22;
// Binning: bins of kBinSweeps kept sweeps aligned to multiples of kBinSweeps in
// the absolute sweep index (the refresh period), merged pairwise over kBinLevels
// levels (bins of 64 ... 8192 sweeps).
constexpr int kBinSweeps = 64;
constexpr int kBinLevels = 8;
// Sweeps from the chains' start whose step size the trace records.
constexpr int kStepTraceMax = 4096;
// Consumer warps per CTA: at most 7, so that a CTA (consumers + the producer)
// has at most 8 warps, two per SM sub-partition, and a thread may hold up to
// 255 registers (9 warps would put three on one sub-partition: 168).
constexpr int kMaxConsumers = 7;
// Deepest ring of move records (stages) a launch may use.
constexpr int kMaxRingDepth = 48;
// Move records of the largest block per ring stage: about kStageBytes of them where shared
// memory allows, at least kRecordsPerStage while three stages fit (a stage costs a consumer
// some 450 cycles: its wait, its release and the start of its loop); smaller blocks put up
// to kMaxRecordsPerStage in a stage of that size.
constexpr int kStageBytes = 32 * 1024;
constexpr int kRecordsPerStage = 4;
constexpr int kMaxRecordsPerStage = 64;
// Most slots of the ring of visit packets.
constexpr int kMaxPacketSlots = 8;
// Largest kv (16-byte vectors per lane and chain): 64 elements per lane.
constexpr int kMaxKvF32 = 16;
constexpr int kMaxKvF64 = 32;
// Largest kv with a kernel of C chains per warp (the lists in asm_sweep_*.cu).
constexpr int max_kv(bool f64, int C) { return C == 4 ? 8 : C == 2 ? 16 : f64 ? kMaxKvF64 : kMaxKvF32; }

}  // namespace asmgb
