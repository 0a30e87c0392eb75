// FP64 chain state, 4 chains per warp: sweep kernels budgeted for one CTA per SM (up to 255 registers per thread).
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(double, f64_c4_m1, 4, 1, false, 1, 2, 4, 8)

}  // namespace asmgb
