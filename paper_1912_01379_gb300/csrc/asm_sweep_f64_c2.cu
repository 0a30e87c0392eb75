// FP64 chain state, 2 chains per warp: sweep kernels budgeted for one CTA per SM (up to 255 registers per thread).
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(double, f64_c2_m1, 2, 1, false, 1, 2, 4, 8, 16)

}  // namespace asmgb
