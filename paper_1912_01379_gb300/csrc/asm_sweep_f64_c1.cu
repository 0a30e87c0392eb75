// FP64 chain state, 1 chain per warp: sweep kernels budgeted for one CTA per SM (up to 255 registers per thread).
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(double, f64_c1_m1, 1, 1, false, 1, 2, 4, 8, 16, 32)

}  // namespace asmgb
