// FP32 chain state (the mixed-precision path): sweep kernels budgeted for two CTAs per SM (128 registers per thread), for the tiles that fit them.
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(float, f32_c1_m2, 1, 2, false, 1, 2, 4, 8)
ASM_DEFINE_SWEEP_LAUNCHER(float, f32_c2_m2, 2, 2, false, 1, 2, 4)
ASM_DEFINE_SWEEP_LAUNCHER(float, f32_c4_m2, 4, 2, false, 1, 2)

}  // namespace asmgb
