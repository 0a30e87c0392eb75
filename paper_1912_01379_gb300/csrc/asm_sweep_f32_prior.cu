// FP32 chain state (the mixed-precision path): sweep kernels with the gamma prior's acceptance step, one chain per warp.
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(float, f32_prior, 1, true, 1, 2, 4, 8, 16)

}  // namespace asmgb
