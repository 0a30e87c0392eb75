// FP32 chain state (the mixed-precision path), 4 chains per warp: sweep kernels.
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(float, f32_c4, 4, false, 1, 2, 4, 8)

}  // namespace asmgb
