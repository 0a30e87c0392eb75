// FP32 chain state (the mixed-precision path), 1 chain per warp: sweep kernels.
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(float, f32_c1, 1, false, 1, 2, 4, 8, 16)

}  // namespace asmgb
