// FP64 chain state, 1 chain per warp: sweep kernels.
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(double, f64_c1, 1, false, 1, 2, 4, 8, 16, 32)

}  // namespace asmgb
