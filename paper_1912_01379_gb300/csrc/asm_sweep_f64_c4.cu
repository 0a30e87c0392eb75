// FP64 chain state, 4 chains per warp: sweep kernels.
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(double, f64_c4, 4, false, 1, 2, 4, 8)

}  // namespace asmgb
