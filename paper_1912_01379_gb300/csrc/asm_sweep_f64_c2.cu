// FP64 chain state, 2 chains per warp: sweep kernels.
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(double, f64_c2, 2, false, 1, 2, 4, 8, 16)

}  // namespace asmgb
