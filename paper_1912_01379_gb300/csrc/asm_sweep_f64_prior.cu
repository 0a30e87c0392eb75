// FP64 chain state: sweep kernels with the gamma prior's acceptance step, one chain per warp.
#include "asm_sweep.cuh"

namespace asmgb {

ASM_DEFINE_SWEEP_LAUNCHER(double, f64_prior, 1, true, 1, 2, 4, 8, 16, 32)

}  // namespace asmgb
