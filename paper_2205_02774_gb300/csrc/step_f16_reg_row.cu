// Step kernels of shifted binary16 storage,
// the regularized collision, lanes 32 cells apart (one of the
// instantiation units of step_kernel.cuh, compiled in parallel).
#include "step_kernel.cuh"

namespace stg {

bool launch_f16_reg_row(const StepArgs &a, bool stats, cudaStream_t s, cudaStream_t side)
{
    return launch_row<__half, 4, true>(a, stats, s, side);
}

}  // namespace stg
