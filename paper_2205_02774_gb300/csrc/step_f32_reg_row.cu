// Step kernels of FP32 storage,
// the regularized collision, lanes 32 cells apart (one of the
// instantiation units of step_kernel.cuh, compiled in parallel).
#include "step_kernel.cuh"

namespace stg {

bool launch_f32_reg_row(const StepArgs &a, bool stats, cudaStream_t s, cudaStream_t side)
{
    if (lane_cells(a) == 1) return launch_row<float, 1, true>(a, stats, s, side);
    return launch_row<float, 2, true>(a, stats, s, side);
}

}  // namespace stg
