// Step kernels of FP32 storage,
// the regularized collision, two cells per lane (one of the instantiation units of step_kernel.cuh,
// compiled in parallel).
#include "step_kernel.cuh"

namespace stg {

bool launch_f32_reg(const StepArgs &a, bool stats, cudaStream_t s, cudaStream_t side)
{
    return launch_typed<float, 2, true>(a, stats, s, side);
}

}  // namespace stg
