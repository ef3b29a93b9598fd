// Block-level reductions shared by the step kernels.
#pragma once

#include "internal.h"

namespace stg {

// Sum of one double per thread over a block of NT threads (a multiple of 32,
// at most 1024) in a fixed order: a butterfly of warp shuffles inside each
// warp, then warp 0 adds the warp sums by the same butterfly.  Every thread of
// the block must call it (it holds a barrier); the result is meant for thread
// 0 (each lane's butterfly associates the terms its own way, lane 0's always
// the same).  ws: shared scratch of NT / 32 doubles.
template <int NT>
__device__ __forceinline__ double block_sum(double v, double *ws)
{
    static_assert(NT % 32 == 0 && NT <= 1024, "whole warps");
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((tid & 31) == 0) ws[tid >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (tid < 32) {
        s = tid < (int)(blockDim.x * blockDim.y) / 32 ? ws[tid] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    return s;
}

// Deterministic FP64 mass of a step pass: each block leaves the sum of its
// threads' (rho - 1) in its own slot, a.slot_base + its linear block index (x
// fastest, then y, then z).  Of every MASS_GROUP consecutive blocks of the pass's
// total_blocks (all kernels) the last to finish adds the group's slots in index
// order (each thread a strided subset, then the block sum), and the last group
// adds the groups' sums and writes nx ny nz + sum.  One level alone left one
// block, of a single warp with quads, to add every slot: 146 000 of them, 1.4 ms,
// on 1536x256x384.  NT = most threads per block.
template <int NT>
__device__ __forceinline__ void mass_finish(const StepArgs &a, float sdr)
{
    __shared__ double ws[NT / 32];
    __shared__ int s_last;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const unsigned nt = blockDim.x * blockDim.y;
    const unsigned groups = (a.total_blocks + MASS_GROUP - 1) / MASS_GROUP;
    const unsigned slot = a.slot_base + (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    const unsigned g = slot / MASS_GROUP;
    double *const gsum = a.mass_partial + a.total_blocks;
    // leaves `v` in *p and returns whether this block is the last of `n` to do so
    auto last_of = [&](double *p, double v, unsigned *count, unsigned n) {
        if (tid == 0) {
            *p = v;
            __threadfence();
            s_last = (atomicAdd(count, 1u) == n - 1);
        }
        __syncthreads();
        const bool last = s_last != 0;
        if (last) {
            __threadfence();
            if (tid == 0) *count = 0u;
        }
        return last;
    };
    auto sum_of = [&](const double *p, unsigned n) {
        double acc = 0.0;
#pragma unroll 4
        for (unsigned k = tid; k < n; k += nt) acc += __ldcg(p + k);
        __syncthreads();  // s_last and ws are read
        return block_sum<NT>(acc, ws);
    };
    const double bs = block_sum<NT>((double)sdr, ws);
    const unsigned gn = min((unsigned)MASS_GROUP, a.total_blocks - g * MASS_GROUP);
    if (!last_of(a.mass_partial + slot, bs, a.mass_counter + g, gn)) return;
    const double gs = sum_of(a.mass_partial + g * MASS_GROUP, gn);
    if (!last_of(gsum + g, gs, a.mass_counter + groups, groups)) return;
    const double tot = sum_of(gsum, groups);
    if (tid == 0) a.mass_out[0] = tot + (double)a.P;
}

}  // namespace stg
