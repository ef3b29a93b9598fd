// Host-side launch of one fused step pass (the kernels: step_kernel.cuh and
// its instantiation units), the initial-state kernel, the statistics
// reduction of sampling steps and the FP64 mass reduction.
#include <algorithm>

#include <cuda_fp16.h>

#include "d3q19.cuh"
#include "internal.h"
#include "lbm_cell.cuh"
#include "reduce.cuh"

namespace stg {

constexpr int BX = 32;

// instantiation units (step_<storage>_<collision>[_quad|_row].cu)
using Pass = bool (*)(const StepArgs &a, bool stats, cudaStream_t s, cudaStream_t side);
bool launch_f32_reg(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f32_bgk(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16_reg(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16_reg_quad(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16_bgk(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16_bgk_quad(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16sr_reg(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16sr_reg_quad(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16sr_bgk(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16sr_bgk_quad(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f32_reg_row(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f32_bgk_row(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16_reg_row(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16_bgk_row(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16sr_reg_row(const StepArgs &, bool, cudaStream_t, cudaStream_t),
    launch_f16sr_bgk_row(const StepArgs &, bool, cudaStream_t, cudaStream_t);

// One plane and 32 cells per item, at most the 65535 runs of a launch per row; lattices
// beyond 32-bit element offsets take one cell per thread in whole columns.
int step_grid_blocks(int nx, int ny, int nz)
{
    const long long col = (long long)((nx + BX - 1) / BX) * ny;
    const long long runs = 19.0 * nx * ny * nz < 4294967296.0 ? std::min(nz, 65535) : 1;
    return (int)(col * runs + 2LL * ny + 64);
}

// The longer a run, the less scratch a sampling step writes and reads (36 B each
// per cell and run), and the longer the serial walk of its warps: 32 planes (8 per
// warp), but less where that leaves the GPU's resident warps less than one and a
// half chunks of 64 cells each (a plane takes a warp 2 to 4 us when little else is
// in flight: 64x32x32 spent 160 us on a sampling step of one 32-plane run per warp).
int stat_group(int nx, int ny, int nz)
{
    const long long rows = (long long)((nx + 2 * BX - 1) / (2 * BX)) * ny;
    int g = 32;
    while (g > STAT_WARPS && rows * ((nz + g - 1) / g) * STAT_WARPS < 152LL * 32 * 3 / 2 && nz / (g / 2) < 65535) g /= 2;
    return std::max(g, (nz + 65534) / 65535);  // a launch holds 65535 runs
}

// the regularized collision without a force, whose kernels have the most warps per SM
static bool lean(const StepArgs &a) { return a.collision == 0 && !a.has_force; }
// FP32 pairs, BGK or a force (24 warps per SM), the last chunk of a row up to three
// quarters full
static bool ragged_fp32(const StepArgs &a)
{
    return a.storage == 0 && !lean(a) && !row_lanes(a) && a.nx % 64 != 0 && a.nx % 64 <= 48;
}

// FP32 lattices with fewer than 4 cells per resident lane (32 warps per SM, 622592
// cells): one cell per lane halves the serial work of a warp (us per step, one cell
// per lane and pairs, each with the better number of launches: 96x16x24 3.7 and 5.2,
// 144x24x36 6.0 and 7.4, 240x40x60 15.0 and 17.8).  The line is on the safe side: one
// cell per lane in two launches stays ahead to about 2 million cells (252x42x63 17.4
// and 22.0, 324x54x81 38.9 and 42.8, 360x60x90 49.6 and 51.3).
static bool small_row(const StepArgs &a)
{
    return std::max<long long>(a.P, a.in_flight) < 4LL * 152 * 32 * 32;
}

// Rows of fewer than 32 cells in binary16: a lane's other three cells lie outside the
// row, and once such rows fill the GPU one cell per thread is the faster form (from 24
// rows x planes per resident warp on, with stochastic rounding 19: 5x300x300 132 against
// 145 us per step, 141 against 171; 31x260x260 126 against 114, 133 against 139).
static bool narrow_rows(const StepArgs &a)
{
    return a.storage != 0 && a.nx < 32 && (long long)a.ny * a.nz >= 152LL * 20 * (a.storage == 2 ? 19 : 24);
}

bool row_lanes(const StepArgs &a)
{
    if (a.aa || a.interior != 0 || 19.0 * a.P >= 4294967296.0) return false;
    if (narrow_rows(a)) return false;
    return a.nx % 2 != 0 || a.nx < 4 || (a.storage == 0 && small_row(a));
}

// Binary16 BGK lattices whose rows split into quads take pairs all the same where the
// quads' wider chunks (128 cells, 16 warps per SM) lose more than their accesses gain:
// at an inlet and an outlet, where the chunks with a node go cell by cell, up to the
// length where the others outweigh them (round to nearest 580 cells, stochastic
// rounding 720: us per step with quads and pairs, 160^3 91.0 and 73.9, 200^3 147 and
// 136, 520x128x128 135.5 and 129.1, 640x128x128 144.5 and 148.4; stochastic rounding
// 160^3 95.6 and 79.2, 700x128x128 183 and 173, 768x128x192 260 and 267); in a periodic
// box with round to nearest (160^3 85.7 and 68.5, 768x128x128 184.6 and 181.8) and, with
// stochastic rounding, where pairs also fill their chunks better (320x160x160 142.5 and
// 133.3, 768x128x128 191 and 207); in place (768x160x160 SR 329 and 318).
static bool bgk_pairs(const StepArgs &a)
{
    const bool sr = a.storage == 2;
    if (a.aa) return true;
    if (a.bc_x != 0) return !sr || 2 * ((a.nx + 127) / 128) != (a.nx + 63) / 64;
    return a.nx <= (sr ? 720 : 580);
}

int lane_cells(const StepArgs &a)
{
    if (row_lanes(a)) return a.storage != 0 ? 4 : (small_row(a) ? 1 : 2);
    const bool quads = a.storage != 0 && quads_fit(a.nx) && vector_fits(a) && !(a.collision != 0 && bgk_pairs(a));
    return quads ? 4 : 2;
}

// Items: one x chunk (32 cpl cells) of one row and plane each, of all lattices
// that advance together.  While the GPU's warps (16 per SM with the registers of
// the kernel for any row) have only a few each, a pass is bound by launches and by
// the latency of one plane, and one launch of all rows saves the branch of the wall
// rows; above that the inner rows' own kernel, with more warps per SM, is the faster
// one.  us per step, one launch and two, by items per warp:
//   FP32, one cell per lane: 0.5 3.7 and 5.7, 1.8 6.0 and 6.9, 2.9 8.0 and 7.7, 3.8
//     9.6 and 8.7, 5.6 12.7 and 11.5, 7.9 18.7 and 15.0 (the line at 4 gives away up to
//     a tenth between 2.5 and 4)
//   binary16 quads (the line at 1.5): 240x40x60 (2.0) 14.4 and 13.2; 324x54x81 (5.4)
//     35.0 and 30.6
//   binary16 pairs (the line at 1.5): 142x24x36 (1.1) 6.8 and 5.2, one step alone 10.7
//     and 11.0; 182x30x45 (1.7) 7.5 and 6.0; 230x38x57 (3.6) 11.6 and 9.2; BGK with
//     stochastic rounding 240x40x60 (4.0) 14.3 and 12.1; in place 206x34x51 (2.9) 10.7
//     and 10.3
//   FP32 pairs (from 622592 cells, 4 items per warp, on: always two): 300x50x75 39.4
//     and 38.2, 324x54x81 51.6 and 42.8, 384x64x96 73 and 57
static long long items_of(const StepArgs &a, int cpl)
{
    const long long own = (long long)((a.nx + BX * cpl - 1) / (BX * cpl)) * a.ny * a.nz;
    return std::max(own, a.in_flight / (BX * cpl));
}

bool one_launch(const StepArgs &a, int cpl)
{
    return a.ny < 3 || items_of(a, cpl) * 2 < 152LL * 16 * (a.storage != 0 ? 3 : 8);
}

// Runs of 4 planes in the wall rows, else 1: where the inner rows take long enough to
// hide the latency of a walk of 4 planes, which FP32 pairs do from 7 items per resident
// warp on (us per step with 1, 2, 4: 264x44x66 20.3, 20.8, 28.4; 300x50x75 30.5, 30.6,
// 36.7; 360x60x90 48.7, 48.9, 49.3; 384x64x96 57.3, 57.1, 56.4; 768x128x192 417, 416,
// 415).  FP32 lanes 32 cells apart are the same either way (240x40x60 13.6, 13.6, 13.6;
// 385x64x96 64.1, 63.9, 64.2).  Binary16 1 (768x128x192 226, 228, 230, 236 with 24), but
// 4 among the members of a batch.
// A run of several planes costs one block start instead of several, but a pass
// ends with its last runs, and a short pass needs every warp from the start: so
// runs grow with the number of items per resident warp, up to what the form takes:
//  FP32 (256 B per row piece) 2 (768x128x192: 415, 418, 425 us with 2, 4, 8;
//    1536x256x384: 3.27, 3.29, 3.31, 3.34 ms with 1, 2, 4, 8), with BGK or a force and
//    a ragged last chunk 4 (200^3 228, 218, 216 us with 2, 4, 8; full rows stay at 2:
//    320x160x160 193, 193, 197, 256x128x128 97.6, 98.4, 106.7);
//  binary16 quads 8 (1536x256x384: 1.82, 1.76, 1.72, 1.72 ms with 1, 2, 4, 8;
//    384x64x96: 2), in place 4 (us with 2, 4, 8: round to nearest 320x128x200 140.9, 140.7,
//    146.1, 512x128x128 121.7, 122.8, 128.5, 768x128x192 246, 248, 253, stochastic rounding
//    276, 273, 276, 1536x128x192 496, 489, 490);
//  binary16 pairs (128 B) 2, with BGK or a force 4 (250x125x125 61.8, 64.9, 69.1 us with
//    2, 4, 8, 770x128x192 282, 293, 305; BGK 200^3 142, 136, 142);
//  binary16 lanes 32 cells apart 2 (767x127x191: 302, 308, 321 us with 2, 4, 8, 63x300x300
//    174, 179, 184).
// The wall rows, beside the inner launch, are spread over as many warps as their
// latency needs (long_walls).
// A tile that was set sets the runs instead.
static bool long_walls(const StepArgs &a, int cpl)
{
    if (a.storage != 0) return a.in_flight > a.P;
    return cpl == 1 || row_lanes(a) || items_of(a, cpl) >= 7 * 152 * 32;
}

int run_planes(const StepArgs &a, int cpl, bool walls)
{
    const int least = (a.nz + 65534) / 65535;  // a launch holds 65535 runs
    const int tile = walls ? a.tile_wall_zc : a.tile_zc;
    if (tile > 0) return std::max(least, std::min(tile, a.nz));
    const bool fp32 = a.storage == 0;
    if (walls) return std::max(least, std::min(a.nz, long_walls(a, cpl) ? 4 : 1));
    int most = ragged_fp32(a) ? 4 : 2;
    if (!fp32 && !row_lanes(a)) most = cpl == 4 ? (a.aa ? 4 : 8) : (lean(a) ? 2 : 4);
    // (binary16: by the cells that the items hold, for rows that fill a fraction of one)
    const long long items = fp32 ? items_of(a, cpl) : std::max<long long>(a.P, a.in_flight) / (BX * cpl);
    const long long per_warp = items / (152 * (fp32 ? 32 : 20));
    int zc = 1;
    while (zc < most && per_warp >= 5 * zc) zc *= 2;
    return std::max(least, std::min(zc, a.nz));
}

// Warps (x chunks) of a block: as many as leave the fewest idle; one where a block of
// several waits for the slowest of chunks that differ: stochastic rounding in pairs
// (210^3 155.8 us per step with one, 157.3 with four, 250x125x125 66.3 and 67.1), and
// ragged FP32 rows (200^3 BGK 209.6 and 217.0, 210^3 249.6 and 256.3).
int block_chunks(const StepArgs &a, int cpl, int chunks, int most)
{
    if ((a.storage == 2 && cpl == 2) || ragged_fp32(a)) return 1;
    int nw = most;
    for (int k = nw - 1; k > 0; --k)
        if ((chunks + k - 1) / k * k < (chunks + nw - 1) / nw * nw) nw = k;
    return nw;
}

// Adds the z-group sums of a sampling step to the FP64 statistics, group by
// group in index order (one thread per (x, y) and moment).
__global__ void stats_reduce_kernel(const float *part, int groups, size_t m, double *stat_mean, double *stat_rey)
{
    const size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x;  // q * m + xy
    if (k >= 9 * m) return;
    // the groups in index order as a compensated FP32 sum (the two-sum error
    // of every addition is kept: hi + lo holds the sum to about 2^-44 of its
    // size), then one FP64 addition into the running sum; GB300's FP64 rate
    // is a small fraction of its FP32 rate, and an FP64 conversion and add per
    // group made this kernel FP64-bound
    float hi = 0.f, lo = 0.f;
#pragma unroll 8
    for (int g = 0; g < groups; ++g) {
        const float x = __ldcs(part + (size_t)g * 9 * m + k);
        const float s = hi + x;
        const float z = s - hi;
        lo += (hi - (s - z)) + (x - z);
        hi = s;
    }
    const double sum = (double)hi + (double)lo;
    if (k < 3 * m) stat_mean[k] += sum;
    else stat_rey[k - 3 * m] += sum;
}

// One fused step pass.  The wall rows (or the edge kernel of the one-cell-per-
// thread path) run on the forked branch `side` beside the inner rows (they write
// disjoint slots); `s` waits for both.  A pass of one launch needs no branch.
cudaError_t launch_step(const StepArgs &a, bool stats, cudaStream_t s, cudaStream_t side, cudaEvent_t fork,
                        cudaEvent_t join)
{
    cudaError_t e = cudaSuccess;
    const int cpl = lane_cells(a);
    const bool one = (vector_fits(a) || row_lanes(a)) && one_launch(a, cpl);
    const bool forked = !one && side != nullptr && fork != nullptr && join != nullptr;
    if (forked) {
        if ((e = cudaEventRecord(fork, s)) != cudaSuccess) return e;
        if ((e = cudaStreamWaitEvent(side, fork, 0)) != cudaSuccess) return e;
    }
    cudaStream_t es = forked ? side : s;
    // by storage and collision: pairs (or one cell per thread), quads, lanes 32 cells apart
    static constexpr Pass passes[3][2][3] = {
        {{launch_f32_reg, nullptr, launch_f32_reg_row}, {launch_f32_bgk, nullptr, launch_f32_bgk_row}},
        {{launch_f16_reg, launch_f16_reg_quad, launch_f16_reg_row}, {launch_f16_bgk, launch_f16_bgk_quad, launch_f16_bgk_row}},
        {{launch_f16sr_reg, launch_f16sr_reg_quad, launch_f16sr_reg_row},
         {launch_f16sr_bgk, launch_f16sr_bgk_quad, launch_f16sr_bgk_row}}};
    const bool reduce = passes[a.storage][a.collision][row_lanes(a) ? 2 : (cpl == 4 ? 1 : 0)](a, stats, s, es);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (forked) {
        if ((e = cudaEventRecord(join, side)) != cudaSuccess) return e;
        if ((e = cudaStreamWaitEvent(s, join, 0)) != cudaSuccess) return e;
    }
    if (reduce) {
        const size_t m = (size_t)a.nx * a.ny;
        const int groups = (a.nz + a.stat_group - 1) / a.stat_group;
        const unsigned blocks = (unsigned)((9 * m + 255) / 256);
        stats_reduce_kernel<<<blocks, 256, 0, s>>>(a.stat_part, groups, m, a.stat_mean, a.stat_rey);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Initial state f^eq(1, (u_int(y), 0, 0)) (u_int == nullptr: rest state),
// stored shifted; `swap` stores population i in slot opp(i) (the in-place
// layout before a step with even index).
template <typename S>
__global__ void init_eq_kernel(S *dst, int nx, int ny, int nz, const float *u_int, int swap)
{
    const size_t P = (size_t)nx * ny * nz;
    for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < P; c += (size_t)gridDim.x * blockDim.x) {
        const int y = (int)((c / nx) % ny);
        const float ux = u_int ? u_int[y] : 0.0f;
#pragma unroll
        for (int i = 0; i < Q; ++i)
            Pop<S>::st(dst + (size_t)(swap ? opp_of(i) : i) * P + c, geq(w_of(i), 0.0f, 1.0f, cx_of(i) * ux, ux * ux));
    }
}

cudaError_t launch_init_equilibrium(void *dst, int storage, int nx, int ny, int nz, const float *u_int, int swap,
                                    cudaStream_t s)
{
    const int blocks = 152 * 8;
    if (storage == 0) init_eq_kernel<float><<<blocks, 256, 0, s>>>(static_cast<float *>(dst), nx, ny, nz, u_int, swap);
    else init_eq_kernel<__half><<<blocks, 256, 0, s>>>(static_cast<__half *>(dst), nx, ny, nz, u_int, swap);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP64 mass of a stored lattice, sum over cells and populations, in a fixed
// reduction order (block partials, then the last block to finish adds them
// in index order).
constexpr int MASS_BLOCKS = 152 * 4;
constexpr int MASS_THREADS = 256;

template <typename S>
__global__ void __launch_bounds__(MASS_THREADS) mass_kernel(const MassArgs a)
{
    const S *src = static_cast<const S *>(a.src);
    __shared__ double ws[MASS_THREADS / 32];
    __shared__ int s_last;
    double acc = 0.0;
    for (size_t c = blockIdx.x * (size_t)MASS_THREADS + threadIdx.x; c < a.P; c += (size_t)gridDim.x * MASS_THREADS) {
        float r = 0.f;
#pragma unroll
        for (int i = 0; i < Q; ++i) r += Pop<S>::ld(src + (size_t)i * a.P + c);
        acc += (double)r;
    }
    const int tid = threadIdx.x;
    const double bs = block_sum<MASS_THREADS>(acc, ws);
    if (tid == 0) {
        a.partial[blockIdx.x] = bs;
        __threadfence();
        s_last = (atomicAdd(a.counter, 1u) == gridDim.x - 1);
    }
    __syncthreads();
    if (s_last) {
        double v = 0.0;
        for (unsigned k = tid; k < gridDim.x; k += MASS_THREADS) v += __ldcg(a.partial + k);
        const double tot = block_sum<MASS_THREADS>(v, ws);
        if (tid == 0) {
            a.out[0] = tot + (double)a.P;
            *a.counter = 0u;
        }
    }
}

int mass_grid_blocks() { return MASS_BLOCKS; }

cudaError_t launch_mass(const MassArgs &a, cudaStream_t s)
{
    if (a.storage == 0) mass_kernel<float><<<MASS_BLOCKS, MASS_THREADS, 0, s>>>(a);
    else mass_kernel<__half><<<MASS_BLOCKS, MASS_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace stg
