// Kernel argument blocks and launcher declarations shared by the library's
// translation units (host API, step kernel, inlet kernel).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace stg {

// Step counter on the device.  Step t reads t[t & 1]; the fused step kernel
// writes t[(t + 1) & 1] = t + 1 when it finishes, so a captured graph can be
// replayed without host-side parameter updates.
struct StepCtl {
    long long t[2];
    long long t0_filter;  // step at which the temporal filter restarts
    long long t_block;    // step at which the current block of steps began
    long long t_probe;    // probed blocks: step index before the first one of the call
    float *probe_out;     // and its samples [steps][3 n]
    unsigned long long err; // error bits set by kernels (none of the current kernels sets one)
};

// Inlet velocity planes are kept in a ring by step index (a power of two).  A
// launch computes at most INLET_MAX_PLANES of them; the steps of a block read the
// planes of one launch while the next launch writes its own.
constexpr int INLET_RING = 32, INLET_MAX_PLANES = 16;

struct StepArgs {
    const void *src;      // post-collision populations of the previous step
    void *dst;            // post-collision populations of this step
    // per-population plane pointers (kernel parameters, so every address is
    // one multiply-add of the cell index onto a constant-bank operand):
    //   srcp[i] = plane i of src, srci[i] = srcp[i] - (c_ix + c_iy nx) elements
    //   (interior pull), dstp[i] = plane i of dst
    //   srcy[i] = srcp[i] - c_iy nx elements (two-cells-per-thread pull)
    const void *srcp[19];
    const void *srci[19];
    const void *srcy[19];
    void *dstp[19];
    int il, ir;             // 32-wide x chunks [il, ir) of rows 1..ny-2 belong to the interior kernel
    int interior;           // interior kernel: 0 best available, 1 one cell per thread, 2 cell pairs
    int aa;                 // 1: one lattice updated in place (AA pattern; src == dst), 0: two lattices
    // z planes per run of the plain (non-sampling) vector launches, inner / wall rows: the
    // set tile's, 0 by the lattice's size (run_planes); in a launch its own
    int tile_zc, tile_wall_zc;
    int row_step;           // vector launches of the rows 0, row_step, ...
    int stat_group;         // z planes per run of the sampling vector launches
    unsigned total_blocks;  // blocks of all step kernels of the pass (mass-check completion count)
    int slot_base;          // first mass-partial slot of this launch's blocks
    int nx, ny, nz;
    unsigned P;           // cells per population plane (nx*ny*nz)
    long long in_flight;  // cells of all lattices advanced together (a batch's members; else P)
    int bc_x, bc_y;       // STG_BC_X_*, STG_BC_Y_*
    int storage, collision;  // stg_domain's
    float tau0, kq;       // kq = 18 sqrt(2) C  (eq. tau_eff)
    float Fx, Fy, Fz;
    int has_force;
    const float *ubc;     // inlet velocity planes [INLET_RING][3][nz][ny], step t in plane t mod INLET_RING
    const float *spf;     // sponge zone: viscosity factor per column x [nx] (eq. sponge_visco); nullptr: off
    StepCtl *ctl;
    int parity;
    int stats_every, check_every;
    double *stat_mean;    // [3][ny][nx]
    double *stat_rey;     // [6][ny][nx]
    float *stat_part;     // sampling steps of the vector kernels: FP32 sums per run of
                          // stat_group z planes, [ceil(nz / stat_group)][9][ny][nx]
    double *mass_partial; // one slot per block, then one per MASS_GROUP blocks
    unsigned *mass_counter;  // one per MASS_GROUP blocks, then one
    double *mass_out;     // [0]: last checked mass
};

struct InletArgs {
    int ny, nz, N;
    const float2 *AS;     // [N][ny]  k^n d^n_y (j + 1/2) mod 2 pi, sqrt(6 q^n(y_j))
    const float *BS;      // [N][nz]  k^n d^n_z k mod 2 pi
    const float *sig;     // [N][3]   sigma^n
    const unsigned long long *phq;  // [N] phi^n / (2 pi) as a Q0.64 fraction of a turn
    const unsigned long long *omq;  // [N] phase advance per step, -d^n_x U_b / max l_e turns, Q0.64
    const float *a6;      // [ny][6]  Cholesky factor a11 a21 a22 a31 a32 a33
    const float *u_int;   // [ny]     interpolated mean streamwise velocity
    float a_filter;
    float *uf;            // [3][nz][ny] filtered fluctuation (state)
    float *ubc;           // inlet velocity planes, as in StepArgs (output)
    int ahead, planes;    // the planes of steps t + ahead .. t + ahead + planes - 1
    int from_block;       // t: 0 ctl->t[parity] (noted as ctl->t_block), 1 ctl->t_block
    StepCtl *ctl;
    int parity;
};

struct MassArgs {
    const void *src;
    unsigned P;
    int storage;
    double *partial;
    unsigned *counter;
    double *out;
};

// launchers (return the launch status)
// `stats` must be true exactly on sampling steps ((t + 1) % stats_every == 0);
// the host tracks t and decides.
cudaError_t launch_step(const StepArgs &a, bool stats, cudaStream_t s, cudaStream_t side, cudaEvent_t fork,
                        cudaEvent_t join);
// whether the rows split into whole quads (four cells per lane, binary16)
inline bool quads_fit(int nx) { return nx % 4 == 0 && nx >= 8; }
// Lattices of aligned vectors (the others take lanes 32 cells apart, or one cell per
// thread): rows of whole pairs and 32-bit element offsets.  The in-place scheme exists for them
// only (the host checks its conditions), so it ignores the interior override.
inline bool vector_fits(const StepArgs &a)
{
    return (a.aa || a.interior == 0 || a.interior == 2) && a.nx % 2 == 0 && a.nx >= 4 &&
           19.0 * a.nx * a.ny * a.nz < 4294967296.0 && (a.bc_x != 0 || a.nx >= 3);
}
// Whether a pass of the vector kernels (cpl cells per lane) is one launch of all
// rows, and the z planes per run of its launches (step_kernel.cu).
bool one_launch(const StepArgs &a, int cpl);
int run_planes(const StepArgs &a, int cpl, bool walls);
// warps of a block of such a launch, `most` of them at most
int block_chunks(const StepArgs &a, int cpl, int chunks, int most);
// cells per lane of the vector kernels, and whether they lie 32 apart
int lane_cells(const StepArgs &a);
bool row_lanes(const StepArgs &a);
cudaError_t launch_inlet(const InletArgs &a, cudaStream_t s);
// FP64 Cholesky factor of the lattice-unit Reynolds stress per inlet node (setup)
cudaError_t launch_setup_nodes(int ny, const double *R6, float *a6, cudaStream_t s);
// swap: store population i in slot opp(i) (the in-place layout before a step of even index)
cudaError_t launch_init_equilibrium(void *dst, int storage, int nx, int ny, int nz, const float *u_int, int swap,
                                    cudaStream_t s);
cudaError_t launch_mass(const MassArgs &a, cudaStream_t s);
// How to find a population in a stored lattice: slot i of the cell for two
// lattices, the in-place arrangement after t completed steps otherwise.
struct LatticeView {
    int nx, ny, nz, bc_x, bc_y, aa;
    size_t P;
    long long t;
};
// velocity of n cells (xyz: device int triples) of the lattice stored after lv.t
// steps, into out or (NULL) the place of that step in the series of ctl, which
// launch_probe_series sets for the steps from t on
cudaError_t launch_probe(const void *src, int storage, const LatticeView &lv, int n, const int *xyz, float Fx,
                         float Fy, float Fz, const StepCtl *ctl, float *out, cudaStream_t s);
cudaError_t launch_probe_series(StepCtl *ctl, long long t, float *out, cudaStream_t s);
// canonical sub-block [19][bz][by][bx] of a stored lattice into device memory `out`
cudaError_t launch_gather_block(const void *src, int storage, const LatticeView &lv, int x0, int y0, int z0, int bx,
                                int by, int bz, void *out, cudaStream_t s);

// Tiles: shortest z chunk that set_tile accepts; the default chunks (layout 1), which
// leave the runs to run_planes; warps that share a chunk of layout 0 or of the wall rows.
constexpr int MIN_ZC = 4, DEFAULT_ZC = 8, DEFAULT_WALL_ZC = 24, TILE_WARPS = 8;
// z planes per run on sampling steps of the vector kernels, walked by STAT_WARPS
// warps: a function of the lattice alone, so the statistics do not depend on the
// launch tile
constexpr int STAT_WARPS = 4;
int stat_group(int nx, int ny, int nz);
// Upper bound of the blocks of one step pass over every tile.
int step_grid_blocks(int nx, int ny, int nz);
// Blocks whose mass partials are added by the last of them to finish.
constexpr int MASS_GROUP = 1024;
inline int mass_groups(int blocks) { return (blocks + MASS_GROUP - 1) / MASS_GROUP; }
int mass_grid_blocks();

}  // namespace stg
