// The plane loop of lattices whose rows do not split into aligned vectors (odd
// nx), and of FP32 lattices too small to give every warp a pair of cells per
// lane: lane l of a warp owns the cells x0 + l, x0 + 32 + l, ... (CPL of them), so
// every access is a coalesced run of single elements at any alignment, and the
// x neighbours are the same runs one element to the side (no shuffle, no halo
// case).  What keeps the bytes in flight that an aligned vector keeps is CPL
// independent loads per population (FP32 2, binary16 4, whose pairs of cells go
// through the packed collision).  One cell per thread in whole-column blocks, the
// form before, and this loop, us per step:
//                        385x65x97     767x127x191
//   FP32                 93 -> 66      733 -> 452    (55 and 423 at the copy rate)
//   binary16             70 -> 54      464 -> 301    (28 and 211)
//   stochastic rounding  73 -> 69      484 -> 379
//   the same, BGK        74 -> 71      483 -> 405
// What is left is the odd alignment (a run of 32 lanes touches one sector more than
// it fills: FP32 4.5 for 4, binary16 2.7 for 2) and, for binary16, instructions: 2-byte
// accesses and a random word per cell, 15.3 per cell and warp against 7.9 with quads.
// (Rows of fewer than 32 cells, large binary16 lattices: one cell per thread, narrow_rows().)
#pragma once

#include <cuda_fp16.h>

#include "d3q19.cuh"
#include "internal.h"
#include "lbm_cell.cuh"
#include "lbm_pair.cuh"

namespace stg {

// The lane's cells of one population: cell j at p + 32 j.
template <typename S, int CPL>
struct Strip;

template <int CPL>
struct Strip<float, CPL> {
    float f[CPL];
    __device__ __forceinline__ void ld(int j, const float *p, bool on) { f[j] = on ? __ldg(p + 32 * j) : 0.f; }
    __device__ __forceinline__ float cell(int j) const { return f[j]; }
    __device__ __forceinline__ float2 pair(int k) const { return make_float2(f[2 * k], f[2 * k + 1]); }
    __device__ __forceinline__ void put(int j, float r) { f[j] = r; }
    __device__ __forceinline__ void st(int j, float *p) const { __stcs(p + 32 * j, f[j]); }
};

template <int CPL>
struct Strip<__half, CPL> {
    static_assert(CPL % 2 == 0, "whole pairs");
    unsigned w[CPL / 2];  // cells 2k (low half) and 2k + 1
    __device__ __forceinline__ void ld(int j, const __half *p, bool on)
    {
        const unsigned h = on ? (unsigned)__half_as_ushort(__ldg(p + 32 * j)) : 0u;
        if (j & 1) w[j / 2] = __byte_perm(w[j / 2], h, 0x5410);
        else w[j / 2] = h;
    }
    __device__ __forceinline__ float cell(int j) const
    {
        return __half2float(__ushort_as_half((unsigned short)(j & 1 ? w[j / 2] >> 16 : w[j / 2] & 0xffffu)));
    }
    __device__ __forceinline__ float2 pair(int k) const
    {
        float2 f;
        asm("{.reg .b16 lo, hi; mov.b32 {lo, hi}, %2; cvt.f32.f16 %0, lo; cvt.f32.f16 %1, hi;}"
            : "=f"(f.x), "=f"(f.y) : "r"(w[k]));
        return f;
    }
    // cells 2k, 2k + 1 in one conversion (round to nearest, or stochastic rounding with bits rb)
    __device__ __forceinline__ void set_pair(int k, float lo, float hi)
    {
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(w[k]) : "f"(hi), "f"(lo));
    }
    __device__ __forceinline__ void set_pair_rs(int k, float lo, float hi, unsigned rb)
    {
        asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(w[k]) : "f"(hi), "f"(lo), "r"(rb));
    }
    __device__ __forceinline__ void st(int j, __half *p) const
    {
        __stcs(p + 32 * j, __ushort_as_half((unsigned short)(j & 1 ? w[j / 2] >> 16 : w[j / 2] & 0xffffu)));
    }
};

// Velocity of a cell from its streamed populations, for the outlet node beside it:
// with the sums in population order (odd nx), or with collide()'s rounding (ORDER
// false: what the pairs of even nx take).
template <bool FORCE, bool ORDER>
__device__ __forceinline__ void cell_velocity(const float (&g)[Q], float Fx, float Fy, float Fz, float &ux, float &uy,
                                              float &uz)
{
    float drho = 0.f, jx = 0.f, jy = 0.f, jz = 0.f;
    if (ORDER) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            drho += g[i];
            if (cx_of(i)) jx += cx_of(i) * g[i];
            if (cy_of(i)) jy += cy_of(i) * g[i];
            if (cz_of(i)) jz += cz_of(i) * g[i];
        }
    } else {
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            const int i = 2 * p + 1;
            const float s = g[i] + g[i + 1], d = g[i] - g[i + 1];
            drho = p ? drho + s : g[0] + s;
            if (cx_of(i)) jx += cx_of(i) * d;
            if (cy_of(i)) jy += cy_of(i) * d;
            if (cz_of(i)) jz += cz_of(i) * d;
        }
    }
    const float irho = 1.0f / (1.0f + drho);
    ux = (FORCE ? fmaf(0.5f, Fx, jx) : jx) * irho;
    uy = (FORCE ? fmaf(0.5f, Fy, jy) : jy) * irho;
    uz = (FORCE ? fmaf(0.5f, Fz, jz) : jz) * irho;
}

// Cells of a row that lie before its first chunk: with an outlet node that would be
// the first of its 32 cells (nx = 1 mod 32) the chunks begin one cell early, so that
// the node's neighbour is always the lane beside it.
__host__ __device__ inline int row_shift(int nx, bool xopen) { return xopen && nx % 32 == 1 ? 1 : 0; }

// Row y, cells x0 .. x0 + 32 CPL - 1 (x0 may be -1, see row_shift) over the planes
// zb, zb + zs, ... below ze, two lattices (pull).  XOPEN: inlet/outlet in x; the cells beside the ends then read
// the element before or after their row (inside the 19-plane allocation, see
// vec_loop) in place of the unknowns that the rebuilds replace.  The other
// arguments and the result are vec_loop's.
template <typename S, int CPL, bool REG, bool FORCE, bool STATS, bool YEDGE, bool SP, bool XOPEN, bool SR>
__device__ __forceinline__ float row_loop(const StepArgs &a, float (*sacc)[9][32 * CPL], unsigned (*keep)[Q], int x0,
                                          int y, int zb, int ze, int zs)
{
    // binary16: pairs of cells in packed FP32, an inlet or outlet node by itself afterwards
    constexpr bool PACKED = sizeof(S) == 2;
    const int nx = a.nx, ny = a.ny, nz = a.nz, nxy = nx * ny;
    const int lane = threadIdx.x, wi = threadIdx.y;
    const int x = x0 + lane;
    auto on = [&](int j) { return (unsigned)(x + 32 * j) < (unsigned)nx; };
    // whether the inlet / outlet node is cell j of some lane
    auto has_inlet = [&](int j) { return XOPEN && j == 0 && x0 <= 0; };
    auto has_outlet = [&](int j) { return XOPEN && x0 + 32 * j < nx && x0 + 32 * j + 32 >= nx; };
    bool ym_bb = false, yp_bb = false;
    int ym_off = nx, yp_off = -nx;
    if (YEDGE) {
        const bool walls = a.bc_y == 0;
        if (y == 0) {
            if (walls) ym_bb = true;
            else ym_off = -(ny - 1) * nx;
        }
        if (y == ny - 1) {
            if (walls) yp_bb = true;
            else yp_off = (ny - 1) * nx;
        }
    }
    const float tau0 = a.tau0, kq = a.kq, Fx = a.Fx, Fy = a.Fy, Fz = a.Fz;
    const S *__restrict__ sbase = static_cast<const S *>(a.src);
    S *__restrict__ dbase = static_cast<S *>(a.dst);
    const unsigned tmix = SR ? sr_tmix(a.ctl->t[a.parity]) : 0u;
    float sdr = 0.f;
    for (int z = zb; z < ze; z += zs) {
        // opaque copies, as in vec_loop: addresses are formed anew in every plane
        unsigned Pb, nxv;
        asm volatile("mov.u32 %0, %1;" : "=r"(Pb) : "r"(a.P * (unsigned)sizeof(S)));
        asm volatile("mov.u32 %0, %1;" : "=r"(nxv) : "r"((unsigned)nx));
        const unsigned row0 = ((unsigned)z * ny + y) * nx;
        const size_t here = (size_t)row0 + x;
        const unsigned dzm = (z == 0) ? -(nz - 1) * nxy : nxy;
        const unsigned dzp = (z == nz - 1) ? (nz - 1) * nxy : -nxy;
        Strip<S, CPL> v[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
            const bool bb = YEDGE && ((cy > 0 && ym_bb) || (cy < 0 && yp_bb));
            const unsigned dz = cz > 0 ? dzm : (cz < 0 ? dzp : 0u);
            const unsigned dy = cy > 0 ? (YEDGE ? (unsigned)ym_off : nxv) : (cy < 0 ? (YEDGE ? (unsigned)yp_off : 0u - nxv) : 0u);
            const size_t ofs = (size_t)(bb ? row0 : row0 - dz - dy);
            const S *p = reinterpret_cast<const S *>(reinterpret_cast<const char *>(sbase + ofs) + (size_t)(bb ? opp_of(i) : i) * Pb) +
                         (x - (bb ? 0 : cx));
#pragma unroll
            for (int j = 0; j < CPL; ++j) {
                const int xj = x + 32 * j;
                const S *q = p;
                if (!XOPEN && cx != 0 && !bb) {
                    if (cx > 0 && xj == 0) q += nx;
                    if (cx < 0 && xj == nx - 1) q -= nx;
                }
                v[i].ld(j, q, on(j));
            }
        }
        auto count = [&](int j, float drho, float ux, float uy, float uz) {
            if (!on(j)) return;
            if (STATS) {
                float *sp = &sacc[wi][0][stat_slot<ROW, CPL>(lane, j)];
                constexpr int L = 32 * CPL;
                sp[0 * L] += ux; sp[1 * L] += uy; sp[2 * L] += uz;
                sp[3 * L] = __fmaf_rn(ux, ux, sp[3 * L]); sp[4 * L] = __fmaf_rn(uy, uy, sp[4 * L]);
                sp[5 * L] = __fmaf_rn(uz, uz, sp[5 * L]); sp[6 * L] = __fmaf_rn(ux, uy, sp[6 * L]);
                sp[7 * L] = __fmaf_rn(ux, uz, sp[7 * L]); sp[8 * L] = __fmaf_rn(uy, uz, sp[8 * L]);
            }
            sdr += drho;
        };
        auto nu_factor = [&](int j) { return SP && on(j) ? __ldg(a.spf + x + 32 * j) : 1.0f; };
        // the node x = 0 or x = nx-1 in g; the outlet: rho = 1 and the velocity u of the
        // neighbour x = nx-2 at this step (the lane beside it: x0 is chosen so)
        auto node_of = [&](float (&g)[Q], int j, float ux, float uy, float uz) {
            if (has_inlet(j) && x + 32 * j == 0) inlet_node(a, g, (size_t)z * ny + y);
            if (has_outlet(j) && x + 32 * j == nx - 1) rebuild<-1>(g, 0.0f, ux, uy, uz);
        };
        auto from_left = [](float f) { return __shfl_up_sync(0xffffffffu, f, 1); };
        if constexpr (PACKED) {
#pragma unroll
            for (int k = 0; k < CPL / 2; ++k) {
                // a last chunk of up to 64 cells (385 = 3 x 128 + 1): one pair per lane, not two
                // (stochastic rounding 71.5 -> 69.1 us per step, BGK 76.1 -> 71.8)
                if (k > 0 && x0 + 64 * k >= nx) continue;
                // stochastic rounding: each cell has its own seed, its bits the low 13 of a word
                const unsigned s0 = SR ? sr_seed((unsigned)here + 64 * k, tmix) : 0u;
                const unsigned s1 = SR ? sr_seed((unsigned)here + 64 * k + 32, tmix) : 0u;
                auto bits = [&](int i) { return sr_bits_low2(s0, s1, i); };
                const float2 nuf = make_float2(nu_factor(2 * k), nu_factor(2 * k + 1));
                const bool nodes = has_inlet(2 * k) || has_outlet(2 * k) || has_outlet(2 * k + 1);
                // the lane of an inlet / outlet node keeps the pair's inputs (in shared
                // memory: no registers in the other warps)
                const int slot = k == 0 && x == 0 ? 0 : 1;
                if (nodes && (slot == 0 || x + 64 * k == nx - 1 || x + 64 * k + 32 == nx - 1)) {
#pragma unroll
                    for (int i = 0; i < Q; ++i) keep[slot][i] = v[i].w[k];
                }
                // the velocity of the cell to the left, for the outlet node
                float lx = 0.f, ly = 0.f, lz = 0.f;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    if (!has_outlet(2 * k + c)) continue;
                    float g[Q];
#pragma unroll
                    for (int i = 0; i < Q; ++i) g[i] = v[i].cell(2 * k + c);
                    cell_velocity<FORCE, true>(g, Fx, Fy, Fz, lx, ly, lz);
                    lx = from_left(lx), ly = from_left(ly), lz = from_left(lz);
                }
                auto pop = [&](int i) { return v[i].pair(k); };
                const PairMoments m = pair_moments(pop);
                float2 drho, ux, uy, uz;
                collide_pair_cell<REG, FORCE, SP>(m, pop, tau0, kq, nuf, Fx, Fy, Fz, [&](int i, float2 r) {
                    if constexpr (SR) v[i].set_pair_rs(k, r.x, r.y, bits(i));
                    else v[i].set_pair(k, r.x, r.y);
                }, drho, ux, uy, uz);
                if (nodes) {
                    // a short row can hold both nodes, in two lanes or in the two cells of one
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int j = 2 * k + c, xj = x + 32 * j;
                        if (!has_inlet(j) && !has_outlet(j)) continue;
                        if (!((has_inlet(j) && xj == 0) || (has_outlet(j) && xj == nx - 1))) continue;
                        float g[Q];
#pragma unroll
                        for (int i = 0; i < Q; ++i) g[i] = __half2float(__ushort_as_half((unsigned short)(c ? keep[slot][i] >> 16 : keep[slot][i])));
                        node_of(g, j, lx, ly, lz);
                        float dr, vx, vy, vz;
                        collide<REG, FORCE, SP>(g, tau0, kq, Fx, Fy, Fz, dr, vx, vy, vz, c ? nuf.y : nuf.x);
#pragma unroll
                        for (int i = 0; i < Q; ++i) {
                            const unsigned w = v[i].w[k];
                            if constexpr (SR) v[i].set_pair_rs(k, g[i], g[i], bits(i));
                            else v[i].set_pair(k, g[i], g[i]);
                            v[i].w[k] = __byte_perm(w, v[i].w[k], c ? 0x7610 : 0x3254);
                        }
                        (c ? drho.y : drho.x) = dr;
                        (c ? ux.y : ux.x) = vx;
                        (c ? uy.y : uy.x) = vy;
                        (c ? uz.y : uz.x) = vz;
                    }
                }
                count(2 * k, drho.x, ux.x, uy.x, uz.x);
                count(2 * k + 1, drho.y, ux.y, uy.y, uz.y);
            }
        } else {
#pragma unroll
            for (int j = 0; j < CPL; ++j) {
                float g[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) g[i] = v[i].cell(j);
                if (has_inlet(j) || has_outlet(j)) {
                    float ux = 0.f, uy = 0.f, uz = 0.f;
                    if (has_outlet(j)) {
                        if (nx & 1) cell_velocity<FORCE, true>(g, Fx, Fy, Fz, ux, uy, uz);
                        else cell_velocity<FORCE, false>(g, Fx, Fy, Fz, ux, uy, uz);
                        ux = from_left(ux), uy = from_left(uy), uz = from_left(uz);
                    }
                    node_of(g, j, ux, uy, uz);
                }
                float drho, ux, uy, uz;
                collide<REG, FORCE, SP>(g, tau0, kq, Fx, Fy, Fz, drho, ux, uy, uz, nu_factor(j));
#pragma unroll
                for (int i = 0; i < Q; ++i) v[i].put(j, g[i]);
                count(j, drho, ux, uy, uz);
            }
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            S *p = reinterpret_cast<S *>(reinterpret_cast<char *>(dbase + here) + (size_t)i * Pb);
#pragma unroll
            for (int j = 0; j < CPL; ++j)
                if (on(j)) v[i].st(j, p);
        }
    }
    return sdr;
}

}  // namespace stg
