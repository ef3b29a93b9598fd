// Synthetic turbulence generator on the inlet plane (Algorithm 1 steps 5-8)
// and the FP64 setup kernel for the per-node inlet tables (steps 3-4).
//
// Per inlet node (j, k) and step t:
//   v'  = sqrt(6) sum_n sqrt(q^n(j)) sigma^n cos(k^n d^n . x' + phi^n)     eq. (aux_vec)
//   with k^n d^n . x' = -2 pi d^n_x U_b t / max l_e + k^n (d^n_y y_j + d^n_z z_k)  eq. (psu), x = 0
//   u'  = a(j) v'                                                           eqs. (v_fluc), (cholesky)
//   u_f = a u_f + (1 - a) u'   (first-order temporal filter; u_f = u' at the first step)
//   u_bc = u_int(j) e_x + u_f                                               eqs. (u_phys), (u_transfer)
// The phase is split into three parts each already reduced to [0, 2 pi):
// the y part and the z part (tables built in FP64 on the host) and the time
// part phi^n + omega^n t, kept as Q0.64 fractions of a turn and advanced by
// wrapping 64-bit integer arithmetic (a phase accumulator: exact modulo a
// turn for any step count, no floating point); their FP32 sum is below 6 pi
// and is reduced to [-pi, pi] before the cosine.
//
// One launch computes the planes of `planes` consecutive steps (a block of steps
// asks for them a few and then 16 at a time, beside its passes, instead of one
// launch in every step).  A block of 8 warps covers 32 consecutive j (one per
// lane) and ITEMS = 8 IPW pairs (span node, step), IPW per warp in registers:
// IPW = 4 for more than 8 planes, 1 up to that, where the latency of the launch
// counts.  Per chunk of modes the block stages the y parts and amplitudes
// sqrt(6 q^n(j)), sigma^n and the items' time and z parts in shared memory, the
// table reads issued a chunk ahead; a mode then costs a warp 2 + IPW shared-memory
// reads and per item the phase sum and its reduction, one cosine and four
// multiply-adds.  The modes of even and of odd index are summed apart, each in
// order, and then added, in every form, so a plane's bits do not depend on how many
// were asked for.  The filter then runs over the steps in order, one thread per
// node.  (cos(a + b) by the addition theorem on sine and cosine tables halves the
// kernel's time, which passes hide almost all of, but rounds its planes otherwise,
// and binary16 storage turns that into differences of whole spacings.)
#include "internal.h"

namespace stg {

constexpr int INLET_J = 32;      // wall-normal nodes per block (one per lane)
constexpr int INLET_WARPS = 8;

template <int IPW>
__global__ void __launch_bounds__(INLET_J * INLET_WARPS, 2) stg_inlet_kernel(const InletArgs a, int kb)
{
    constexpr int ITEMS = IPW * INLET_WARPS;
    constexpr int CHUNK = IPW == 1 ? 96 : 32;              // modes staged per pass through shared memory
    constexpr int NT = INLET_J * INLET_WARPS;
    __shared__ float2 ys[CHUNK][INLET_J];                  // (y part, amplitude) per mode and wall-normal node
    __shared__ float2 is[CHUNK][ITEMS];                    // (time part, z part) per mode and item
    __shared__ float4 sg[CHUNK];                           // sigma^n
    __shared__ float vs[ITEMS][3][INLET_J];                // v' per item and node
    const int lane = threadIdx.x, w = threadIdx.y;
    const int tid = w * INLET_J + lane;
    const int ny = a.ny, nz = a.nz, N = a.N, T = a.planes;
    const int j0 = blockIdx.y * INLET_J;
    const int k0 = blockIdx.x * kb;   // the block's span nodes k0 .. k0 + kb - 1; item q = (k0 + q / T, step q % T)
    const int items = kb * T;         // <= ITEMS
    const float af = a.a_filter, bf = 1.0f - a.a_filter;
    const size_t plane = (size_t)ny * nz;
    float v[2][IPW][3];  // modes of even and odd index
#pragma unroll
    for (int q = 0; q < 2 * IPW; ++q) v[q & 1][q >> 1][0] = v[q & 1][q >> 1][1] = v[q & 1][q >> 1][2] = 0.f;
    // The table reads of a chunk are issued together, a chunk ahead of their use:
    // their latency is most of what a chunk costs a launch of few blocks.
    constexpr int NB = CHUNK * ITEMS / NT, NY = CHUNK * INLET_J / NT;
    float b[NB];
    float2 y[NY];
    unsigned long long ph[NB], om[NB];
    float4 sgr;
    auto fetch = [&](int n0) {
        const int cn = min(CHUNK, N - n0);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int e = tid + i * NT, m = e / ITEMS, q = e % ITEMS;
            if (m >= cn || q >= items) continue;
            ph[i] = a.phq[n0 + m], om[i] = a.omq[n0 + m];
            b[i] = a.BS[(size_t)(n0 + m) * nz + min(k0 + q / T, nz - 1)];  // nodes past nz are not stored
        }
#pragma unroll
        for (int i = 0; i < NY; ++i) {
            const int m = w + i * INLET_WARPS;
            if (m < cn) y[i] = a.AS[(size_t)(n0 + m) * ny + min(j0 + lane, ny - 1)];  // nor are rows past ny
        }
        if (tid < cn) sgr = make_float4(a.sig[3 * (n0 + tid)], a.sig[3 * (n0 + tid) + 1], a.sig[3 * (n0 + tid) + 2], 0.f);
    };
    // the filter state and tables of the thread's first node, early as well
    float L[6], ui = 0.f, f[3];
    auto fetch_node = [&](int e) {
        const int j = j0 + e % INLET_J, k = k0 + e / INLET_J;
        if (e >= kb * INLET_J || j >= ny || k >= nz) return false;
#pragma unroll
        for (int c = 0; c < 6; ++c) L[c] = a.a6[6 * j + c];
        ui = a.u_int[j];
#pragma unroll
        for (int c = 0; c < 3; ++c) f[c] = a.uf[c * plane + (size_t)k * ny + j];
        return true;
    };
    fetch(0);
    // step of the first plane: a later launch of a block of steps, beside which the
    // step counter moves on, counts from the block's first one
    const long long t = (a.from_block ? a.ctl->t_block : a.ctl->t[a.parity]) + a.ahead;
    if (!a.from_block && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) a.ctl->t_block = t - a.ahead;
    const long long t0f = a.ctl->t0_filter;
    bool mine = fetch_node(tid);
    for (int n0 = 0; n0 < N; n0 += CHUNK) {
        const int cn = min(CHUNK, N - n0);
        __syncthreads();  // the previous chunk is consumed
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int e = tid + i * NT, m = e / ITEMS, q = e % ITEMS;
            if (m >= cn || q >= items) continue;
            // time part of the phase: phi^n + omega^n t modulo one turn
            const unsigned long long p = ph[i] + om[i] * (unsigned long long)(t + q % T);
            is[m][q] = make_float2((float)(unsigned)(p >> 32) * 1.4629180792671596e-09f, b[i]);  // 2 pi / 2^32
        }
#pragma unroll
        for (int i = 0; i < NY; ++i) {
            const int m = w + i * INLET_WARPS;
            if (m < cn) ys[m][lane] = y[i];
        }
        if (tid < cn) sg[tid] = sgr;
        __syncthreads();
        if (n0 + CHUNK < N) fetch(n0 + CHUNK);
        // (a chunk's length is even: the parity of m is the mode's)
        auto term = [&](int m, float (&vp)[IPW][3]) {
            const float2 ya = ys[m][lane];
            const float4 s = sg[m];
#pragma unroll
            for (int q = 0; q < IPW; ++q) {
                const float2 tb = is[m][w * IPW + q];
                float arg = ya.x + tb.x;                       // in [0, 4 pi)
                arg = arg + tb.y;                              // in [0, 6 pi)
                arg -= 6.2831853f * rintf(arg * 0.15915494f);  // to [-pi, pi]
                const float amp = ya.y * __cosf(arg);
                vp[q][0] = fmaf(amp, s.x, vp[q][0]);
                vp[q][1] = fmaf(amp, s.y, vp[q][1]);
                vp[q][2] = fmaf(amp, s.z, vp[q][2]);
            }
        };
        int m = 0;
#pragma unroll 2
        for (; m + 1 < cn; m += 2) {
            term(m, v[0]);
            term(m + 1, v[1]);
        }
        if (m < cn) term(m, v[0]);
    }
#pragma unroll
    for (int q = 0; q < IPW; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) vs[w * IPW + q][c][lane] = v[0][q][c] + v[1][q][c];
    __syncthreads();
    for (int e = tid; e < kb * INLET_J; e += NT, mine = fetch_node(e)) {
        if (!mine) continue;
        const int jj = e % INLET_J, kk = e / INLET_J;
        const size_t node = (size_t)(k0 + kk) * ny + j0 + jj;
        for (int s = 0; s < T; ++s) {
            const float *vq = &vs[kk * T + s][0][jj];
            const float v0 = vq[0], v1 = vq[INLET_J], v2 = vq[2 * INLET_J];
            const float u[3] = {__fmul_rn(L[0], v0), fmaf(L[1], v0, __fmul_rn(L[2], v1)),
                                fmaf(L[5], v2, fmaf(L[3], v0, __fmul_rn(L[4], v1)))};
            const bool first = (t + s == t0f);
            float *o = a.ubc + (size_t)((t + s) & (INLET_RING - 1)) * 3 * plane + node;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                f[c] = first ? u[c] : fmaf(bf, u[c], __fmul_rn(af, f[c]));
                o[c * plane] = c == 0 ? ui + f[c] : f[c];
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) a.uf[c * plane + node] = f[c];
    }
}

cudaError_t launch_inlet(const InletArgs &a, cudaStream_t s)
{
    if (a.planes < 1 || a.planes > INLET_MAX_PLANES) return cudaErrorInvalidValue;
    const int ipw = a.planes > INLET_WARPS ? 4 : 1;
    const int kb = ipw * INLET_WARPS / a.planes;
    // span nodes along x: nz may be longer than the 65535 blocks of the other axes (ny may not)
    const dim3 grid((a.nz + kb - 1) / kb, (a.ny + INLET_J - 1) / INLET_J);
    const dim3 block(INLET_J, INLET_WARPS);
    if (ipw == 4) stg_inlet_kernel<4><<<grid, block, 0, s>>>(a, kb);
    else stg_inlet_kernel<1><<<grid, block, 0, s>>>(a, kb);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP64 setup per inlet node j: Cholesky factor of the lattice-unit Reynolds
// stress (eq. cholesky; a negative radicand counts as zero, a zero pivot
// zeroes the column).  The mode amplitudes are built on the host.
__global__ void setup_nodes_kernel(int ny, const double *R6, float *a6)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= ny) return;
    const double *R = R6 + 6 * j;  // 11 22 33 12 13 23
    const double l11 = sqrt(fmax(R[0], 0.0));
    const double l21 = l11 > 0.0 ? R[3] / l11 : 0.0;
    const double l31 = l11 > 0.0 ? R[4] / l11 : 0.0;
    const double l22 = sqrt(fmax(R[1] - l21 * l21, 0.0));
    const double l32 = l22 > 0.0 ? (R[5] - l21 * l31) / l22 : 0.0;
    const double l33 = sqrt(fmax(R[2] - l31 * l31 - l32 * l32, 0.0));
    float *o = a6 + 6 * j;
    o[0] = (float)l11; o[1] = (float)l21; o[2] = (float)l22;
    o[3] = (float)l31; o[4] = (float)l32; o[5] = (float)l33;
}

cudaError_t launch_setup_nodes(int ny, const double *R6, float *a6, cudaStream_t s)
{
    setup_nodes_kernel<<<(ny + 127) / 128, 128, 0, s>>>(ny, R6, a6);
    return cudaGetLastError();
}

}  // namespace stg
