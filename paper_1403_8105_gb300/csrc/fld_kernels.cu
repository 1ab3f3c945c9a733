// fld_kernels.cu -- CUDA kernels of the GB300 FLD solver (sm_103a).
//
// Koerner et al., "Flux-Limited Diffusion for Multiple Scattering in
// Participating Media", CGF 33(2) 2014:
//   * medium preparation and initialisation (Algorithm 1, first steps);
//   * one colour pass of the red-black SOR relaxation (Algorithm 1) with the
//     Knudsen number (Eq. 35), D update (Eq. 33), face coefficients
//     D_ps = (D_p + D_s)/2, local update (Eq. 32) and SOR blend (Eq. 36);
//   * the residual of Eq. 37 with D recomputed from phi, reduced on the
//     device (warp shuffles, block tree, deterministic second pass);
//   * the single-scatter source q_ri = L sigma_s T (Sec. 3 after Eq. 6) by
//     a transmittance march (Eq. 3).
//
// The stencil is memory-bound: no tensor-core formulation applies.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "fld_cell.cuh"
#include "fld_device.cuh"
#include "fld_internal.h"

namespace fld {

namespace {

using namespace cell;

constexpr int kRedThreads = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sum of v over the block; valid in thread 0.  blockDim <= 1024.
__device__ __forceinline__ double block_sum(double v, double *sh) {
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int nthr = blockDim.x * blockDim.y * blockDim.z;
    v = warp_sum(v);
    __syncthreads();
    if ((tid & 31) == 0) sh[tid >> 5] = v;
    __syncthreads();
    double r = 0.0;
    if (tid < 32) {
        r = (tid < (nthr + 31) / 32) ? sh[tid] : 0.0;
        r = warp_sum(r);
    }
    return r;
}

// Second pass: fixed-order sum of the per-block partial pairs.
__global__ void __launch_bounds__(kRedThreads) k_finalize(const double *__restrict__ partials, int nblocks,
                                                         double *__restrict__ result) {
    __shared__ double sh[32];
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nblocks; i += blockDim.x) {
        a += partials[2 * i];
        b += partials[2 * i + 1];
    }
    a = block_sum(a, sh);
    __syncthreads();
    b = block_sum(b, sh);
    if (threadIdx.x == 0) {
        result[0] = a;
        result[1] = b;
    }
}

// ---------------------------------------------------------------------------
// Preparation
// ---------------------------------------------------------------------------
// sigma' = max(sigma_t, sigma_eps) and sigma_a' = (1 - albedo) sigma' in
// single precision; with BF both are rounded to bfloat16 (nearest, ties to
// even), the bit patterns kept for the sweeps that read bfloat16 and the
// rounded values, upcast exactly, stored in sp / ah2 for all other kernels.
template <bool BF>
__global__ void k_prep_f(Layout L, const float *__restrict__ st, const float *__restrict__ alb,
                         const float *__restrict__ js, float *__restrict__ sp, float *__restrict__ ah2,
                         float *__restrict__ jh2, uint16_t *__restrict__ spb, uint16_t *__restrict__ sab, float seps,
                         float h2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= L.nx || j >= L.ny) return;
    const long long v = ((long long)k * L.ny + j) * L.nx + i;
    const int q = L.at(i, j, k);
    float s = fmaxf(st[v], seps);                                 // Algorithm 1: sigma floor
    float a = __fmul_rn(__fsub_rn(1.0f, alb[v]), s);              // (1 - albedo) sigma'
    if (BF) {
        const uint16_t sb = __bfloat16_as_ushort(__float2bfloat16_rn(s));
        const uint16_t ab = __bfloat16_as_ushort(__float2bfloat16_rn(a));
        spb[q] = sb;
        sab[q] = ab;
        s = bf16_bits_to_f(sb);
        a = bf16_bits_to_f(ab);
    }
    sp[q] = s;
    ah2[q] = __fmul_rn(a, h2);                                    // sigma_a' dl^2
    jh2[q] = __fmul_rn(js[v], h2);
}

template <bool BF>
__global__ void k_prep_d(Layout L, const float *__restrict__ st, const float *__restrict__ alb,
                         const float *__restrict__ js, double *__restrict__ sp, double *__restrict__ ah2,
                         double *__restrict__ jh2, double seps, double h2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= L.nx || j >= L.ny) return;
    const long long v = ((long long)k * L.ny + j) * L.nx + i;
    const int q = L.at(i, j, k);
    double s, a;
    if (BF) {   // the rounded medium of k_prep_f<true>, exactly
        const float s32 = fmaxf(st[v], (float)seps);
        const float a32 = __fmul_rn(__fsub_rn(1.0f, alb[v]), s32);
        s = (double)bf16_bits_to_f(__bfloat16_as_ushort(__float2bfloat16_rn(s32)));
        a = (double)bf16_bits_to_f(__bfloat16_as_ushort(__float2bfloat16_rn(a32)));
    } else {
        s = fmax((double)st[v], seps);
        a = __dmul_rn(1.0 - (double)alb[v], s);
    }
    sp[q] = s;
    ah2[q] = __dmul_rn(a, h2);
    jh2[q] = __dmul_rn((double)js[v], h2);
}

// Every element of both colour arrays: unknowns get (phi0, D0), the ghost
// layer (phi_b, D_b), the alignment slack of each half row 0.  Four elements of
// a half row per thread, stored together (512^3: 552 -> 261 us).
template <typename T>
__device__ __forceinline__ void store4(T *p, const T v[4]) {
    if (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]);
    } else {
        reinterpret_cast<double2 *>(p)[0] = make_double2((double)v[0], (double)v[1]);
        reinterpret_cast<double2 *>(p)[1] = make_double2((double)v[2], (double)v[3]);
    }
}

template <typename T>
__global__ void k_init(Layout L, Divisor by_quads, Divisor by_py, T *__restrict__ phi, float *__restrict__ phlo,
                       T *__restrict__ D, T phi0, T D0, T phi_b, T D_b) {
    const uint32_t e4 = blockIdx.x * blockDim.x + threadIdx.x;      // quad of elements
    if (e4 >= (uint32_t)L.total >> 2) return;
    const uint32_t row = by_quads.quot(e4);                         // row of either colour
    const int rows = L.py * (L.nz + 2), c = (int)row >= rows ? 1 : 0;
    const uint32_t r = row - c * rows;
    const int K = (int)by_py.quot(r), J = (int)r - K * L.py;
    const int par = (J + K + 1 + c) & 1;                            // I & 1 of this row's cells
    T p[4], d[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int pos = 4 * (int)(e4 - row * ((uint32_t)L.hpx >> 2)) + u - kXoff;   // = (I + 1) >> 1 for a cell
        const int I = par ? 2 * pos - 1 : 2 * pos;
        p[u] = d[u] = T(0);
        if (pos >= 0 && I >= 0 && I <= L.nx + 1) {
            const bool ghost = I == 0 || J == 0 || K == 0 || I == L.nx + 1 || J == L.ny + 1 || K == L.nz + 1;
            p[u] = ghost ? phi_b : phi0;
            d[u] = ghost ? D_b : D0;
        }
    }
    store4(phi + 4 * (size_t)e4, p);
    store4(D + 4 * (size_t)e4, d);
    const float zero[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (phlo) store4(phlo + 4 * (size_t)e4, zero);
}

// Packed (nx+2)(ny+2)(nz+2) <-> device layout.  A thread moves four values a
// block's width apart, loads before stores, and finds their places by
// multiplication; blocks run over the whole array.  (One value per thread in
// 128-thread blocks of a row each, whose last one is nearly empty, packed a
// 512^3 field at 2.0 TB/s.)
constexpr int kMoveThreads = 256, kMovePer = 4;

struct PackedIndex {
    uint32_t row, rows, total;   // values per row, rows per plane, values in all
    Divisor by_row, by_rows;
};

template <typename Load, typename Store>
__device__ __forceinline__ void move_packed(const Layout &L, const PackedIndex &ix, Load &&load, Store &&store) {
    const uint32_t e0 = blockIdx.x * (uint32_t)(kMoveThreads * kMovePer) + threadIdx.x;
    int q[kMovePer];
    double v[kMovePer];
#pragma unroll
    for (int k = 0; k < kMovePer; ++k) {
        const uint32_t e = e0 + k * kMoveThreads;
        const uint32_t r = ix.by_row.quot(e < ix.total ? e : 0), K = ix.by_rows.quot(r);
        q[k] = L.at((int)((e < ix.total ? e : 0) - r * ix.row) - 1, (int)(r - K * ix.rows) - 1, (int)K - 1);
        v[k] = load(e < ix.total ? e : 0, q[k]);
    }
#pragma unroll
    for (int k = 0; k < kMovePer; ++k)
        if (e0 + k * kMoveThreads < ix.total) store(e0 + k * kMoveThreads, q[k], v[k]);
}

// into the single-precision fields (lo may be null) and the FP64 one at once
__global__ void __launch_bounds__(kMoveThreads) k_unpack(Layout L, PackedIndex ix, const double *__restrict__ src,
                                                         float *__restrict__ hi, float *__restrict__ lo,
                                                         double *__restrict__ dst) {
    move_packed(L, ix, [&](uint32_t e, int) { return src[e]; },
                [&](uint32_t, int q, double x) {
                    const float h = (float)x;
                    hi[q] = h;
                    if (lo) lo[q] = (float)(x - (double)h);
                    dst[q] = x;
                });
}

__global__ void __launch_bounds__(kMoveThreads) k_pack_from_f(Layout L, PackedIndex ix, const float *__restrict__ hi,
                                                              const float *__restrict__ lo,
                                                              double *__restrict__ dst) {
    move_packed(L, ix, [&](uint32_t, int q) { return (double)hi[q] + (lo ? (double)lo[q] : 0.0); },
                [&](uint32_t e, int, double x) { dst[e] = x; });
}

__global__ void __launch_bounds__(kMoveThreads) k_pack_from_d(Layout L, PackedIndex ix,
                                                              const double *__restrict__ src,
                                                              double *__restrict__ dst) {
    move_packed(L, ix, [&](uint32_t, int q) { return src[q]; }, [&](uint32_t e, int, double x) { dst[e] = x; });
}

__global__ void k_f_to_d(long long n, const float *__restrict__ hi, const float *__restrict__ lo,
                         double *__restrict__ dst) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) dst[e] = (double)hi[e] + (lo ? (double)lo[e] : 0.0);
}

__global__ void k_d_to_f(long long n, const double *__restrict__ src, float *__restrict__ hi,
                         float *__restrict__ lo) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const double x = src[e];
    const float h = (float)x;
    hi[e] = h;
    if (lo) lo[e] = (float)(x - (double)h);
}

// ---------------------------------------------------------------------------
// Red-black pass.
//
// Thread (t, J, K) of colour c updates the t-th unknown of colour c in row
// (J, K) (padded I = 2t + 2 - ((J + K + 1 + c) & 1)) if the row has one.  All six neighbours have the other colour, so a pass is
// free of races and its result does not depend on thread order.  Within a
// warp every access is a run of consecutive elements of one colour array.
//
// Update in residual form: with d_s = phi_s - phi_p and D_ps = (D_p + D_s)/2,
//   S(D_p)   = j dl^2 - sigma_a' dl^2 phi_p + sum_s D_ps d_s
//            = jh2 - ah2 phi_p + (D_p/2) sum_s d_s + (1/2) sum_s D_s d_s
//   den(D_p) = ah2 + sum_s D_ps = ah2 + 3 D_p + (1/2) sum_s D_s
// and Eq. 32 reads phi' = phi_p + S/den (num/den of the paper with num - phi_p
// den = S).  Each local round recomputes D_p (Eq. 35, 33) at the current
// point value phi_p + delta and sets delta = S(D_p)/den(D_p); the SOR blend
// (Eq. 36) is phi_p + omega * delta.  One round is Algorithm 1 as printed.
// ---------------------------------------------------------------------------

struct Nbrs {
    int own, nb[6];
};

// Offsets of the t-th unknown of colour c in row (J, K) and of its
// neighbours (x-, x+, y-, y+, z-, z+); false if the row has fewer unknowns
// of that colour.  The row's unknowns of colour c are I = 2t + 2 - par,
// par = (J + K + 1 + c) & 1, i.e. every other I starting at 1 or 2.
__device__ __forceinline__ bool pass_cell(const Layout &L, int c, int t, int J, int K, Nbrs &o) {
    const int par = (J + K + 1 + c) & 1;
    const int I = 2 * t + 2 - par;
    if (I > L.nx) return false;
    const int row = L.row(J, K);
    const int ob = (1 - c) * L.cs;
    const int h = I >> 1;
    const int pos = (I + 1) >> 1;
    o.own = c * L.cs + row + pos;
    o.nb[0] = ob + row + h;
    o.nb[1] = ob + row + h + 1;
    o.nb[2] = ob + row - L.hpx + pos;
    o.nb[3] = ob + row + L.hpx + pos;
    o.nb[4] = ob + row - L.hpx * L.py + pos;
    o.nb[5] = ob + row + L.hpx * L.py + pos;
    return true;
}

// How the threads of a launched pass take the items (pairs, or single unknowns
// for the float-float pass) of its rows: 32 x 4 tiles of a plane, or, running,
// item e of all rows by thread e, so that rows shorter or a little longer than
// a multiple of 32 items leave no lanes idle.
struct PassIndex {
    uint32_t per_row, total;     // items per row, items of all ny x nz rows
    Divisor by_items, by_rows;
};
constexpr int kPassThreads = 128;
constexpr long long kSmallCtas = 760;      // all resident at five per SM

template <bool RUN>
__device__ __forceinline__ bool pass_item(const Layout &L, const PassIndex &ix, int &t, int &J, int &K) {
    if (RUN) {
        const uint32_t e = blockIdx.x * (uint32_t)kPassThreads + threadIdx.x;
        if (e >= ix.total) return false;
        const uint32_t row = ix.by_items.quot(e);
        t = (int)(e - row * ix.per_row);
        K = (int)ix.by_rows.quot(row);
        J = (int)row - K * L.ny + 1;
        ++K;
    } else {
        t = blockIdx.x * 32 + (threadIdx.x & 31);
        J = blockIdx.y * (kPassThreads / 32) + (threadIdx.x >> 5) + 1;
        K = blockIdx.z + 1;
        if (J > L.ny) return false;
    }
    return true;
}

// Two adjacent unknowns t, t+1 (t even) of one colour in row (J, K) per
// thread: in the colour-split layout they are one aligned float2 of every
// field, their x-neighbours three consecutive elements of the other colour's
// row and their y/z-neighbours a float2 one row/plane away.
struct Pair {
    int own, xv, ym, yp, zm, zp;              // offsets of the float2s (own colour at own, the other at the rest)
    bool first, second;                       // which of the two cells are unknowns
    bool left;                                // x-neighbours at xv-1, xv, xv+1 (else xv, xv+1, xv+2)
};

__device__ __forceinline__ void pair_cells(const Layout &L, int c, int t, int J, int K, Pair &q) {
    const int par = (J + K + 1 + c) & 1;
    const int I0 = 2 * t + 2 - par;                 // padded I of cell t
    q.first = I0 <= L.nx;
    q.second = I0 + 2 <= L.nx;
    const int row = (K * L.py + J) * L.hpx + kXoff + 1;   // element of the row's first unknown
    const int ob = (1 - c) * L.cs;
    q.own = c * L.cs + row + t;
    q.left = par == 1;                              // x-neighbours of cell t: (I0 - 1) and (I0 + 1)
    q.xv = ob + row + t;
    q.ym = ob + row - L.hpx + t;
    q.yp = ob + row + L.hpx + t;
    q.zm = ob + row - L.hpx * L.py + t;
    q.zp = ob + row + L.hpx * L.py + t;
}

__device__ __forceinline__ float2 ld2(const float *__restrict__ p, int off) {
    return *reinterpret_cast<const float2 *>(p + off);
}


// Gather the six neighbours of the two cells of a pair from one field.
__device__ __forceinline__ void gather_pair(const float *f, const Pair &q, float v0[6], float v1[6]) {
    const float2 xv = ld2(f, q.xv);
    const float xe = q.left ? f[q.xv - 1] : f[q.xv + 2];
    if (q.left) {
        v0[0] = xe; v0[1] = xv.x; v1[0] = xv.x; v1[1] = xv.y;
    } else {
        v0[0] = xv.x; v0[1] = xv.y; v1[0] = xv.y; v1[1] = xe;
    }
    const float2 ym = ld2(f, q.ym), yp = ld2(f, q.yp), zm = ld2(f, q.zm), zp = ld2(f, q.zp);
    v0[2] = ym.x; v0[3] = yp.x; v0[4] = zm.x; v0[5] = zp.x;
    v1[2] = ym.y; v1[3] = yp.y; v1[4] = zm.y; v1[5] = zp.y;
}

// sigma' and sigma_a' h^2 of the two cells of a pair: the single-precision
// fields, or the bfloat16 copies (one 32-bit load each; the first cell is the
// low half) with sigma_a' scaled by h^2 as k_prep_f scales it.
template <bool BF>
__device__ __forceinline__ void medium_pair(const float *__restrict__ sp, const float *__restrict__ ah2,
                                            const uint16_t *__restrict__ spb, const uint16_t *__restrict__ sab,
                                            float h2, int off, float2 &s2, float2 &a2) {
    if (BF) {
        const uint32_t us = *reinterpret_cast<const uint32_t *>(spb + off);
        const uint32_t ua = *reinterpret_cast<const uint32_t *>(sab + off);
        s2 = make_float2(__uint_as_float(us << 16), __uint_as_float(us & 0xFFFF0000u));
        a2 = make_float2(__fmul_rn(__uint_as_float(ua << 16), h2), __fmul_rn(__uint_as_float(ua & 0xFFFF0000u), h2));
    } else {
        s2 = ld2(sp, off);
        a2 = ld2(ah2, off);
    }
}

// Single-precision pass (the bulk sweeps), two unknowns per thread: the pair
// (t, t+1) of row (J, K); waits for the preceding grid (pdl_wait) before
// reading phi / D.
template <int LIM, int ROUNDS, bool BF>
__device__ __forceinline__ void tile_f32(const Layout &L, const float *__restrict__ sp,
                                         const float *__restrict__ ah2, const float *__restrict__ jh2,
                                         const uint16_t *__restrict__ spb, const uint16_t *__restrict__ sab, float h2,
                                         float *phi, float *D, int colour, int lim_rt, float larsen_n, float omega,
                                         float inv2h, float floor_, int rounds_rt, int t, int J, int K) {
    if (J > L.ny) return;
    Pair q;
    pair_cells(L, colour, t, J, K, q);
    if (!q.first) return;
    float2 s2, a2;
    medium_pair<BF>(sp, ah2, spb, sab, h2, q.own, s2, a2);
    const float2 j2 = ld2(jh2, q.own);
    pdl_wait();
    float ps0[6], ps1[6], Ds0[6], Ds1[6];
    gather_pair(phi, q, ps0, ps1);
    gather_pair(D, q, Ds0, Ds1);
    const float2 p0 = ld2(phi, q.own);
    float pn0, dn0, pn1, dn1;
    cell_f32<LIM, ROUNDS>(p0.x, ps0, Ds0, s2.x, a2.x, j2.x, lim_rt, larsen_n, omega, inv2h, floor_, rounds_rt, pn0,
                          dn0);
    if (q.second) {
        cell_f32<LIM, ROUNDS>(p0.y, ps1, Ds1, s2.y, a2.y, j2.y, lim_rt, larsen_n, omega, inv2h, floor_, rounds_rt,
                              pn1, dn1);
        *reinterpret_cast<float2 *>(phi + q.own) = make_float2(pn0, pn1);
        *reinterpret_cast<float2 *>(D + q.own) = make_float2(dn0, dn1);
    } else {
        phi[q.own] = pn0;          // the element after the last unknown is a ghost: left untouched
        D[q.own] = dn0;
    }
}

// The launched FP32 pass.  Its threads wait on memory (a CDA limiter with one
// round, a third of the arithmetic, takes 101 of 113 us per iteration at
// 256^3), so registers are left to hold all of a thread's loads in flight (48),
// and 128-thread CTAs, which a finished warp keeps waiting less, hold ten of
// them per SM: 13.7 -> 13.4 us per iteration at 128^3, 113.9 -> 108.9 at 256^3
// against 256 threads.
template <int LIM, int ROUNDS, bool BF, bool RUN>
__global__ void __launch_bounds__(kPassThreads, 10) k_pass2_f32(Layout L, PassIndex ix, const float *__restrict__ sp,
                                                   const float *__restrict__ ah2, const float *__restrict__ jh2,
                                                   const uint16_t *__restrict__ spb,
                                                   const uint16_t *__restrict__ sab, float h2,
                                                   float *__restrict__ phi, float *__restrict__ D, int colour,
                                                   int lim_rt, float larsen_n, float omega, float inv2h,
                                                   float floor_, int rounds_rt) {
    pdl_launch_dependents();
    int t, J, K;
    if (!pass_item<RUN>(L, ix, t, J, K)) return;
    tile_f32<LIM, ROUNDS, BF>(L, sp, ah2, jh2, spb, sab, h2, phi, D, colour, lim_rt, larsen_n, omega, inv2h, floor_,
                              rounds_rt, 2 * t, J, K);
}

// Middle pass (phi as a hi/lo pair, FP32-summed update, cell::cell_fh):
// tile_fh is the arithmetic of a pair of unknowns; k_pass2_fh launches it.
template <int LIM, int ROUNDS, bool BF>
__device__ __forceinline__ void tile_fh(const Layout &L, const float *__restrict__ sp,
                                        const float *__restrict__ ah2, const float *__restrict__ jh2,
                                        const uint16_t *__restrict__ spb, const uint16_t *__restrict__ sab, float h2,
                                        float *phi, float *phlo, float *D, int colour, int lim_rt, float larsen_n,
                                        float omega, float inv2h, float floor_, int rounds_rt, int t, int J, int K) {
    if (J > L.ny) return;
    Pair q;
    pair_cells(L, colour, t, J, K, q);
    if (!q.first) return;
    float2 s2, a2;
    medium_pair<BF>(sp, ah2, spb, sab, h2, q.own, s2, a2);
    const float2 j2 = ld2(jh2, q.own);
    pdl_wait();
    float ps0[6], ps1[6], ls0[6], ls1[6], Ds0[6], Ds1[6];
    gather_pair(phi, q, ps0, ps1);
    gather_pair(phlo, q, ls0, ls1);
    gather_pair(D, q, Ds0, Ds1);
    const float2 p0 = ld2(phi, q.own), l0 = ld2(phlo, q.own);
    float h0, lo0, d0, h1, lo1, d1;
    cell_fh<LIM, ROUNDS, true>(p0.x, l0.x, ps0, ls0, Ds0, s2.x, a2.x, j2.x, lim_rt, larsen_n, omega, inv2h, floor_,
                         rounds_rt, h0, lo0, d0);
    if (q.second) {
        cell_fh<LIM, ROUNDS, true>(p0.y, l0.y, ps1, ls1, Ds1, s2.y, a2.y, j2.y, lim_rt, larsen_n, omega, inv2h, floor_,
                             rounds_rt, h1, lo1, d1);
        *reinterpret_cast<float2 *>(phi + q.own) = make_float2(h0, h1);
        *reinterpret_cast<float2 *>(phlo + q.own) = make_float2(lo0, lo1);
        *reinterpret_cast<float2 *>(D + q.own) = make_float2(d0, d1);
    } else {
        phi[q.own] = h0;
        phlo[q.own] = lo0;
        D[q.own] = d0;
    }
}

// The launched hi/lo pass (64 registers, eight CTAs per SM, no spills; with 48
// registers it spilled and ran 25 % slower at 256^3).
template <int LIM, int ROUNDS, bool BF, bool RUN>
__global__ void __launch_bounds__(kPassThreads, 8) k_pass2_fh(Layout L, PassIndex ix, const float *__restrict__ sp,
                                                  const float *__restrict__ ah2, const float *__restrict__ jh2,
                                                  const uint16_t *__restrict__ spb,
                                                  const uint16_t *__restrict__ sab, float h2,
                                                  float *__restrict__ phi, float *__restrict__ phlo,
                                                  float *__restrict__ D, int colour, int lim_rt, float larsen_n,
                                                  float omega, float inv2h, float floor_, int rounds_rt) {
    pdl_launch_dependents();
    int t, J, K;
    if (!pass_item<RUN>(L, ix, t, J, K)) return;
    tile_fh<LIM, ROUNDS, BF>(L, sp, ah2, jh2, spb, sab, h2, phi, phlo, D, colour, lim_rt, larsen_n, omega, inv2h,
                             floor_, rounds_rt, 2 * t, J, K);
}

// One unknown per thread, FP32 or hi/lo, the limiter without branches: on grids too
// small to fill the GPU a pass takes as long as one thread's chain of dependent
// operations, which the pair pass goes through twice (us per iteration, pairs and
// this, timed by the tuner: 32^3 FP32 4.1 / 2.8, 50^3 4.5 / 3.5, hi/lo 5.4 / 4.8; 80^3 6.9 / 6.1).
template <int LIM, int ROUNDS, bool HL>
__global__ void __launch_bounds__(kPassThreads) k_pass1(Layout L, PassIndex ix, const float *__restrict__ sp,
                                                        const float *__restrict__ ah2,
                                                        const float *__restrict__ jh2, float *__restrict__ phi,
                                                        float *__restrict__ phlo, float *__restrict__ D, int colour,
                                                        int lim_rt, float larsen_n, float omega, float inv2h,
                                                        float floor_, int rounds_rt) {
    pdl_launch_dependents();
    int t, J, K;
    Nbrs o;
    if (!pass_item<true>(L, ix, t, J, K) || !pass_cell(L, colour, t, J, K, o)) return;
    const float s_ = sp[o.own], ah = ah2[o.own], jj = jh2[o.own];
    pdl_wait();
    const float p0 = phi[o.own], p0lo = HL ? phlo[o.own] : 0.0f;
    float ps[6], ls[6], Ds[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        ps[s] = phi[o.nb[s]];
        if (HL) ls[s] = phlo[o.nb[s]];
        Ds[s] = D[o.nb[s]];
    }
    float hi, lo, Dp;
    if (HL) {
        cell_fh<LIM, ROUNDS, true>(p0, p0lo, ps, ls, Ds, s_, ah, jj, lim_rt, larsen_n, omega, inv2h, floor_,
                                   rounds_rt, hi, lo, Dp);
        phlo[o.own] = lo;
    } else {
        cell_f32<LIM, ROUNDS, true>(p0, ps, Ds, s_, ah, jj, lim_rt, larsen_n, omega, inv2h, floor_, rounds_rt, hi, Dp);
    }
    phi[o.own] = hi;
    D[o.own] = Dp;
}

// Four adjacent unknowns t .. t+3 (t a multiple of 4) of one colour in row
// (J, K) per thread: one aligned 128-bit load per own field and per y/z
// neighbour row/plane, the x-neighbours five consecutive elements of the other
// colour's row (a 128-bit load and one scalar).  Same per-cell arithmetic as
// the pair passes (cell::cell_f32 / cell::cell_fh), so the results agree bit
// for bit; more independent cells per thread, fewer loads and address
// computations per cell.
struct Quad {
    int own, xv, ym, yp, zm, zp;              // offsets of the float4s (own colour at own, the other at the rest)
    int n;                                    // unknowns among the four (1 .. 4)
    bool left;                                // x-neighbours at xv-1 .. xv+3 (else xv .. xv+4)
};

__device__ __forceinline__ bool quad_cells(const Layout &L, int c, int t, int J, int K, Quad &q) {
    const int par = (J + K + 1 + c) & 1;
    const int I0 = 2 * t + 2 - par;                 // padded I of cell t
    if (I0 > L.nx) return false;
    q.n = min(4, (L.nx - I0) / 2 + 1);
    const int row = (K * L.py + J) * L.hpx + kXoff + 1;   // element of the row's first unknown
    const int ob = (1 - c) * L.cs;
    q.own = c * L.cs + row + t;
    q.left = par == 1;
    q.xv = ob + row + t;
    q.ym = ob + row - L.hpx + t;
    q.yp = ob + row + L.hpx + t;
    q.zm = ob + row - L.hpx * L.py + t;
    q.zp = ob + row + L.hpx * L.py + t;
    return true;
}

__device__ __forceinline__ float4 ld4(const float *__restrict__ p, int off) {
    return *reinterpret_cast<const float4 *>(p + off);
}

__device__ __forceinline__ float f4_at(const float4 &v, int m) {
    return m == 0 ? v.x : m == 1 ? v.y : m == 2 ? v.z : v.w;
}

// The six neighbours of the four cells of a quad from one field: v[m][s].
__device__ __forceinline__ void gather_quad(const float *f, const Quad &q, float v[4][6]) {
    const float4 xv = ld4(f, q.xv);
    const float xe = q.left ? f[q.xv - 1] : f[q.xv + 4];
    const float x5[5] = {q.left ? xe : xv.x, q.left ? xv.x : xv.y, q.left ? xv.y : xv.z, q.left ? xv.z : xv.w,
                         q.left ? xv.w : xe};
    const float4 ym = ld4(f, q.ym), yp = ld4(f, q.yp), zm = ld4(f, q.zm), zp = ld4(f, q.zp);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        v[m][0] = x5[m];
        v[m][1] = x5[m + 1];
        v[m][2] = f4_at(ym, m);
        v[m][3] = f4_at(yp, m);
        v[m][4] = f4_at(zm, m);
        v[m][5] = f4_at(zp, m);
    }
}

template <bool BF>
__device__ __forceinline__ void medium_quad(const float *__restrict__ sp, const float *__restrict__ ah2,
                                            const uint16_t *__restrict__ spb, const uint16_t *__restrict__ sab,
                                            float h2, int off, float s4[4], float a4[4]) {
    if (BF) {
        const uint2 us = *reinterpret_cast<const uint2 *>(spb + off);
        const uint2 ua = *reinterpret_cast<const uint2 *>(sab + off);
        const uint32_t w[4] = {us.x << 16, us.x & 0xFFFF0000u, us.y << 16, us.y & 0xFFFF0000u};
        const uint32_t z[4] = {ua.x << 16, ua.x & 0xFFFF0000u, ua.y << 16, ua.y & 0xFFFF0000u};
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            s4[m] = __uint_as_float(w[m]);
            a4[m] = __fmul_rn(__uint_as_float(z[m]), h2);
        }
    } else {
        const float4 s = ld4(sp, off), a = ld4(ah2, off);
        s4[0] = s.x; s4[1] = s.y; s4[2] = s.z; s4[3] = s.w;
        a4[0] = a.x; a4[1] = a.y; a4[2] = a.z; a4[3] = a.w;
    }
}

__device__ __forceinline__ void store_quad(float *p, const Quad &q, const float v[4]) {
    if (q.n == 4) {
        *reinterpret_cast<float4 *>(p + q.own) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
        // the element after the last unknown is a ghost: left untouched
        for (int m = 0; m < q.n; ++m) p[q.own + m] = v[m];
    }
}

// Four unknowns per thread, single precision (k_pass4_f32) or hi/lo (HL,
// k_pass4_fh).
template <int LIM, int ROUNDS, bool BF, bool HL>
__device__ __forceinline__ void tile4(const Layout &L, const float *__restrict__ sp, const float *__restrict__ ah2,
                                      const float *__restrict__ jh2, const uint16_t *__restrict__ spb,
                                      const uint16_t *__restrict__ sab, float h2, float *phi, float *phlo, float *D,
                                      int colour, int lim_rt, float larsen_n, float omega, float inv2h, float floor_,
                                      int rounds_rt, int t, int J, int K) {
    if (J > L.ny) return;
    Quad q;
    if (!quad_cells(L, colour, t, J, K, q)) return;
    float s4[4], a4[4];
    medium_quad<BF>(sp, ah2, spb, sab, h2, q.own, s4, a4);
    const float4 j4 = ld4(jh2, q.own);
    const float jj[4] = {j4.x, j4.y, j4.z, j4.w};
    pdl_wait();
    float ps[4][6], Ds[4][6];
    gather_quad(phi, q, ps);
    gather_quad(D, q, Ds);
    const float4 p4 = ld4(phi, q.own);
    const float p0[4] = {p4.x, p4.y, p4.z, p4.w};
    float pn[4], dn[4], ln[4];
    if (HL) {
        float ls[4][6];
        gather_quad(phlo, q, ls);
        const float4 l4 = ld4(phlo, q.own);
        const float l0[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
        for (int m = 0; m < 4; ++m)
            cell_fh<LIM, ROUNDS>(p0[m], l0[m], ps[m], ls[m], Ds[m], s4[m], a4[m], jj[m], lim_rt, larsen_n, omega,
                                 inv2h, floor_, rounds_rt, pn[m], ln[m], dn[m]);
    } else {
#pragma unroll
        for (int m = 0; m < 4; ++m)
            cell_f32<LIM, ROUNDS>(p0[m], ps[m], Ds[m], s4[m], a4[m], jj[m], lim_rt, larsen_n, omega, inv2h, floor_,
                                  rounds_rt, pn[m], dn[m]);
    }
    store_quad(phi, q, pn);
    store_quad(D, q, dn);
    if (HL) store_quad(phlo, q, ln);
}

template <int LIM, int ROUNDS, bool BF, bool HL>
__global__ void __launch_bounds__(128) k_pass4(Layout L, const float *__restrict__ sp, const float *__restrict__ ah2,
                                               const float *__restrict__ jh2, const uint16_t *__restrict__ spb,
                                               const uint16_t *__restrict__ sab, float h2, float *__restrict__ phi,
                                               float *__restrict__ phlo, float *__restrict__ D, int colour,
                                               int lim_rt, float larsen_n, float omega, float inv2h, float floor_,
                                               int rounds_rt) {
    pdl_launch_dependents();
    tile4<LIM, ROUNDS, BF, HL>(L, sp, ah2, jh2, spb, sab, h2, phi, phlo, D, colour, lim_rt, larsen_n, omega, inv2h,
                               floor_, rounds_rt, 4 * (blockIdx.x * blockDim.x + threadIdx.x),
                               blockIdx.y * blockDim.y + threadIdx.y + 1, blockIdx.z + 1);
}

// Multi-grid colour pass: one launch updates one colour of every grid in a
// table of SweepDescs.  The CTAs are persistent (all resident) and walk the
// work items of all grids with a grid-wide stride; item i belongs to the last
// grid whose first item is <= i (binary search over the firsts, staged in
// shared memory).  An item is 32 x 8 pairs of unknowns of a z-plane, which
// go through tile_f32 / tile_fh with the grid's own parameters, so
// every grid gets the bits of its solo passes.  The table and both counts
// are read on the device: one captured graph of these launches serves any
// set of grids.
__device__ __forceinline__ SweepDesc load_sweep_desc(const SweepDesc *__restrict__ p) {
    SweepDesc d;
    const int4 *src = reinterpret_cast<const int4 *>(p);
    int4 *dst = reinterpret_cast<int4 *>(&d);
#pragma unroll
    for (int i = 0; i < (int)(sizeof(SweepDesc) / 16); ++i) dst[i] = __ldg(src + i);
    return d;
}

constexpr int kMultiThreadsX = 32, kMultiThreadsY = 8;

// One instantiation per limiter fast path, medium and family (a table holds
// grids of one family; limiter and medium are the batch's own).
template <int LIM, int ROUNDS, bool BF, bool HL>
__global__ void __launch_bounds__(kMultiThreadsX * kMultiThreadsY, 4)
    k_pass2_multi(const SweepDesc *__restrict__ descs, const int *__restrict__ counts, int colour) {
    __shared__ int first[kMultiMaxGrids];
    pdl_launch_dependents();
    const int ng = min(__ldg(counts), kMultiMaxGrids), total = __ldg(counts + 1);
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    for (int g = tid; g < ng; g += blockDim.x * blockDim.y) first[g] = __ldg(&descs[g].first);
    __syncthreads();
    for (int item = blockIdx.x; item < total; item += gridDim.x) {
        int lo = 0, hi = ng - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (first[mid] <= item) lo = mid;
            else hi = mid - 1;
        }
        const SweepDesc d = load_sweep_desc(descs + lo);
        const int local = item - d.first;
        const int bx = local % d.bx, rest = local / d.bx;
        const int by = rest % d.by, bz = rest / d.by;
        if (bz >= d.L.nz) continue;
        const int t = 2 * (bx * kMultiThreadsX + threadIdx.x);
        const int J = by * kMultiThreadsY + threadIdx.y + 1;
        if (HL)
            tile_fh<LIM, ROUNDS, BF>(d.L, d.sp, d.ah2, d.jh2, d.spb, d.sab, d.h2, d.phi, d.phlo, d.D, colour, d.lim,
                                     d.larsen_n, d.omega, d.inv2h, d.floor_, d.local_iters, t, J, bz + 1);
        else
            tile_f32<LIM, ROUNDS, BF>(d.L, d.sp, d.ah2, d.jh2, d.spb, d.sab, d.h2, d.phi, d.D, colour, d.lim,
                                      d.larsen_n, d.omega, d.inv2h, d.floor_, d.local_iters, t, J, bz + 1);
    }
    // a table of one-voxel grids has passes without unknowns: one CTA waits all the
    // same, so that the pass does not end before the preceding one
    if (blockIdx.x == 0) pdl_wait();
}

template <bool BF, bool HL>
auto multi_kernel(int lim, int local_iters) {
    if (local_iters == 2 && lim == LIM_LP) return k_pass2_multi<LIM_LP, 2, BF, HL>;
    return k_pass2_multi<-1, 0, BF, HL>;
}

// Float-float correction pass (cell::cell_ff), two unknowns per thread in
// packed arithmetic (cell::cell_ff_pair).
__device__ __forceinline__ void gather_packed(const float *f, const Pair &q, float2 v[6]) {
    const float2 xv = ld2(f, q.xv);
    const float xe = q.left ? f[q.xv - 1] : f[q.xv + 2];
    v[0] = q.left ? make_float2(xe, xv.x) : xv;
    v[1] = q.left ? xv : make_float2(xv.y, xe);
    v[2] = ld2(f, q.ym);
    v[3] = ld2(f, q.yp);
    v[4] = ld2(f, q.zm);
    v[5] = ld2(f, q.zp);
}

// Registers: with seven CTAs per SM (70 registers) the passes of grids that fill
// the GPU are fastest (us per iteration at 256^3 with 4, 6, 7, 8 CTAs: 295, 267,
// 241, 244; one unknown per thread 268, before quotient_rn 287; at 128^3 31.3,
// 35.0 and 36.6); left alone (90) those of small ones, whose CTAs are all
// resident at once and only wait longer for loads taken in turns (40^3: 6.5 against 11.1).
template <int LIM, int ROUNDS, bool RUN, int MINB>
__global__ void __launch_bounds__(kPassThreads, MINB) k_pass2_ff(Layout L, PassIndex ix, const float *__restrict__ sp,
                                                  const float *__restrict__ ah2, const float *__restrict__ jh2,
                                                  float *__restrict__ phi, float *__restrict__ phlo,
                                                  float *__restrict__ D, int colour, int lim_rt, float larsen_n,
                                                  float omega, float inv2h, float floor_, int rounds_rt) {
    pdl_launch_dependents();
    int t, J, K;
    if (!pass_item<RUN>(L, ix, t, J, K)) return;
    Pair q;
    pair_cells(L, colour, 2 * t, J, K, q);
    if (!q.first) return;
    const float2 s2 = ld2(sp, q.own), a2 = ld2(ah2, q.own), j2 = ld2(jh2, q.own);
    pdl_wait();
    float2 ps[6], ls[6], Ds[6], hi, lo, dn;
    gather_packed(phi, q, ps);
    gather_packed(phlo, q, ls);
    gather_packed(D, q, Ds);
    cell_ff_pair<LIM, ROUNDS>(ld2(phi, q.own), ld2(phlo, q.own), ps, ls, Ds, s2, a2, j2, lim_rt, larsen_n, omega,
                              inv2h, floor_, rounds_rt, hi, lo, dn);
    if (q.second) {
        *reinterpret_cast<float2 *>(phi + q.own) = hi;
        *reinterpret_cast<float2 *>(phlo + q.own) = lo;
        *reinterpret_cast<float2 *>(D + q.own) = dn;
    } else {
        phi[q.own] = hi.x;         // the element after the last unknown is a ghost: left untouched
        phlo[q.own] = lo.x;
        D[q.own] = dn.x;
    }
}

// The same pass with one unknown per thread: still the fastest on some grids of
// about 50^3, which have too few pairs for the GPU (us per iteration at 50^3:
// 9.2 against 10.7).
template <int LIM, int ROUNDS>
__device__ __forceinline__ void pass_ff_body(const Layout &L, const float *__restrict__ sp,
                                             const float *__restrict__ ah2, const float *__restrict__ jh2,
                                             float *__restrict__ phi, float *__restrict__ phlo,
                                             float *__restrict__ D, int colour, int t, int J, int K, int lim_rt,
                                             float larsen_n, float omega, float inv2h, float floor_,
                                             int rounds_rt) {
    Nbrs o;
    if (J > L.ny || !pass_cell(L, colour, t, J, K, o)) return;
    const float s_ = sp[o.own], ah = ah2[o.own], jj = jh2[o.own];
    pdl_wait();
    const float p0 = phi[o.own], p0lo = phlo[o.own];
    float ps[6], ls[6], Ds[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        ps[s] = phi[o.nb[s]];
        ls[s] = phlo[o.nb[s]];
        Ds[s] = D[o.nb[s]];
    }
    float hi, lo, Dp;
    cell_ff<LIM, ROUNDS>(p0, p0lo, ps, ls, Ds, s_, ah, jj, lim_rt, larsen_n, omega, inv2h, floor_, rounds_rt, hi, lo,
                         Dp);
    phi[o.own] = hi;
    phlo[o.own] = lo;
    D[o.own] = Dp;
}

template <int LIM, int ROUNDS>
__global__ void __launch_bounds__(256) k_pass_ff(Layout L, const float *__restrict__ sp,
                                                 const float *__restrict__ ah2, const float *__restrict__ jh2,
                                                 float *__restrict__ phi, float *__restrict__ phlo,
                                                 float *__restrict__ D, int colour, int lim_rt, float larsen_n,
                                                 float omega, float inv2h, float floor_, int rounds_rt) {
    pdl_launch_dependents();
    pass_ff_body<LIM, ROUNDS>(L, sp, ah2, jh2, phi, phlo, D, colour, blockIdx.x * blockDim.x + threadIdx.x,
                              blockIdx.y * blockDim.y + threadIdx.y + 1, blockIdx.z + 1, lim_rt, larsen_n, omega,
                              inv2h, floor_, rounds_rt);
}

// Jacobi variant: phi^{k+1} at every unknown (both colours) from phi^k
// (src) and D^k (written by the preceding fresh-D pass), into dst.  The update
// is the residual form of Eq. 32 damped by omega (Eq. 36): phi' = phi_p +
// omega S / den, S = j h^2 - sigma_a' h^2 phi_p + 1/2 (D_p sum d + sum D_s d),
// den = sigma_a' h^2 + 3 D_p + 1/2 sum D_s, d = phi_s - phi_p.
template <typename T>
__global__ void __launch_bounds__(256) k_jacobi(Layout L, const T *__restrict__ ah2, const T *__restrict__ jh2,
                                                const T *__restrict__ src, const T *__restrict__ D,
                                                T *__restrict__ dst, T omega) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= L.nx || j >= L.ny) return;
    const int q = L.at(i, j, k);
    const int nb[6] = {L.at(i - 1, j, k), L.at(i + 1, j, k), L.at(i, j - 1, k),
                       L.at(i, j + 1, k), L.at(i, j, k - 1), L.at(i, j, k + 1)};
    const T p0 = src[q], Dp = D[q], ah = ah2[q];
    T A = 0, B = 0, C = 0;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        const T d = src[nb[s]] - p0;
        const T Ds = D[nb[s]];
        A += d;
        B += Ds * d;
        C += Ds;
    }
    const T S = jh2[q] - ah * p0 + T(0.5) * (Dp * A + B);
    const T den = ah + T(3) * Dp + T(0.5) * C;
    dst[q] = p0 + omega * (S / den);
}

// Descriptor of a batched grid, read by every thread with uniform 16-byte
// loads (one transaction per warp, no shared-memory staging or barrier).
__device__ __forceinline__ BatchDesc load_desc(const BatchDesc *__restrict__ p) {
    BatchDesc d;
    const int4 *src = reinterpret_cast<const int4 *>(p);
    int4 *dst = reinterpret_cast<int4 *>(&d);
#pragma unroll
    for (int i = 0; i < (int)(sizeof(BatchDesc) / 16); ++i) dst[i] = __ldg(src + i);
    return d;
}

// FP64 colour pass.  The FP64 pipe takes 16 clocks a warp instruction (a 64th of
// the FP32 rate) whatever its active lanes, so what counts is instructions times
// warps.  Unknowns go by running number: a 32^3 grid's rows have 16 of a colour, and
// tiles of 32 left half of every warp idle.  And quotients are combined:
// R = g / d and 1 / R from one reciprocal of g d; Levermore-Pomraning as P / Q,
// P = ((1 - r)(1 - e) + 2 e) r / sigma', Q = 1 - e, r = 1/R, e = exp(-2 R), so that D = P / Q and
// delta = (P A / 2 + base Q) / ((sigma_a' h^2 + C / 2) Q + 3 P) share the reciprocal of Q times
// that denominator.  Two reciprocals per round instead of six quotients, a few ulp.
// 32^3: 19 -> 9.7 us a pass.
constexpr int kPassDThreads = 64;

template <int LIM, int ROUNDS>
__global__ void __launch_bounds__(kPassDThreads) k_pass_d(Layout L, PassIndex ix, const double *__restrict__ sp,
                                                const double *__restrict__ ah2, const double *__restrict__ jh2,
                                                double *__restrict__ phi, double *__restrict__ D, int colour,
                                                int lim_rt, double larsen_n, double omega, double inv2h,
                                                double floor_, int rounds_rt) {
    pdl_launch_dependents();
    const uint32_t e = blockIdx.x * (uint32_t)kPassDThreads + threadIdx.x;
    if (e >= ix.total) return;
    const uint32_t row = ix.by_items.quot(e);
    const int K = (int)ix.by_rows.quot(row), J = (int)row - K * L.ny;
    Nbrs o;
    if (!pass_cell(L, colour, (int)(e - row * ix.per_row), J + 1, K + 1, o)) return;
    const double s_ = sp[o.own], ah = ah2[o.own], jj = jh2[o.own];
    pdl_wait();
    const double p0 = phi[o.own];
    double ps[6], Ds[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        ps[s] = phi[o.nb[s]];
        Ds[s] = D[o.nb[s]];
    }
    const double gx = ps[1] - ps[0], gy = ps[3] - ps[2], gz = ps[5] - ps[4];
    const double gmax = fmax(inv2h * sqrt(fma(gx, gx, fma(gy, gy, gz * gz))), floor_);
    double A = 0.0, B = 0.0, C = 0.0;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        const double d = ps[s] - p0;
        A += d;
        B = fma(Ds[s], d, B);
        C += Ds[s];
    }
    const double base = fma(0.5, B, fma(-ah, p0, jj)), den0 = fma(0.5, C, ah);
    const double inv_sp = 1.0 / s_;
    const int lim = LIM >= 0 ? LIM : lim_rt;
    const int local_iters = ROUNDS > 0 ? ROUNDS : rounds_rt;
    double delta = 0.0, Dp = 0.0;
#pragma unroll(ROUNDS > 0 ? ROUNDS : 1)
    for (int r = 0; r < (ROUNDS > 0 ? ROUNDS : local_iters); ++r) {
        const double den = fmax(s_ * (p0 + delta), floor_);
        double P, Q = 1.0;
        // (the product of the two must stay a normal number)
        const bool ranged = LIM == LIM_LP && gmax > 1e-130 && gmax < 1e130 && den > 1e-130 && den < 1e130;
        if (ranged) {
            const double both = 1.0 / (gmax * den);
            const double R = gmax * gmax * both;
            if (R < 0.2) {
                P = lp_series_d(R) * inv_sp;
            } else {
                const double q = den * den * both;            // 1 / R
                double w = 1.0 - q;
                if (R < 20.0) {                                // exp(-40) is far below an ulp of 1 - 1/R
                    const double ex = exp(-2.0 * R);
                    Q = 1.0 - ex;
                    w = fma(w, Q, 2.0 * ex);
                }
                P = w * q * inv_sp;
            }
        } else {
            P = limiter_d(lim, larsen_n, gmax / den) * inv_sp;
        }
        const double N = fma(0.5 * P, A, base * Q), W = fma(3.0, P, den0 * Q);
        const double both = 1.0 / (Q * W);
        delta = N * (Q * both);     // (P W overflows where sigma' is below 1e-154)
        Dp = P * (W * both);
    }
    phi[o.own] = fma(omega, delta, p0);
    D[o.own] = Dp;
}

// ---------------------------------------------------------------------------
// Residual (Eq. 37) with D recomputed from the current phi.
// ---------------------------------------------------------------------------
// In single precision two kernels share this walk: CTA `cta` of `ctas` takes
// pairs of adjacent unknowns of one colour by running number (row by row, the
// two colours of a row after one another, so both find the fields they share in
// the caches), in strides of all CTAs.  One voxel per thread, the sums cost as
// much as the residual itself and left one pair of partial sums per 256 voxels
// for the last block to add: at 256^3 fresh D, residual and final sum took 104,
// 362 and 79 us; now 108, 179 and 7 (the residual: 448 instructions a pair, issue 49 %
// active, 72 registers; fresh D: 370 a pair, issue 73 %).
constexpr int kCheckThreads = 128;
constexpr int kCheckCtas = 2128;       // two waves of the residual's seven per SM of 152

template <typename F>
__device__ __forceinline__ void for_pairs(const Layout &L, const CheckIndex &ix, int cta, int ctas, F &&body) {
    for (uint32_t e = (uint32_t)cta * kCheckThreads + threadIdx.x; e < ix.total; e += (uint32_t)ctas * kCheckThreads) {
        const uint32_t row2 = ix.by_pairs.quot(e);
        const int t = 2 * (int)(e - row2 * ix.pairs);
        const int c = row2 & 1;
        const uint32_t row = row2 >> 1;
        const int K = (int)ix.by_rows.quot(row);
        const int J = (int)row - K * L.ny + 1;
        Pair q;
        pair_cells(L, c, t, J, K + 1, q);
        if (q.first) body(q, c, t, J, K + 1);
    }
}

// D from the current phi (hi + lo, LO; else hi alone) at every unknown.
template <bool LO>
__device__ __forceinline__ void fresh_D_pairs(const Layout &L, const CheckIndex &ix, int cta, int ctas,
                                              const float *__restrict__ sp, const float *__restrict__ phi,
                                              const float *__restrict__ phlo, float *__restrict__ Df, int lim,
                                              float larsen_n, float inv2h, float floor_) {
    for_pairs(L, ix, cta, ctas, [&](const Pair &q, int, int, int, int) {
        float2 ps[6], ls[6];
        gather_packed(phi, q, ps);
        if (LO) gather_packed(phlo, q, ls);
        const float2 s2 = ld2(sp, q.own), p0 = ld2(phi, q.own);
        const float2 g = grad_pair<LO>(ps, ls, inv2h, floor_);
        const float dx = D_of_f(D_point(g.x, s2.x), p0.x, floor_, lim, larsen_n);
        if (q.second) {
            const float dy = D_of_f(D_point(g.y, s2.y), p0.y, floor_, lim, larsen_n);
            *reinterpret_cast<float2 *>(Df + q.own) = make_float2(dx, dy);
        } else {
            Df[q.own] = dx;
        }
    });
}

__global__ void __launch_bounds__(kCheckThreads) k_fresh_D_f(Layout L, CheckIndex ix, const float *__restrict__ sp,
                                                              const float *__restrict__ phi,
                                                              const float *__restrict__ phlo, float *__restrict__ Df,
                                                              int lim, float larsen_n, float inv2h, float floor_) {
    if (phlo)
        fresh_D_pairs<true>(L, ix, blockIdx.x, gridDim.x, sp, phi, phlo, Df, lim, larsen_n, inv2h, floor_);
    else
        fresh_D_pairs<false>(L, ix, blockIdx.x, gridDim.x, sp, phi, phlo, Df, lim, larsen_n, inv2h, floor_);
}

__global__ void k_fresh_D_d(Layout L, const double *__restrict__ sp, const double *__restrict__ phi,
                            double *__restrict__ Df, int lim, double larsen_n, double inv2h, double floor_) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= L.nx || j >= L.ny) return;
    const int q = L.at(i, j, k);
    Df[q] = knudsen_D_d(phi[L.at(i + 1, j, k)] - phi[L.at(i - 1, j, k)],
                        phi[L.at(i, j + 1, k)] - phi[L.at(i, j - 1, k)],
                        phi[L.at(i, j, k + 1)] - phi[L.at(i, j, k - 1)], inv2h, sp[q], phi[q], floor_, lim, larsen_n);
}

// The two running sums of a residual check (in x and y) in three words each: every
// TwoSum's error is added to the next word, so that hundreds of terms a thread
// leave no more than one does. (By float-float additions 980 equal terms, whose
// roundings do not cancel, were 7e-13 off.) Packed, both take 11 us of the 179 at
// 256^3 more than float-float additions (scalar: 22).
struct Sums {
    float2 hi, lo, err;
};
__device__ __forceinline__ void sums_add(Sums &s, ff2 x) {
    const ff2 t = two_sum2(s.hi, x.hi), u = two_sum2(s.lo, t.lo), v = two_sum2(u.hi, x.lo);
    s.hi = t.hi;
    s.lo = v.hi;
    s.err = add2(s.err, add2(u.lo, v.lo));
}

// Their sums over the CTA, into its pair of partials: shuffles within each warp,
// then the warps' sums in FP64 in warp order (GB300's FP64 rate is a small
// fraction of its FP32 rate, so the per-element sums stay on the FP32 pipes).
__device__ __forceinline__ void store_partials(Sums v, double *__restrict__ p) {
    __shared__ double sh[2][kCheckThreads / 32];
    auto down = [](float2 a, int o) {
        return make_float2(__shfl_down_sync(0xffffffffu, a.x, o), __shfl_down_sync(0xffffffffu, a.y, o));
    };
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const ff2 u{down(v.hi, o), down(v.lo, o)};
        const float2 e = down(v.err, o);
        sums_add(v, u);
        v.err = add2(v.err, e);
    }
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = (double)v.hi.x + ((double)v.lo.x + (double)v.err.x);
        sh[1][threadIdx.x >> 5] = (double)v.hi.y + ((double)v.lo.y + (double)v.err.y);
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double a = 0.0;
#pragma unroll
        for (int w = 0; w < kCheckThreads / 32; ++w) a += sh[threadIdx.x][w];
        p[threadIdx.x] = a;
    }
}

// Residual R_p dl^2 = jh2 - ah2 phi_p + sum_s D_ps (phi_s - phi_p) in
// float-float (packed, as the correction pass forms it): per thread the sums of
// its square over the margin set and of the source's square over all unknowns.
template <bool LO>
__device__ __forceinline__ void residual_pairs(const Layout &L, const CheckIndex &ix, int cta, int ctas,
                                               const float *__restrict__ ah2, const float *__restrict__ jh2,
                                               const float *__restrict__ phi, const float *__restrict__ phlo,
                                               const float *__restrict__ Df, const float *__restrict__ Dghost,
                                               int margin, Sums &sums) {
    sums = Sums{both(0.0f), both(0.0f), both(0.0f)};
    for_pairs(L, ix, cta, ctas, [&](const Pair &q, int c, int t, int J, int K) {
        float2 ps[6], ls[6], Ds[6];
        gather_packed(phi, q, ps);
        if (LO) gather_packed(phlo, q, ls);
        const int I0 = 2 * t + 2 - ((J + K + 1 + c) & 1);      // padded I of the first unknown
        // ghost neighbours keep their Dirichlet D (never recomputed)
        const float2 xv = ld2(Df, q.xv);
        const float xe = q.left ? (I0 == 1 ? Dghost : Df)[q.xv - 1] : (I0 + 2 == L.nx ? Dghost : Df)[q.xv + 2];
        Ds[0] = q.left ? make_float2(xe, xv.x) : xv;
        Ds[1] = q.left ? xv : make_float2(xv.y, xe);
        if (I0 == L.nx) Ds[1].x = Dghost[q.left ? q.xv : q.xv + 1];
        if (q.left && I0 + 2 == L.nx) Ds[1].y = Dghost[q.xv + 1];
        Ds[2] = ld2(J == 1 ? Dghost : Df, q.ym);
        Ds[3] = ld2(J == L.ny ? Dghost : Df, q.yp);
        Ds[4] = ld2(K == 1 ? Dghost : Df, q.zm);
        Ds[5] = ld2(K == L.nz ? Dghost : Df, q.zp);
        const float2 jj = ld2(jh2, q.own);
        const FFTerms2 T = ff_terms_pair<LO>(ld2(phi, q.own), LO ? ld2(phlo, q.own) : both(0.0f), ps, ls, Ds,
                                         ld2(ah2, q.own), jj);
        const ff2 S = ff_S_pair(T, ld2(Df, q.own));
        const ff sx{S.hi.x, S.lo.x}, sy{S.hi.y, S.lo.y};
        const bool in = J > margin && J <= L.ny - margin && K > margin && K <= L.nz - margin;
        ff r0{0.0f, 0.0f}, r1{0.0f, 0.0f}, j0 = two_prod(jj.x, jj.x), j1{0.0f, 0.0f};
        if (in && I0 > margin && I0 <= L.nx - margin) r0 = ff_mul(sx, sx);
        if (q.second) {
            if (in && I0 + 2 > margin && I0 + 2 <= L.nx - margin) r1 = ff_mul(sy, sy);
            j1 = two_prod(jj.y, jj.y);
        }
        // the pair's two terms first (ff_add)
        const ff2 two = two_sum2(make_float2(r0.hi, j0.hi), make_float2(r1.hi, j1.hi));
        sums_add(sums, fast_two_sum2(two.hi, add2(two.lo, add2(make_float2(r0.lo, j0.lo), make_float2(r1.lo, j1.lo)))));
    });
}

__global__ void __launch_bounds__(kCheckThreads) k_residual_f(Layout L, CheckIndex ix, const float *__restrict__ ah2,
                                                               const float *__restrict__ jh2,
                                                               const float *__restrict__ phi,
                                                               const float *__restrict__ phlo,
                                                               const float *__restrict__ Df,
                                                               const float *__restrict__ Dghost, int margin,
                                                               double *__restrict__ partials) {
    Sums sums;
    if (phlo) residual_pairs<true>(L, ix, blockIdx.x, gridDim.x, ah2, jh2, phi, phlo, Df, Dghost, margin, sums);
    else residual_pairs<false>(L, ix, blockIdx.x, gridDim.x, ah2, jh2, phi, phlo, Df, Dghost, margin, sums);
    store_partials(sums, partials + 2 * (long long)blockIdx.x);
}

// Batched fresh D / residual / finalize: CTA b works on grid cta_grid[b] as CTA
// b - res_first of the solo launch's res_n, writes its partial sums to the grid's
// own slots, and one block per grid sums them in the solo order.
__global__ void __launch_bounds__(kCheckThreads) k_fresh_D_batch(const BatchDesc *__restrict__ descs,
                                                                  const int *__restrict__ cta_grid, int lim) {
    const BatchDesc d = load_desc(descs + __ldg(cta_grid + blockIdx.x));
    if (!d.active) return;
    const int local = blockIdx.x - d.res_first;
    if (d.mode)
        fresh_D_pairs<true>(d.L, d.ix, local, d.res_n, d.sp, d.phi, d.phlo, d.Df, lim, d.larsen_n, d.inv2h, d.floor_);
    else
        fresh_D_pairs<false>(d.L, d.ix, local, d.res_n, d.sp, d.phi, d.phlo, d.Df, lim, d.larsen_n, d.inv2h, d.floor_);
}

__global__ void __launch_bounds__(kCheckThreads) k_residual_batch(const BatchDesc *__restrict__ descs,
                                                                   const int *__restrict__ cta_grid, int margin,
                                                                   double *__restrict__ partials) {
    const BatchDesc d = load_desc(descs + __ldg(cta_grid + blockIdx.x));
    if (!d.active) return;
    const int local = blockIdx.x - d.res_first;
    Sums sums;
    if (d.mode) residual_pairs<true>(d.L, d.ix, local, d.res_n, d.ah2, d.jh2, d.phi, d.phlo, d.Df, d.D, margin, sums);
    else residual_pairs<false>(d.L, d.ix, local, d.res_n, d.ah2, d.jh2, d.phi, d.phlo, d.Df, d.D, margin, sums);
    store_partials(sums, partials + 2 * (long long)(d.res_slot + local));
}

__global__ void __launch_bounds__(kRedThreads) k_finalize_batch(const BatchDesc *__restrict__ descs,
                                                                const int *__restrict__ res_count,
                                                                const double *__restrict__ partials,
                                                                double *__restrict__ result) {
    __shared__ double sh[32];
    const BatchDesc &d = descs[blockIdx.x];
    if (!d.active) return;
    const int n = res_count[blockIdx.x];
    const double *p = partials + 2 * (long long)d.res_slot;
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        a += p[2 * i];
        b += p[2 * i + 1];
    }
    a = block_sum(a, sh);
    __syncthreads();
    b = block_sum(b, sh);
    if (threadIdx.x == 0) {
        result[2 * blockIdx.x] = a;
        result[2 * blockIdx.x + 1] = b;
    }
}

__global__ void __launch_bounds__(256) k_residual_d(Layout L, const double *__restrict__ ah2,
                                                    const double *__restrict__ jh2, const double *__restrict__ phi,
                                                    const double *__restrict__ Df, const double *__restrict__ Dghost,
                                                    int margin, double *__restrict__ partials) {
    __shared__ double sh[32];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    double r2 = 0.0, j2 = 0.0;
    if (i < L.nx && j < L.ny) {
        const int q = L.at(i, j, k);
        const int nb[6] = {L.at(i - 1, j, k), L.at(i + 1, j, k), L.at(i, j - 1, k),
                           L.at(i, j + 1, k), L.at(i, j, k - 1), L.at(i, j, k + 1)};
        const bool onface[6] = {i == 0, i == L.nx - 1, j == 0, j == L.ny - 1, k == 0, k == L.nz - 1};
        const double p0 = phi[q], Dp = Df[q];
        double A = 0.0, B = 0.0;
#pragma unroll
        for (int s = 0; s < 6; ++s) {
            const double Dn = onface[s] ? Dghost[nb[s]] : Df[nb[s]];
            const double d = phi[nb[s]] - p0;
            A += d;
            B = fma(Dn, d, B);
        }
        const double S = fma(0.5 * Dp, A, fma(0.5, B, fma(-ah2[q], p0, jh2[q])));
        const bool in = i >= margin && i < L.nx - margin && j >= margin && j < L.ny - margin && k >= margin &&
                        k < L.nz - margin;
        r2 = in ? S * S : 0.0;
        j2 = jh2[q] * jh2[q];
    }
    r2 = block_sum(r2, sh);
    __syncthreads();
    j2 = block_sum(j2, sh);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        const long long b = blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z);
        partials[2 * b] = r2;
        partials[2 * b + 1] = j2;
    }
}

__global__ void __launch_bounds__(256) k_sumsq(long long n, const float *__restrict__ x,
                                               double *__restrict__ partials) {
    __shared__ double sh[32];
    double a = 0.0;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const double v = (double)x[e];
        a += v * v;
    }
    a = block_sum(a, sh);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = a;
        partials[2 * blockIdx.x + 1] = 0.0;
    }
}

// Input validation counters: [0] bad sigma (NaN/neg/inf), [1] bad albedo, [2] bad j.
__global__ void __launch_bounds__(256) k_validate(long long n, const float *__restrict__ st,
                                                  const float *__restrict__ alb, const float *__restrict__ js,
                                                  double *__restrict__ partials) {
    __shared__ double sh[32];
    double bs = 0.0, ba = 0.0;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        if (st) {
            const float s = st[e];
            bs += !(s >= 0.0f && s <= 3.0e38f) ? 1.0 : 0.0;
        }
        if (alb) {
            const float a = alb[e];
            ba += !(a >= 0.0f && a <= 1.0f) ? 1.0 : 0.0;
        }
        if (js) {
            const float v = js[e];
            bs += !(v >= 0.0f && v <= 3.0e38f) ? 1.0 : 0.0;
        }
    }
    bs = block_sum(bs, sh);
    __syncthreads();
    ba = block_sum(ba, sh);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = bs;
        partials[2 * blockIdx.x + 1] = ba;
    }
}

// ---------------------------------------------------------------------------
// Single-scatter source.
// ---------------------------------------------------------------------------

// exp(-(t.hi + t.lo)) for an optical depth held as a float-float pair
// (|t.lo| <= ulp(t.hi)/2, so exp(-t.lo) = 1 - t.lo to single precision)
__device__ __forceinline__ float transmittance(ff t) { return expf(-t.hi) * (1.0f - t.lo); }

// Light along -z with step h/2: the samples at quarter-voxel offsets blend the
// two nearest centres 3:1 and 1:3, so the optical depth above voxel k is the
// trapezoid sum over the centres above it plus half a voxel of the top
// centre -- an exclusive scan down each column.  Each trapezoid term
// (h/2)(s + s_above) is formed exactly as a float-float pair (TwoSum, then
// TwoProd by h/2) and summed in float-float, so the depth is as accurate as
// a double-precision sum without double-precision arithmetic.
__global__ void k_bake_scan_negz(Layout L, const float *__restrict__ st, const float *__restrict__ alb,
                                 float *__restrict__ js, float h, float radiance, int accumulate) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= L.nx || j >= L.ny) return;
    const long long col = (long long)j * L.nx + i;
    const long long sk = (long long)L.nx * L.ny;
    const float hh = 0.5f * h;
    ff tau = {0.0f, 0.0f};
    float above = 0.0f;
    // eight voxels at a time, their loads before the chain of sums (128^3: 93 -> 76 us)
    constexpr int kBatch = 8;
    for (int k0 = L.nz - 1; k0 >= 0; k0 -= kBatch) {
        float sb[kBatch], ab[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const long long v = col + (long long)max(k0 - u, 0) * sk;
            sb[u] = st[v];
            ab[u] = alb[v];
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int k = k0 - u;
            if (k < 0) break;
            const long long v = col + (long long)k * sk;
            const float s = sb[u];
            const ff sum = (k == L.nz - 1) ? ff{s, 0.0f} : two_sum(s, above);
            const ff p = two_prod(sum.hi, hh);
            tau = ff_add(tau, fast_two_sum(p.hi, fmaf(sum.lo, hh, p.lo)));
            above = s;
            const float q = radiance * (ab[u] * s) * transmittance(tau);
            js[v] = accumulate ? js[v] + q : q;
        }
    }
}

// General march: from the voxel centre towards the light, samples at the
// midpoints of steps of length `step`, the last step shortened to end at the
// grid boundary (or at a point light inside the grid).  Lengths are in voxels, so a
// sample's coordinate between centres is i + t w, one FMA per axis.  Bound by
// issue (about 60 instructions a sample) and the loads of the eight corners from
// L1 (two samples at a time in packed sums and blends: 2 % only): its
// predecessor divided by h three times, floored by conversions and formed 64-bit
// indices for every sample, and marched for voxels that scatter nothing, whose
// source is zero whatever the transmittance (62 % of the box of a sphere cloud).
// A point light over a 160^3 cloud: 4.27 -> 0.87 ms, and 0.77 with the fraction
// saturated instead of the coordinate clamped, the sample's number counted in
// float and 32-bit byte offsets (the same bits); an oblique light, 200^3: 8.4 ->
// 1.9 -> 1.7 ms.  Error against 64 bits 9.8e-7 -> 5.2e-7.
//
// t = (u - 1/2) + M, M = 1.5 2^23, rounds u - 1/2 to an integer in t's low bits:
// the lower corner b (u itself if it is one: the blend is the same from either
// side).  That needs n <= 2^20; WIDE converts instead, and takes axes of one voxel
// (whose upper corner is the lower one), more voxels than a byte offset reaches and
// steps so short that the count would lose its half.
constexpr float kRound = 12582912.0f;
constexpr int kRoundMax = 1 << 20;

struct MarchAxis {
    float top, last;             // n - 1; the largest lower corner, plus kRound
    int n, stride;               // voxels; elements to the upper corner
};

__device__ __forceinline__ float lower_corner(const MarchAxis &a, float &u, int &b) {
    u = fminf(fmaxf(u, 0.0f), a.top);
    b = min(max((int)floorf(u), 0), max(a.n - 2, 0));
    return u - (float)b;
}

// Two instructions, as a + f (b - a) takes, but exact at both ends and never off by
// more than two roundings of the result: that one reads 9.77e-4 at f = 1 between
// 1e4 and 1e-3, the rounding of the dense side.
__device__ __forceinline__ float blend(float f, float a, float b) { return fmaf(f, b, fmaf(-f, a, a)); }

template <bool WIDE>
__device__ __forceinline__ float sigma_at(const float *__restrict__ st, const MarchAxis ax[3], const int sy, const int sz,
                                          const int bias, float ux, float uy, float uz) {
    const float *p, *py, *pz, *pyz;
    float fx, fy, fz;
    if (WIDE) {
        int bx, by, bz;
        fx = lower_corner(ax[0], ux, bx);
        fy = lower_corner(ax[1], uy, by);
        fz = lower_corner(ax[2], uz, bz);
        p = st + (bz * sz + by * sy + bx);
        py = p + ax[1].stride;
        pz = p + ax[2].stride;
        pyz = py + ax[2].stride;
    } else {
        // outside the centres the corner is held and the fraction saturates
        const float tx = fminf(fmaxf(__fadd_rn(__fadd_rn(ux, -0.5f), kRound), kRound), ax[0].last);
        const float ty = fminf(fmaxf(__fadd_rn(__fadd_rn(uy, -0.5f), kRound), kRound), ax[1].last);
        const float tz = fminf(fmaxf(__fadd_rn(__fadd_rn(uz, -0.5f), kRound), kRound), ax[2].last);
        fx = __saturatef(ux - __fsub_rn(tx, kRound));
        fy = __saturatef(uy - __fsub_rn(ty, kRound));
        fz = __saturatef(uz - __fsub_rn(tz, kRound));
        // offsets in bytes, 32 bits (the bits of M cancel in `bias`, modulo 2^32)
        const uint32_t q = (uint32_t)__float_as_int(tz) * (4u * (uint32_t)sz) +
                           (uint32_t)__float_as_int(ty) * (4u * (uint32_t)sy) +
                           (uint32_t)__float_as_int(tx) * 4u - (uint32_t)bias;
        const char *at = (const char *)st;
        p = (const float *)(at + q);
        py = (const float *)(at + (q + 4u * (uint32_t)sy));
        pz = (const float *)(at + (q + 4u * (uint32_t)sz));
        pyz = (const float *)(at + (q + 4u * (uint32_t)(sy + sz)));
    }
    const int dx = WIDE ? ax[0].stride : 1;
    const float a0 = __ldg(p), a1 = __ldg(p + dx), b0 = __ldg(py), b1 = __ldg(py + dx);
    const float c0 = __ldg(pz), c1 = __ldg(pz + dx), d0 = __ldg(pyz), d1 = __ldg(pyz + dx);
    const float a = blend(fx, a0, a1), b = blend(fx, b0, b1), c = blend(fx, c0, c1), d = blend(fx, d0, d1);
    return blend(fz, blend(fy, a, b), blend(fy, c, d));
}

// Where the light is, in voxels: the unit direction towards it, or its position.
// Beyond kFarLight (of a voxel, or of the world's unit) squares near the end of
// the range of a float; beyond kFarthest the host scales the position nearer,
// where the direction from every voxel is the same to the last bit.
constexpr float kFarLight = 1e18f;
constexpr double kFarthest = 1e30;
struct MarchLight {
    float w[3], pos[3];
    int point;
    float value, step, h;
    float unit;                  // world length of a unit of pos: h, unless the light is scaled nearer
};

template <bool WIDE>
__global__ void __launch_bounds__(256) k_bake_march(Layout L, const float *__restrict__ st,
                                                    const float *__restrict__ alb, float *__restrict__ js,
                                                    MarchLight m, int accumulate) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= L.nx || j >= L.ny) return;
    const long long v = ((long long)k * L.ny + j) * L.nx + i;
    const float scatter = __fmul_rn(alb[v], st[v]);
    if (scatter == 0.0f) {
        if (!accumulate) js[v] = 0.0f;
        return;
    }
    const int n[3] = {L.nx, L.ny, L.nz};
    const float x[3] = {(float)i, (float)j, (float)k};       // the centre, from the first centre
    float w[3] = {m.w[0], m.w[1], m.w[2]};
    float r = 0.0f;
    if (m.point) {
        float d[3] = {m.pos[0] - x[0], m.pos[1] - x[1], m.pos[2] - x[2]};
        // for a light so far that the squares overflow the march would find neither
        // direction nor end (2^31 samples): the components go relative to the largest
        const float most = fmaxf(fmaxf(fabsf(d[0]), fabsf(d[1])), fabsf(d[2]));
        const float scale = most > kFarLight ? most : 1.0f;
        if (most > kFarLight) {
            d[0] /= scale; d[1] /= scale; d[2] /= scale;
        }
        r = sqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
        if (r > 0.0f) {
            w[0] = d[0] / r; w[1] = d[1] / r; w[2] = d[2] / r;
        }
        r *= scale;
    }
    float len = INFINITY;
    MarchAxis ax[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (w[a] > 0.0f) len = fminf(len, ((float)n[a] - 0.5f - x[a]) / w[a]);
        else if (w[a] < 0.0f) len = fminf(len, (-0.5f - x[a]) / w[a]);
        ax[a].top = (float)(n[a] - 1);
        ax[a].last = kRound + (float)max(n[a] - 2, 0);
        ax[a].n = n[a];
        ax[a].stride = n[a] == 1 ? 0 : a == 0 ? 1 : a == 1 ? L.nx : L.nx * L.ny;
    }
    if (m.point) len = (r > 0.0f) ? fminf(len, r) : 0.0f;
    const int sy = L.nx, sz = L.nx * L.ny;
    const uint32_t mb = (uint32_t)__float_as_int(kRound);
    const int bias = (int)(4u * (mb * (uint32_t)sz + mb * (uint32_t)sy + mb));
    // sum of the samples in float-float: TwoSum, the errors in a word of their own
    // that every fourth sample folds back (left to grow, its own rounding reached 9e-7 of
    // the sum over 1e5 equal samples)
    ff sum = {0.0f, 0.0f};
    const int m_full = (int)floorf(len / m.step);
    float mid = 0.5f;            // q + 1/2 (exact; WIDE takes marches of over 2^20 steps)
    auto sample = [&](int q) {
        const float t = (WIDE ? (float)q + 0.5f : mid) * m.step;
        mid += 1.0f;
        const float s = sigma_at<WIDE>(st, ax, sy, sz, bias, fmaf(t, w[0], x[0]), fmaf(t, w[1], x[1]),
                                       fmaf(t, w[2], x[2]));
        const ff u = two_sum(sum.hi, s);
        sum.hi = u.hi;
        sum.lo = __fadd_rn(sum.lo, u.lo);
    };
    int q = 0;
    for (; q < m_full - 3; q += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) sample(q + u);
        sum = fast_two_sum(sum.hi, sum.lo);
    }
    for (; q < m_full; ++q) sample(q);
    ff tau = ff_mul_f(fast_two_sum(sum.hi, sum.lo), m.step);
    const float rem = len - (float)m_full * m.step;
    if (rem > 1e-6f * m.step) {
        const float t = (float)m_full * m.step + 0.5f * rem;
        tau = ff_add_f(tau, sigma_at<WIDE>(st, ax, sy, sz, bias, fmaf(t, w[0], x[0]), fmaf(t, w[1], x[1]),
                                           fmaf(t, w[2], x[2])) * rem);
    }
    float e = m.value * scatter * transmittance(ff_mul_f(tau, m.h));
    if (m.point) {
        const float rr = fmaxf(r, 0.5f) * m.unit;
        const float area = 4.0f * 3.14159265358979f * rr;
        e = rr > kFarLight ? e / area / rr : e / (area * rr);
    }
    js[v] = accumulate ? js[v] + e : e;
}

// One thread per unknown of the colour in a row (ceil(nx/2) of them), one
// y-row per thread row, one z-plane per block z.
inline dim3 pass_grid(const Layout &L, dim3 blk) {
    const int half = (L.nx + 1) / 2;
    return dim3((half + blk.x - 1) / blk.x, (L.ny + blk.y - 1) / blk.y, L.nz);
}

// Grid and item numbering of a launched pass with the given number of items per
// row; run: by running number (pass_item).
inline dim3 item_grid(const Layout &L, int per_row, bool run, PassIndex *ix) {
    ix->per_row = (uint32_t)per_row;
    ix->total = (uint32_t)per_row * (uint32_t)L.ny * (uint32_t)L.nz;
    ix->by_items.set((uint32_t)per_row);
    ix->by_rows.set((uint32_t)L.ny);
    if (run) return dim3((ix->total + kPassThreads - 1) / kPassThreads);
    const int rows = kPassThreads / 32;
    return dim3((per_row + 31) / 32, (L.ny + rows - 1) / rows, L.nz);
}

// work items of the multi-grid pass: ceil(half / 2) pairs per half row
inline dim3 pass2_grid(const Layout &L, dim3 blk) {
    const int pairs = ((L.nx + 1) / 2 + 1) / 2;
    return dim3((pairs + blk.x - 1) / blk.x, (L.ny + blk.y - 1) / blk.y, L.nz);
}

// four unknowns per thread (k_pass4): ceil(half / 4) threads per half row
inline dim3 pass4_grid(const Layout &L, dim3 blk) {
    const int quads = ((L.nx + 1) / 2 + 3) / 4;
    return dim3((quads + blk.x - 1) / blk.x, (L.ny + blk.y - 1) / blk.y, L.nz);
}

// Whether a pass takes its items by running number: as asked (0 tiles, 1
// running), or (-1) where 32-wide tiles would leave more than a sixth of the
// lanes idle.  Measured at the ends: 33 items a row (131 x 97 x 115 hi/lo) 20.6 ->
// 13.4 us per iteration, 40 (160^3) 51.8 -> 37.0; 32 (128^3) 17.0 tiled against
// 17.7 running.
// A launch's y and z extents end at 65535: longer grids run.
inline bool pass_runs(const Layout &L, int per_row, int asked) {
    if ((L.ny + kPassThreads / 32 - 1) / (kPassThreads / 32) > 65535 || L.nz > 65535) return true;
    if (asked >= 0) return asked != 0;
    return 6 * per_row < 5 * 32 * ((per_row + 31) / 32);
}

inline dim3 vox_block() { return dim3(32, 8, 1); }
inline dim3 vox_grid(const Layout &L) {
    return dim3((L.nx + 31) / 32, (L.ny + 7) / 8, L.nz);
}

}  // namespace

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
cudaError_t launch_prep_f(const Layout &L, const Fields &f, float sigma_eps, float h2, bool bf16, cudaStream_t s) {
    auto k = bf16 ? k_prep_f<true> : k_prep_f<false>;
    k<<<vox_grid(L), vox_block(), 0, s>>>(L, f.sigma_t, f.albedo, f.jsrc, f.sp, f.ah2, f.jh2, f.spb, f.sab, sigma_eps,
                                          h2);
    return cudaGetLastError();
}

cudaError_t launch_prep_d(const Layout &L, const Fields &f, double sigma_eps, double h2, bool bf16,
                          cudaStream_t s) {
    auto k = bf16 ? k_prep_d<true> : k_prep_d<false>;
    k<<<vox_grid(L), vox_block(), 0, s>>>(L, f.sigma_t, f.albedo, f.jsrc, f.sp64, f.ah264, f.jh264, sigma_eps, h2);
    return cudaGetLastError();
}

cudaError_t launch_init_f(const Layout &L, float *phi, float *phlo, float *D, double phi0, double D0, double phi_b,
                          double D_b, cudaStream_t s) {
    const int blk = 256;
    const int nb = (L.total / 4 + blk - 1) / blk;
    Divisor by_quads, by_py;
    by_quads.set((uint32_t)L.hpx / 4);
    by_py.set((uint32_t)L.py);
    k_init<float><<<nb, blk, 0, s>>>(L, by_quads, by_py, phi, phlo, D, (float)phi0, (float)D0, (float)phi_b, (float)D_b);
    return cudaGetLastError();
}

cudaError_t launch_init_d(const Layout &L, double *phi, double *D, double phi0, double D0, double phi_b, double D_b,
                          cudaStream_t s) {
    const int blk = 256;
    const int nb = (L.total / 4 + blk - 1) / blk;
    Divisor by_quads, by_py;
    by_quads.set((uint32_t)L.hpx / 4);
    by_py.set((uint32_t)L.py);
    k_init<double><<<nb, blk, 0, s>>>(L, by_quads, by_py, phi, nullptr, D, phi0, D0, phi_b, D_b);
    return cudaGetLastError();
}

static PackedIndex packed_index(const Layout &L, unsigned *blocks) {
    PackedIndex ix;
    ix.row = (uint32_t)(L.nx + 2);
    ix.rows = (uint32_t)(L.ny + 2);
    ix.total = ix.row * ix.rows * (uint32_t)(L.nz + 2);
    ix.by_row.set(ix.row);
    ix.by_rows.set(ix.rows);
    const unsigned per = kMoveThreads * kMovePer;
    *blocks = (ix.total + per - 1) / per;
    return ix;
}

cudaError_t launch_unpack(const Layout &L, const double *src, float *hi, float *lo, double *dst, cudaStream_t s) {
    unsigned nb;
    const PackedIndex ix = packed_index(L, &nb);
    k_unpack<<<nb, kMoveThreads, 0, s>>>(L, ix, src, hi, lo, dst);
    return cudaGetLastError();
}
cudaError_t launch_pack_from_f(const Layout &L, const float *hi, const float *lo, double *dst, cudaStream_t s) {
    unsigned nb;
    const PackedIndex ix = packed_index(L, &nb);
    k_pack_from_f<<<nb, kMoveThreads, 0, s>>>(L, ix, hi, lo, dst);
    return cudaGetLastError();
}
cudaError_t launch_pack_from_d(const Layout &L, const double *src, double *dst, cudaStream_t s) {
    unsigned nb;
    const PackedIndex ix = packed_index(L, &nb);
    k_pack_from_d<<<nb, kMoveThreads, 0, s>>>(L, ix, src, dst);
    return cudaGetLastError();
}
cudaError_t launch_f_to_d(const Layout &L, const float *hi, const float *lo, double *dst, cudaStream_t s) {
    k_f_to_d<<<(L.total + 255) / 256, 256, 0, s>>>(L.total, hi, lo, dst);
    return cudaGetLastError();
}
cudaError_t launch_d_to_f(const Layout &L, const double *src, float *hi, float *lo, cudaStream_t s) {
    k_d_to_f<<<(L.total + 255) / 256, 256, 0, s>>>(L.total, src, hi, lo);
    return cudaGetLastError();
}

// Launch with programmatic stream serialisation (early): the kernel may be
// scheduled while the preceding grid in the stream finishes (see pdl_wait).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(bool early, void (*k)(KArgs...), dim3 grd, dim3 blk, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grd;
    cfg.blockDim = blk;
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

// Whether a pass of so many CTAs is launched early.  The CTAs of a small grid, placed
// around those of the preceding pass that still run, end up two or three on some SMs and
// none on others, and from pass to pass the placement gets worse (50^3 FP32, us per
// iteration: 3.5 over 16 iterations, 4.1 over 64, 5.5 over 512; never early 4.3).  So every
// kSettleEvery-th of their passes waits for the preceding one to end, and the
// next start from an even placement again: 3.2.  Measured so, FP32 / hi/lo / float-float:
// 32^3 2.7 / 3.3 / 4.5 (all early 2.6 / 3.3 / 5.2), 50^3 3.2 / 4.5 / 6.4 (5.5 / 7.2 / 6.6), 64^3 4.2 / 5.3 / 8.0
// (6.1 / 5.4 / 8.0); 4, 16 and 32 launches differ by 3 %.  From 80^3 on all early is as fast
// or faster (96^3 7.7 against 7.9).  Otherwise as asked by the tuner, or (-1) if there
// are more than six CTAs per SM.  Launches that do not come from a graph are 4 us apart
// unless early: those only settle (256 iterations of 54^3 FP32 through fld_iterate, us
// each: 6.1 all early, 4.7; start 6.0), up to a size at which it costs more than it saves
// (80^3 hi/lo 7.5, settled 8.1); FP64 passes take longer than that
// (32^3, a pass in a graph: all early 20 us, never 9.9, settled 9.7).
// A grid of one voxel is never early: no thread of its black pass has an unknown, so
// none waits for the red pass, and the next one would follow an empty pass alone.
constexpr long long kEarlyCtas = 912, kSettleCtas = 1216;
bool pass_early(const PassParams &p, Family fam, const Layout &L, dim3 g) {
    const long long ctas = (long long)g.x * g.y * g.z;
    if (p.settle == 2 || (L.nx == 1 && L.ny == 1 && L.nz == 1)) return false;
    if (p.settle && ctas <= (p.direct ? kEarlyCtas : kSettleCtas)) return false;
    if (fam != FAM_F64 && p.direct) return true;
    const int asked = fam == FAM_F32 ? p.early_f32 : fam == FAM_FH ? p.early_fh : fam == FAM_FF ? p.early_ff : 1;
    return asked >= 0 ? asked != 0 : ctas > kEarlyCtas;
}

cudaError_t launch_pass(Family fam, const Layout &L, const Fields &f, const PassParams &p, int colour,
                        cudaStream_t s) {
    const dim3 blk(32, 8, 1);
    const dim3 grd = pass_grid(L, blk);
    const int pairs = ((L.nx + 1) / 2 + 1) / 2;
    if (fam != FAM_F64 && fam != FAM_FF && (fam == FAM_F32 ? p.single_f32 : p.single_fh)) {
        PassIndex ix;
        const dim3 g1 = item_grid(L, (L.nx + 1) / 2, true, &ix);
        auto k = fam == FAM_FH ? k_pass1<-1, 0, true> : k_pass1<-1, 0, false>;
        if (p.local_iters == 2 && p.lim == LIM_LP) k = fam == FAM_FH ? k_pass1<LIM_LP, 2, true> : k_pass1<LIM_LP, 2, false>;
        else if (p.local_iters == 2 && p.lim == LIM_KERSHAW)
            k = fam == FAM_FH ? k_pass1<LIM_KERSHAW, 2, true> : k_pass1<LIM_KERSHAW, 2, false>;
        else if (p.local_iters == 2 && p.lim == LIM_LARSEN)
            k = fam == FAM_FH ? k_pass1<LIM_LARSEN, 2, true> : k_pass1<LIM_LARSEN, 2, false>;
        return launch_pdl(pass_early(p, fam, L, g1), k, g1, dim3(kPassThreads), s, L, ix, f.sp, f.ah2, f.jh2, f.phi,
                          f.phlo, f.D, colour, p.lim, (float)p.larsen_n, (float)p.omega, (float)p.inv2h,
                          (float)p.floor_, p.local_iters);
    }
    switch (fam) {
    case FAM_F32:
    case FAM_FH:
        if (fam == FAM_F32 ? p.quad_f32 : p.quad_fh) {
            const dim3 blk4(32, 4, 1);
            const dim3 grd4 = pass4_grid(L, blk4);
            auto pick4 = [&](auto bf, auto hl) {
                constexpr bool B = decltype(bf)::value, H = decltype(hl)::value;
                auto k = k_pass4<-1, 0, B, H>;
                if (p.local_iters == 2 && p.lim == LIM_LP) k = k_pass4<LIM_LP, 2, B, H>;
                return launch_pdl(pass_early(p, fam, L, grd4), k, grd4, blk4, s, L, f.sp, f.ah2, f.jh2, f.spb, f.sab, (float)p.h2, f.phi, f.phlo,
                                  f.D, colour, p.lim, (float)p.larsen_n, (float)p.omega, (float)p.inv2h,
                                  (float)p.floor_, p.local_iters);
            };
            if (fam == FAM_FH)
                return p.bf16 ? pick4(std::true_type{}, std::true_type{}) : pick4(std::false_type{}, std::true_type{});
            return p.bf16 ? pick4(std::true_type{}, std::false_type{}) : pick4(std::false_type{}, std::false_type{});
        }
        if (fam == FAM_FH) break;
        {
        auto pick = [&](auto bf, auto run) {
            constexpr bool B = decltype(bf)::value, R = decltype(run)::value;
            auto k = k_pass2_f32<-1, 0, B, R>;
            if (p.local_iters == 2 && p.lim == LIM_LP) k = k_pass2_f32<LIM_LP, 2, B, R>;
            else if (p.local_iters == 2 && p.lim == LIM_KERSHAW) k = k_pass2_f32<LIM_KERSHAW, 2, B, R>;
            else if (p.local_iters == 2 && p.lim == LIM_LARSEN) k = k_pass2_f32<LIM_LARSEN, 2, B, R>;
            PassIndex ix;
            const dim3 g2 = item_grid(L, pairs, R, &ix);
            return launch_pdl(pass_early(p, fam, L, g2), k, g2, dim3(kPassThreads), s, L, ix, f.sp, f.ah2, f.jh2, f.spb, f.sab, (float)p.h2, f.phi, f.D, colour,
                              p.lim, (float)p.larsen_n, (float)p.omega, (float)p.inv2h, (float)p.floor_,
                              p.local_iters);
        };
        if (pass_runs(L, pairs, p.run_f32))
            return p.bf16 ? pick(std::true_type{}, std::true_type{}) : pick(std::false_type{}, std::true_type{});
        return p.bf16 ? pick(std::true_type{}, std::false_type{}) : pick(std::false_type{}, std::false_type{});
        }
    default:
        break;
    }
    switch (fam) {
    case FAM_FF: {
        PassIndex ix;
        if (p.ff_form == 2) {
            auto k = k_pass_ff<-1, 0>;
            if (p.local_iters == 2 && p.lim == LIM_LP) k = k_pass_ff<LIM_LP, 2>;
            else if (p.local_iters == 2 && p.lim == LIM_KERSHAW) k = k_pass_ff<LIM_KERSHAW, 2>;
            else if (p.local_iters == 2 && p.lim == LIM_LARSEN) k = k_pass_ff<LIM_LARSEN, 2>;
            return launch_pdl(pass_early(p, fam, L, grd), k, grd, blk, s, L, f.sp, f.ah2, f.jh2, f.phi, f.phlo, f.D, colour, p.lim,
                              (float)p.larsen_n, (float)p.omega, (float)p.inv2h, (float)p.floor_, p.local_iters);
        }
        auto pick = [&](auto run) {
            constexpr bool R = decltype(run)::value;
            const dim3 g2 = item_grid(L, pairs, R, &ix);
            auto k = k_pass2_ff<-1, 0, R, 7>;
            if (p.local_iters == 2 && p.lim == LIM_LP)
                k = p.ff_form == 1 || (p.ff_form < 0 && (long long)g2.x * g2.y * g2.z <= kSmallCtas)
                        ? k_pass2_ff<LIM_LP, 2, R, 5> : k_pass2_ff<LIM_LP, 2, R, 7>;
            else if (p.local_iters == 2 && p.lim == LIM_KERSHAW) k = k_pass2_ff<LIM_KERSHAW, 2, R, 7>;
            else if (p.local_iters == 2 && p.lim == LIM_LARSEN) k = k_pass2_ff<LIM_LARSEN, 2, R, 7>;
            return launch_pdl(pass_early(p, fam, L, g2), k, g2, dim3(kPassThreads), s, L, ix, f.sp, f.ah2, f.jh2, f.phi, f.phlo, f.D, colour,
                              p.lim, (float)p.larsen_n, (float)p.omega, (float)p.inv2h, (float)p.floor_,
                              p.local_iters);
        };
        return pass_runs(L, pairs, -1) ? pick(std::true_type{}) : pick(std::false_type{});
    }
    case FAM_FH: {
        auto pick = [&](auto bf, auto run) {
            constexpr bool B = decltype(bf)::value, R = decltype(run)::value;
            auto k = k_pass2_fh<-1, 0, B, R>;
            if (p.local_iters == 2 && p.lim == LIM_LP) k = k_pass2_fh<LIM_LP, 2, B, R>;
            else if (p.local_iters == 2 && p.lim == LIM_KERSHAW) k = k_pass2_fh<LIM_KERSHAW, 2, B, R>;
            else if (p.local_iters == 2 && p.lim == LIM_LARSEN) k = k_pass2_fh<LIM_LARSEN, 2, B, R>;
            PassIndex ix;
            const dim3 g2 = item_grid(L, pairs, R, &ix);
            return launch_pdl(pass_early(p, fam, L, g2), k, g2, dim3(kPassThreads), s, L, ix, f.sp, f.ah2, f.jh2, f.spb, f.sab, (float)p.h2, f.phi, f.phlo,
                              f.D, colour, p.lim, (float)p.larsen_n, (float)p.omega, (float)p.inv2h,
                              (float)p.floor_, p.local_iters);
        };
        if (pass_runs(L, pairs, p.run_fh))
            return p.bf16 ? pick(std::true_type{}, std::true_type{}) : pick(std::false_type{}, std::true_type{});
        return p.bf16 ? pick(std::true_type{}, std::false_type{}) : pick(std::false_type{}, std::false_type{});
    }
    case FAM_F64:
        {
        PassIndex ix;
        item_grid(L, (L.nx + 1) / 2, true, &ix);
        auto k = k_pass_d<-1, 0>;
        if (p.local_iters == 2 && p.lim == LIM_LP) k = k_pass_d<LIM_LP, 2>;
        const dim3 gd((ix.total + kPassDThreads - 1) / kPassDThreads);
        return launch_pdl(pass_early(p, fam, L, gd), k, gd, dim3(kPassDThreads), s, L, ix,
                          f.sp64, f.ah264, f.jh264, f.phi64, f.D64, colour, p.lim, p.larsen_n, p.omega, p.inv2h,
                          p.floor_, p.local_iters);
        }
    }
    return cudaGetLastError();
}

CheckIndex check_index(const Layout &L, int *ctas) {
    CheckIndex ix;
    ix.pairs = (uint32_t)(((L.nx + 1) / 2 + 1) / 2);
    ix.total = 2u * ix.pairs * (uint32_t)L.ny * (uint32_t)L.nz;
    ix.by_pairs.set(ix.pairs);
    ix.by_rows.set((uint32_t)L.ny);
    const uint32_t want = (ix.total + kCheckThreads - 1) / kCheckThreads;
    *ctas = (int)(want < (uint32_t)kCheckCtas ? want : (uint32_t)kCheckCtas);
    return ix;
}

cudaError_t launch_residual_batch(const BatchDesc *descs, const int *cta_grid, int nctas, int ngrids,
                                  const int *res_count, double *partials, double *result, int lim, int margin,
                                  cudaStream_t s) {
    if (nctas <= 0) return cudaSuccess;
    k_fresh_D_batch<<<nctas, kCheckThreads, 0, s>>>(descs, cta_grid, lim);
    k_residual_batch<<<nctas, kCheckThreads, 0, s>>>(descs, cta_grid, margin, partials);
    k_finalize_batch<<<ngrids, kRedThreads, 0, s>>>(descs, res_count, partials, result);
    return cudaGetLastError();
}

void multi_dims(const Layout &L, int *bx, int *by) {
    const dim3 g = pass2_grid(L, dim3(kMultiThreadsX, kMultiThreadsY, 1));
    *bx = (int)g.x;
    *by = (int)g.y;
}

int multi_ctas(int nsm, int hl, int bf16, int lim, int local_iters) {
    auto k = hl ? (bf16 ? multi_kernel<true, true>(lim, local_iters) : multi_kernel<false, true>(lim, local_iters))
                : (bf16 ? multi_kernel<true, false>(lim, local_iters) : multi_kernel<false, false>(lim, local_iters));
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kMultiThreadsX * kMultiThreadsY, 0) !=
            cudaSuccess ||
        per_sm < 1) {
        (void)cudaGetLastError();
        per_sm = 1;
    }
    return per_sm * (nsm > 0 ? nsm : 1);
}

cudaError_t launch_pass_multi(const SweepDesc *descs, const int *counts, int hl, int bf16, int lim, int local_iters,
                              int colour, int nctas, cudaStream_t s) {
    if (nctas <= 0) return cudaSuccess;
    auto k = hl ? (bf16 ? multi_kernel<true, true>(lim, local_iters) : multi_kernel<false, true>(lim, local_iters))
                : (bf16 ? multi_kernel<true, false>(lim, local_iters) : multi_kernel<false, false>(lim, local_iters));
    return launch_pdl(true, k, dim3(nctas), dim3(kMultiThreadsX, kMultiThreadsY, 1), s, descs, counts, colour);
}

int reduction_blocks(const Layout &L) {
    const dim3 g = vox_grid(L);
    const long long n = (long long)g.x * g.y * g.z;
    return (int)(n > 4096 ? n : 4096);
}

cudaError_t launch_fresh_D_into(const Layout &L, Fields &f, const PassParams &p, cudaStream_t s) {
    int ctas;
    const CheckIndex ix = check_index(L, &ctas);
    k_fresh_D_f<<<ctas, kCheckThreads, 0, s>>>(L, ix, f.sp, f.phi, nullptr, f.D, p.lim, (float)p.larsen_n,
                                               (float)p.inv2h, (float)p.floor_);
    return cudaGetLastError();
}

cudaError_t launch_jacobi(Family fam, const Layout &L, const Fields &f, const PassParams &p, int to_second,
                          cudaStream_t s) {
    const dim3 grd = vox_grid(L), blk = vox_block();
    if (fam == FAM_F64) {
        const double *src = to_second ? f.phi64 : f.phi642;
        double *dst = to_second ? f.phi642 : f.phi64;
        k_fresh_D_d<<<grd, blk, 0, s>>>(L, f.sp64, src, f.D64, p.lim, p.larsen_n, p.inv2h, p.floor_);
        k_jacobi<double><<<grd, blk, 0, s>>>(L, f.ah264, f.jh264, src, f.D64, dst, p.omega);
    } else {
        const float *src = to_second ? f.phi : f.phi2;
        float *dst = to_second ? f.phi2 : f.phi;
        int ctas;
        const CheckIndex ix = check_index(L, &ctas);
        k_fresh_D_f<<<ctas, kCheckThreads, 0, s>>>(L, ix, f.sp, src, nullptr, f.D, p.lim, (float)p.larsen_n,
                                                   (float)p.inv2h, (float)p.floor_);
        k_jacobi<float><<<grd, blk, 0, s>>>(L, f.ah2, f.jh2, src, f.D, dst, (float)p.omega);
    }
    return cudaGetLastError();
}

cudaError_t launch_residual(Family fam, const Layout &L, const Fields &f, const PassParams &p, int margin,
                            cudaStream_t s) {
    const dim3 grd = vox_grid(L), blk = vox_block();
    int nblocks = (int)(grd.x * grd.y * grd.z);
    if (nblocks > f.partial_cap) return cudaErrorInvalidValue;
    if (fam == FAM_F64) {
        k_fresh_D_d<<<grd, blk, 0, s>>>(L, f.sp64, f.phi64, f.Df64, p.lim, p.larsen_n, p.inv2h, p.floor_);
        k_residual_d<<<grd, blk, 0, s>>>(L, f.ah264, f.jh264, f.phi64, f.Df64, f.D64, margin, f.partials);
    } else {
        const float *lo = fam == FAM_F32 ? nullptr : f.phlo;
        const CheckIndex ix = check_index(L, &nblocks);
        k_fresh_D_f<<<nblocks, kCheckThreads, 0, s>>>(L, ix, f.sp, f.phi, lo, f.Df, p.lim, (float)p.larsen_n,
                                                      (float)p.inv2h, (float)p.floor_);
        k_residual_f<<<nblocks, kCheckThreads, 0, s>>>(L, ix, f.ah2, f.jh2, f.phi, lo, f.Df, f.D, margin, f.partials);
    }
    k_finalize<<<1, kRedThreads, 0, s>>>(f.partials, nblocks, f.result);
    return cudaGetLastError();
}

cudaError_t launch_sumsq_source(const Layout &L, const Fields &f, cudaStream_t s) {
    const long long n = (long long)L.nx * L.ny * L.nz;
    int nb = (int)((n + 255) / 256);
    if (nb > 1024) nb = 1024;
    if (nb > f.partial_cap) nb = f.partial_cap;
    k_sumsq<<<nb, 256, 0, s>>>(n, f.jsrc, f.partials);
    k_finalize<<<1, kRedThreads, 0, s>>>(f.partials, nb, f.result);
    return cudaGetLastError();
}

cudaError_t launch_validate(long long n, const Fields &f, const float *st, const float *alb, const float *js,
                            cudaStream_t s) {
    int nb = (int)((n + 255) / 256);
    if (nb > 1024) nb = 1024;
    if (nb > f.partial_cap) nb = f.partial_cap;
    if (nb < 1) nb = 1;
    k_validate<<<nb, 256, 0, s>>>(n, st, alb, js, f.partials);
    k_finalize<<<1, kRedThreads, 0, s>>>(f.partials, nb, f.result);
    return cudaGetLastError();
}

cudaError_t launch_bake_scan_negz(const Layout &L, const Fields &f, float h, float radiance, int accumulate,
                                  cudaStream_t s) {
    const dim3 blk(32, 4, 1);
    const dim3 grd((L.nx + 31) / 32, (L.ny + 3) / 4, 1);
    k_bake_scan_negz<<<grd, blk, 0, s>>>(L, f.sigma_t, f.albedo, f.jsrc, h, radiance, accumulate);
    return cudaGetLastError();
}

cudaError_t launch_bake_march(const Layout &L, const Fields &f, double h, const double w[3], const double pos[3],
                              int point, float value, double step, int accumulate, cudaStream_t s) {
    MarchLight m;
    for (int a = 0; a < 3; ++a) {
        m.w[a] = (float)w[a];
    }
    double far = 0.0;            // of the light, in voxels and units of kFarthest
    for (int a = 0; a < 3; ++a) far = fmax(far, fabs(pos[a]) / kFarthest / h);
    for (int a = 0; a < 3; ++a) m.pos[a] = (float)(far > 1.0 ? pos[a] / far / h : pos[a] / h - 0.5);
    m.unit = (float)(far > 1.0 ? h * far : h);
    m.point = point;
    m.value = value;
    m.step = (float)(step / h < 1e30 ? step / h : 1e30);
    m.h = (float)h;
    const int most = L.nx > L.ny ? (L.nx > L.nz ? L.nx : L.nz) : (L.ny > L.nz ? L.ny : L.nz);
    // (no ray is longer than sqrt(3) times the longest edge: up to 2^20 samples counted in float)
    const bool wide = L.nx == 1 || L.ny == 1 || L.nz == 1 || most > kRoundMax || (float)most * 2.0f > 1048576.0f * m.step ||
                      (long long)L.nx * L.ny * L.nz > (1ll << 30);
    (wide ? k_bake_march<true> : k_bake_march<false>)<<<vox_grid(L), vox_block(), 0, s>>>(L, f.sigma_t, f.albedo,
                                                                                         f.jsrc, m, accumulate);
    return cudaGetLastError();
}

}  // namespace fld
