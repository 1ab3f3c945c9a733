// fld_rows.cu -- whole red-black iterations of the smallest grids, one launch
// each (sm_103a).
//
// On a grid of 24^3 to 32^3 a launched colour pass (fld_kernels.cu) is little more
// than the step from one launch to the next and one thread's chain of dependent
// operations.  Here one launch runs a whole iteration of
// Algorithm 1 (Koerner et al. 2014: the red pass, then the black one).  A CTA
// owns TJ x TK rows (full in x).  It copies their state with a halo of two rows into
// shared memory, updates the red unknowns of its rows and of the rows next to
// them (the neighbours its black ones need; the redundant red updates are the
// price of one exchange per iteration instead of two), then the black unknowns of
// its rows, and writes its rows to the other buffer of a ping-pong pair, so no
// CTA reads what another writes in the same launch.  The medium does not
// change: its rows are copied before the launch waits for the preceding one.
// Half of its ~1300 instructions per warp (50^3) find addresses, and larger grids
// repeat ever more red updates, so one pass per launch wins from 40^3 on, and in the
// float-float family everywhere (us per iteration, hi/lo, passes / this: 24^3 3.5 / 2.8,
// 32^3 3.7 / 3.3, 40^3 3.7 / 5.0).
//
// Every update is cell::cell_f32 / cell_fh, the code of the launched passes, so
// the state is theirs bit for bit.  (The bfloat16 medium needs no
// form of its own: sp and ah2 hold its values, exactly.)
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "fld_cell.cuh"
#include "fld_device.cuh"
#include "fld_internal.h"

namespace fld {
namespace {

using namespace cell;

constexpr int kThreads = 512;
constexpr int kFirst = 28;                   // first element copied of a half row (16-byte aligned; unknowns start at 32)
constexpr size_t kPairSmem = 110 * 1024;     // two CTAs per SM: one runs while the next launch's copies its medium
constexpr size_t kMaxSmem = 220 * 1024;

struct RowsArgs {
    Layout L;
    const float *sp, *ah2, *jh2;
    const float *src[3];                     // phi, D, phi lo
    float *dst[3];
    int TJ, TK, tiles_j;
    int P;                                   // elements per row in shared memory
    int R, Rr, Rb;                           // rows: with the halo of 2, red region (halo of 1), own
    int half;                                // unknowns of a colour per row, at most
    Divisor by_chunk, by_R, by_J4, by_M, by_J2, by_J, by_half;
    int ghosts;                              // 1: also write the ghosts next to the own rows
    int lim, rounds;
    float larsen_n, omega, inv2h, floor_;
};

__device__ __forceinline__ void copy16(float *dst, const float *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One unknown of a colour as a thread updates it: where it lies in shared
// memory (o), its medium (md), its element in the grid's fields (q); write: it
// is an unknown of the region; keep: of an own row.
struct Item {
    int o, md, q, par;
    bool write, keep;
};

template <int FAM, int LIM, int ROUNDS>
__global__ void __launch_bounds__(kThreads, 2) k_iter_rows(const RowsArgs a) {
    constexpr int NF = FAM == FAM_F32 ? 2 : 3;
    constexpr int kAhead = 6;                                // state copies a thread has addressed before the wait
    extern __shared__ __align__(16) float sm[];              // state [NF][2][R][P], then medium [3][Rr + Rb][P]
    pdl_launch_dependents();
    const Layout &L = a.L;
    const int tid = threadIdx.x;
    const int tk = blockIdx.x / a.tiles_j, tj = blockIdx.x - tk * a.tiles_j;
    const int J0 = 1 + tj * a.TJ, K0 = 1 + tk * a.TK;        // first own row
    const int J1 = min(L.ny + 1, J0 + a.TJ), K1 = min(L.nz + 1, K0 + a.TK);
    const int chunks = a.P >> 2, M = a.Rr + a.Rb, J2 = a.TJ + 2, J4 = a.TJ + 4;
    const int field = 2 * a.R * a.P;                          // from one field to the next
    const int plane = J4 * a.P;
    float *med = sm + NF * field;

    // medium: the red unknowns of the own rows and the rows next to them, the
    // black ones of the own rows
    for (int i = tid; i < 3 * M * chunks; i += kThreads) {
        const int row = a.by_chunk.quot(i), ch = i - row * chunks;
        const int f = a.by_M.quot(row), m = row - f * M;
        int J, K, c;
        if (m < a.Rr) {
            const int k = a.by_J2.quot(m);
            J = J0 - 1 + (m - k * J2);
            K = K0 - 1 + k;
            c = 0;
        } else {
            const int k = a.by_J.quot(m - a.Rr);
            J = J0 + (m - a.Rr - k * a.TJ);
            K = K0 + k;
            c = 1;
        }
        if (J < 1 || J > L.ny || K < 1 || K > L.nz) continue;
        const float *g = f == 0 ? a.sp : f == 1 ? a.ah2 : a.jh2;
        copy16(med + 4 * i, g + c * L.cs + (K * L.py + J) * L.hpx + kFirst + 4 * ch);
    }
    // state: every row within two of an own one, ghosts included; element of
    // copy i in its field, or -1
    const int copies = NF * 2 * a.R * chunks;
    auto source = [&](int i) {
        const int row = a.by_chunk.quot(i), ch = i - row * chunks;
        const int fc = a.by_R.quot(row), r = row - fc * a.R;
        const int k = a.by_J4.quot(r);
        const int J = J0 - 2 + (r - k * J4), K = K0 - 2 + k;
        if (i >= copies || J < 0 || J > L.ny + 1 || K < 0 || K > L.nz + 1) return -1;
        return (fc & 1) * L.cs + (K * L.py + J) * L.hpx + kFirst + 4 * ch;
    };
    auto copy = [&](int i, int from) {
        const int f1 = 2 * a.R * chunks;
        const float *g = i < f1 ? a.src[0] : NF == 2 || i < 2 * f1 ? a.src[1] : a.src[2];
        if (from >= 0) copy16(sm + 4 * i, g + from);
    };
    auto item = [&](int c, int i) {
        Item it;
        const int m = a.by_half.quot(i), t = i - m * a.half;
        const int k = c == 0 ? (int)a.by_J2.quot(m) : (int)a.by_J.quot(m);
        const int j = m - k * (c == 0 ? J2 : a.TJ);           // row within the region
        const int J = c == 0 ? J0 - 1 + j : J0 + j, K = c == 0 ? K0 - 1 + k : K0 + k;
        it.par = (J + K + 1 + c) & 1;
        const bool inj = J >= J0 && J < J1, ink = K >= K0 && K < K1;
        // (a corner of the red region has no own black unknown next to it)
        it.write = i < (c == 0 ? a.Rr : a.Rb) * a.half && J >= 1 && J <= L.ny && K >= 1 && K <= L.nz && (inj || ink) &&
                   2 * t + 2 - it.par <= L.nx;
        it.keep = it.write && inj && ink;
        it.o = it.write ? ((K - K0 + 2) * J4 + (J - J0 + 2)) * a.P + (kXoff + 1 - kFirst) + t : plane + a.P + 1;
        it.md = it.write ? ((c == 0 ? m : a.Rr + m)) * a.P + (kXoff + 1 - kFirst) + t : 0;
        it.q = c * L.cs + (K * L.py + J) * L.hpx + kXoff + 1 + t;
        return it;
    };
    int from[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) from[u] = source(tid + u * kThreads);
    const int lim = LIM >= 0 ? LIM : a.lim;
    // new values of an unknown (of any address in shared memory: the values of
    // those that are not written are not used)
    auto update = [&](int c, const Item &it, float &pn, float &dn, float &ln) {
        const float *other = sm + (1 - c) * a.R * a.P, *own = sm + c * a.R * a.P;
        const float s_ = med[it.md], ah = med[M * a.P + it.md], jj = med[2 * M * a.P + it.md];
        const int xm = it.o - it.par;                         // x-neighbours at xm, xm + 1
        const int nb[6] = {xm, xm + 1, it.o - a.P, it.o + a.P, it.o - plane, it.o + plane};
        float ps[6], Ds[6], ls[6];
#pragma unroll
        for (int s = 0; s < 6; ++s) {
            ps[s] = other[nb[s]];
            Ds[s] = other[field + nb[s]];
            if (NF == 3) ls[s] = other[2 * field + nb[s]];
        }
        if (FAM == FAM_F32)
            cell_f32<LIM, ROUNDS, true>(own[it.o], ps, Ds, s_, ah, jj, lim, a.larsen_n, a.omega, a.inv2h, a.floor_,
                                        a.rounds, pn, dn);
        else
            cell_fh<LIM, ROUNDS, true>(own[it.o], own[2 * field + it.o], ps, ls, Ds, s_, ah, jj, lim, a.larsen_n,
                                       a.omega, a.inv2h, a.floor_, a.rounds, pn, ln, dn);
    };
    auto store = [&](int c, const Item &it, float pn, float dn, float ln) {
        if (c == 0 && it.write) {
            float *own = sm + it.o;
            own[0] = pn;
            own[field] = dn;
            if (NF == 3) own[2 * field] = ln;
        }
        if (it.keep) {
            a.dst[0][it.q] = pn;
            a.dst[1][it.q] = dn;
            if (NF == 3) a.dst[2][it.q] = ln;
        }
    };
    Item r0 = item(0, tid), r1 = item(0, tid + kThreads), b0 = item(1, tid);

    pdl_wait();
#pragma unroll
    for (int u = 0; u < kAhead; ++u) copy(tid + u * kThreads, from[u]);
    for (int i = tid + kAhead * kThreads; i < copies; i += kThreads) copy(i, source(i));
    copy_wait();
    __syncthreads();

    // two unknowns at a time: their chains of dependent operations overlap
    const int red = a.Rr * a.half, black = a.Rb * a.half;
    for (int i = tid;;) {
        float p0, d0, l0, p1, d1, l1;
        if (i + kThreads < red) {
            update(0, r0, p0, d0, l0);
            update(0, r1, p1, d1, l1);
            store(0, r0, p0, d0, l0);
            store(0, r1, p1, d1, l1);
        } else if (i < red) {
            update(0, r0, p0, d0, l0);
            store(0, r0, p0, d0, l0);
        }
        i += 2 * kThreads;
        if (i >= red) break;
        r0 = item(0, i);
        r1 = item(0, i + kThreads);
    }
    __syncthreads();
    for (int i = tid;;) {
        float p0, d0, l0;
        if (i < black) {
            update(1, b0, p0, d0, l0);
            store(1, b0, p0, d0, l0);
        }
        i += kThreads;
        if (i >= black) break;
        b0 = item(1, i);
    }
    if (a.ghosts) {
        // the ghosts of the own rows, and the ghost rows next to them, as they came
        const int w = (L.nx + 2) / 2 + 1;                      // elements of a half row with its ghosts
        for (int i = tid; i < 2 * a.R * w; i += kThreads) {
            const int row = i / w, p = i - row * w;
            const int c = row >= a.R ? 1 : 0, r = row - c * a.R;
            const int k = a.by_J4.quot(r), J = J0 - 2 + (r - k * J4), K = K0 - 2 + k;
            if (J < J0 - 1 || J > J1 || K < K0 - 1 || K > K1) continue;
            const int par = (J + K + 1 + c) & 1;
            const int I = par ? 2 * p - 1 : 2 * p;
            if (I < 0 || I > L.nx + 1) continue;
            const bool ghost = I == 0 || I == L.nx + 1 || J == 0 || J == L.ny + 1 || K == 0 || K == L.nz + 1;
            if (!ghost) continue;
            const int q = c * L.cs + (K * L.py + J) * L.hpx + kXoff + p;
            const float *s = sm + row * a.P + (kXoff - kFirst) + p;
#pragma unroll
            for (int f = 0; f < NF; ++f) a.dst[f][q] = s[f * field];
        }
    }
}

using RowsKernel = void (*)(const RowsArgs);

template <int FAM>
RowsKernel pick(int lim, int rounds) {
    if (rounds == 2 && lim == LIM_LP) return k_iter_rows<FAM, LIM_LP, 2>;
    return k_iter_rows<FAM, -1, 0>;
}

RowsKernel rows_kernel(Family fam, int lim, int rounds) {
    return fam == FAM_F32 ? pick<FAM_F32>(lim, rounds) : pick<FAM_FH>(lim, rounds);
}

size_t rows_bytes(const Layout &L, int TJ, int TK, int nf) {
    const int P = ((L.nx + 2) / 2 + 4 + 3) / 4 * 4;
    return sizeof(float) * (size_t)P *
           (2 * nf * (TJ + 4) * (TK + 4) + 3 * ((TJ + 2) * (TK + 2) + TJ * TK));
}

}  // namespace

// The tile with the least work on the busiest SM, the time of a launch that
// has no work counted as 2500 updates of one SM (about 1.6 clocks each).
// Empty (TJ = 0) where a halo of two rows around a single one does not fit.
RowsTile rows_tile(const Layout &L, Family fam, int nsm) {
    const int nf = fam == FAM_F32 ? 2 : 3, half = (L.nx + 1) / 2;
    RowsTile best{0, 0};
    double cost = 1e300;
    for (int TJ = 1; TJ <= std::min(L.ny, 16); ++TJ)
        for (int TK = 1; TK <= std::min(L.nz, 16); ++TK) {
            if (rows_bytes(L, TJ, TK, nf) > kMaxSmem) continue;
            const long long ctas = (long long)((L.ny + TJ - 1) / TJ) * ((L.nz + TK - 1) / TK);
            const double rows = TJ * TK * 2 + 2 * (TJ + TK);
            const double c = (double)((ctas + nsm - 1) / nsm) * (rows * half + 2500.0) +
                             (rows_bytes(L, TJ, TK, nf) > kPairSmem ? 800.0 : 0.0);
            if (c < cost) {
                cost = c;
                best = RowsTile{TJ, TK};
            }
        }
    return best;
}

cudaError_t rows_prepare(Family fam, const PassParams &p) {
    return cudaFuncSetAttribute(rows_kernel(fam, p.lim, p.local_iters), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kMaxSmem);
}

cudaError_t launch_rows(Family fam, const Layout &L, const Fields &f, const PassParams &p, const RowsTile &t,
                        const float *const src[3], float *const dst[3], bool first, cudaStream_t s) {
    if (t.TJ < 1 || (fam != FAM_F32 && fam != FAM_FH)) return cudaErrorInvalidValue;
    RowsArgs a;
    a.L = L;
    a.sp = f.sp; a.ah2 = f.ah2; a.jh2 = f.jh2;
    for (int k = 0; k < 3; ++k) {
        a.src[k] = src[k];
        a.dst[k] = dst[k];
    }
    a.TJ = t.TJ; a.TK = t.TK;
    a.tiles_j = (L.ny + t.TJ - 1) / t.TJ;
    a.P = ((L.nx + 2) / 2 + 4 + 3) / 4 * 4;
    a.R = (t.TJ + 4) * (t.TK + 4);
    a.Rr = (t.TJ + 2) * (t.TK + 2);
    a.Rb = t.TJ * t.TK;
    a.half = (L.nx + 1) / 2;
    a.by_chunk.set(a.P / 4);
    a.by_R.set(a.R);
    a.by_J4.set(t.TJ + 4);
    a.by_M.set(a.Rr + a.Rb);
    a.by_J2.set(t.TJ + 2);
    a.by_J.set(t.TJ);
    a.by_half.set(a.half);
    a.ghosts = first ? 1 : 0;
    a.lim = p.lim; a.rounds = p.local_iters;
    a.larsen_n = (float)p.larsen_n; a.omega = (float)p.omega; a.inv2h = (float)p.inv2h; a.floor_ = (float)p.floor_;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.tiles_j * ((L.nz + t.TK - 1) / t.TK)));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = rows_bytes(L, t.TJ, t.TK, fam == FAM_F32 ? 2 : 3);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = first ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, rows_kernel(fam, p.lim, p.local_iters), (const RowsArgs)a);
}

}  // namespace fld
