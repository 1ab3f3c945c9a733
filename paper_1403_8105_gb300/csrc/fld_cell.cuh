// fld_cell.cuh -- arithmetic of one point update of the single-precision
// sweeps (Algorithm 1 of Koerner et al. 2014: Knudsen number Eq. 35, D by
// Eq. 33 with a Table 2 limiter, local update Eq. 32, SOR blend Eq. 36),
// shared by every kernel that runs these sweeps (launched colour passes,
// temporally blocked passes), so all of them produce the same bits for the
// same inputs.
#pragma once

#include <cuda_runtime.h>

#include "fld_device.cuh"

namespace fld {
namespace cell {

// The hardware's approximate reciprocal (PTX rcp.approx.ftz.f32, one
// special-function-unit instruction, within 1 ulp).  Its operands here are
// floored well above the denormal range (sigma' >= sigma_eps, the Knudsen
// denominators >= eps jbar, the update's denominator > 0), so flushing
// denormals changes nothing.
__device__ __forceinline__ float fast_rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Limiter (Table 2) with approximate reciprocals, for the bulk
// single-precision sweeps, whose accuracy is bounded by phi stored in float;
// the correction sweeps and the residual use the correctly rounded forms.
// The sums below are written with explicit round-to-nearest adds: an
// operand here can be a product (the approximate quotients are x * rcp(y)),
// and a plain `+` could then be contracted into an FMA in one kernel and not
// in another, so kernels sharing this code would differ in the last bit.
__device__ __forceinline__ float limiter_fast(int kind, float larsen_n, float R) {
    switch (kind) {
    case LIM_CDA: return 1.0f / 3.0f;
    case LIM_SUM: return fast_rcp(__fadd_rn(3.0f, R));
    case LIM_MAX: return fast_rcp(fmaxf(3.0f, R));
    case LIM_KERSHAW: return 2.0f * fast_rcp(__fadd_rn(3.0f, hypotf(3.0f, 2.0f * R)));
    case LIM_LARSEN: {
        const float m = fmaxf(3.0f, R), s = fminf(3.0f, R);
        return fast_rcp(m * __powf(__fadd_rn(1.0f, __powf(s * fast_rcp(m), larsen_n)), fast_rcp(larsen_n)));
    }
    default: {
        if (R < 1.0f) return lp_series_f(R);
        const float r = fast_rcp(R);
        // 2e/(1-e), e = exp(-2R), is below 3.4e-8 of (1 - 1/R) once R > 9
        const float tail = R < 9.0f ? 2.0f * fast_rcp(__fsub_rn(__expf(2.0f * R), 1.0f)) : 0.0f;
        return r * __fadd_rn(__fsub_rn(1.0f, r), tail);
    }
    }
}

// limiter_fast without branches for Levermore-Pomraning: both forms, then a
// select (the same bits).  For kernels with few warps per SM, whose threads
// update several unknowns: without branches between them their chains of
// dependent operations overlap.
__device__ __forceinline__ float limiter_fast_sel(int kind, float larsen_n, float R) {
    if (kind != LIM_LP) return limiter_fast(kind, larsen_n, R);
    const float S = lp_series_f(R);
    const float r = fast_rcp(R);
    const float e = 2.0f * fast_rcp(__fsub_rn(__expf(2.0f * R), 1.0f));
    const float tail = R < 9.0f ? e : 0.0f;
    const float G = r * __fadd_rn(__fsub_rn(1.0f, r), tail);
    return R < 1.0f ? S : G;
}

// Arithmetic of one FP32 point update from its gathered values: the
// neighbours' phi and D, its own phi and medium; returns the new phi and D.
template <int LIM, int ROUNDS, bool SEL = false>
__device__ __forceinline__ void cell_f32(float p0, const float ps[6], const float Ds[6], float s_, float ah, float jj,
                                         int lim_rt, float larsen_n, float omega, float inv2h, float floor_,
                                         int rounds_rt, float &phi_new, float &D_new) {
    const int lim = LIM >= 0 ? LIM : lim_rt;
    const int local_iters = ROUNDS > 0 ? ROUNDS : rounds_rt;
    const float gx = ps[1] - ps[0], gy = ps[3] - ps[2], gz = ps[5] - ps[4];
    const float g2 = fmaf(gx, gx, fmaf(gy, gy, gz * gz));
    const float g = g2 > 0.0f ? g2 * rsqrtf(g2) * inv2h : 0.0f;     // |grad phi| (Eq. 34)
    const float gmax = fmaxf(g, floor_);
    const float inv_sp = fast_rcp(s_);
    float A = 0.0f, B = 0.0f, C = 0.0f;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        const float d = ps[s] - p0;
        A += d;
        B = fmaf(Ds[s], d, B);
        C += Ds[s];
    }
    const float base = fmaf(0.5f, B, fmaf(-ah, p0, jj));
    const float den0 = fmaf(0.5f, C, ah);
    float delta = 0.0f, Dp = 0.0f;
#pragma unroll(ROUNDS > 0 ? ROUNDS : 1)
    for (int r = 0; r < (ROUNDS > 0 ? ROUNDS : local_iters); ++r) {
        const float R = gmax * fast_rcp(fmaxf(s_ * __fadd_rn(p0, delta), floor_));     // Eq. 35
        Dp = (SEL ? limiter_fast_sel(lim, larsen_n, R) : limiter_fast(lim, larsen_n, R)) * inv_sp;                          // Eq. 33
        delta = fmaf(0.5f * Dp, A, base) * fast_rcp(fmaf(3.0f, Dp, den0));   // Eq. 32
    }
    phi_new = fmaf(omega, delta, p0);                                          // Eq. 36
    D_new = Dp;
}

// Middle pass: phi kept as a hi/lo pair (no storage floor) but the update
// summed in plain FP32 with the approximate D of the bulk sweeps -- about the
// cost of the FP32 pass, reaching residuals a few times above the
// float-float pass's.  cell_fh is the arithmetic of one point.
template <int LIM, int ROUNDS, bool SEL = false>
__device__ __forceinline__ void cell_fh(float p0, float p0lo, const float ps[6], const float ls[6],
                                        const float Ds[6], float s_, float ah, float jj, int lim_rt, float larsen_n,
                                        float omega, float inv2h, float floor_, int rounds_rt, float &hi_new,
                                        float &lo_new, float &D_new) {
    const int lim = LIM >= 0 ? LIM : lim_rt;
    const int local_iters = ROUNDS > 0 ? ROUNDS : rounds_rt;
    float d[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) d[s] = (ps[s] - p0) + (ls[s] - p0lo);   // phi_s - phi_p
    const float gx = d[1] - d[0], gy = d[3] - d[2], gz = d[5] - d[4];
    const float g2 = fmaf(gx, gx, fmaf(gy, gy, gz * gz));
    const float g = g2 > 0.0f ? g2 * rsqrtf(g2) * inv2h : 0.0f;
    const float gmax = fmaxf(g, floor_);
    const float inv_sp = fast_rcp(s_);
    float A = 0.0f, B = 0.0f, C = 0.0f;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        A += d[s];
        B = fmaf(Ds[s], d[s], B);
        C += Ds[s];
    }
    const float base = fmaf(0.5f, B, fmaf(-ah, p0, fmaf(-ah, p0lo, jj)));
    const float den0 = fmaf(0.5f, C, ah);
    float delta = 0.0f, Dp = 0.0f;
#pragma unroll(ROUNDS > 0 ? ROUNDS : 1)
    for (int r = 0; r < (ROUNDS > 0 ? ROUNDS : local_iters); ++r) {
        const float R = gmax * fast_rcp(fmaxf(s_ * __fadd_rn(p0, delta), floor_));
        Dp = (SEL ? limiter_fast_sel(lim, larsen_n, R) : limiter_fast(lim, larsen_n, R)) * inv_sp;
        delta = fmaf(0.5f * Dp, A, base) * fast_rcp(fmaf(3.0f, Dp, den0));
    }
    const ff nw = ff_add_f(ff{p0, p0lo}, __fmul_rn(omega, delta));
    hi_new = nw.hi;
    lo_new = nw.lo;
    D_new = Dp;
}

// Terms of the residual-form update that do not depend on D_p, for one unknown;
// ff_terms_pair below forms them for two, with the same bits, in the sweeps and in the
// residual kernel, so both evaluate the same discrete equation:  A = sum_s d_s,  B = sum_s D_s d_s,  C = sum_s D_s,
// base = jh2 - ah2 phi_p + B/2, and the central differences.  A and B are
// compensated sums (Ogita-Rump-Oishi style): each difference d_s =
// phi_s - phi_p is formed exactly as a pair (TwoSum of the high words plus
// the low words), each product D_s d_s exactly by TwoProd, and the running
// sums carry their rounding errors in a separate low word.
struct FFTerms {
    ff A, base;
    float C, gx, gy, gz;
};

__device__ __forceinline__ FFTerms ff_terms(float p0, float p0lo, const float ps[6], const float ls[6],
                                            const float Ds[6], float ah, float jj) {
    FFTerms t;
    t.gx = __fadd_rn(__fsub_rn(ps[1], ps[0]), __fsub_rn(ls[1], ls[0]));
    t.gy = __fadd_rn(__fsub_rn(ps[3], ps[2]), __fsub_rn(ls[3], ls[2]));
    t.gz = __fadd_rn(__fsub_rn(ps[5], ps[4]), __fsub_rn(ls[5], ls[4]));
    float Ah = 0.0f, Al = 0.0f, Bh = 0.0f, Bl = 0.0f, C = 0.0f;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        const ff dh = two_sum(ps[s], -p0);                                  // exact high part
        const float dl = __fadd_rn(__fsub_rn(ls[s], p0lo), dh.lo);          // low part
        const ff pr = two_prod(Ds[s], dh.hi);
        const float pe = fmaf(Ds[s], dl, pr.lo);
        if (s == 0) {                          // the sums so far are zero
            Ah = dh.hi; Al = dl;
            Bh = pr.hi; Bl = pe;
            C = Ds[0];
            continue;
        }
        const ff a = two_sum(Ah, dh.hi);
        Ah = a.hi;
        Al = __fadd_rn(Al, __fadd_rn(dl, a.lo));
        const ff b = two_sum(Bh, pr.hi);
        Bh = b.hi;
        Bl = __fadd_rn(Bl, __fadd_rn(pe, b.lo));
        C = __fadd_rn(C, Ds[s]);
    }
    const ff B = fast_two_sum(Bh, Bl);
    ff base = ff_add_f(ff_mul_f(ff{p0, p0lo}, -ah), jj);
    t.base = ff_add(base, ff{0.5f * B.hi, 0.5f * B.lo});
    t.A = fast_two_sum(Ah, Al);
    t.C = C;
    return t;
}

// S(D_p) = base + (D_p / 2) A  and  den(D_p) = ah2 + 3 D_p + C / 2.
__device__ __forceinline__ ff ff_S(const FFTerms &t, float Dp) { return ff_add(t.base, ff_mul_f(t.A, 0.5f * Dp)); }
__device__ __forceinline__ float ff_den(const FFTerms &t, float ah, float Dp) {
    return __fadd_rn(__fadd_rn(ah, 3.0f * Dp), 0.5f * t.C);
}

// One point of the float-float correction pass: phi kept as a hi/lo pair, S
// summed so the update is accurate to the pair's precision; correctly rounded
// D (the same function the residual kernel evaluates).
template <int LIM, int ROUNDS>
__device__ __forceinline__ void cell_ff(float p0, float p0lo, const float ps[6], const float ls[6],
                                        const float Ds[6], float s_, float ah, float jj, int lim_rt, float larsen_n,
                                        float omega, float inv2h, float floor_, int rounds_rt, float &hi_new,
                                        float &lo_new, float &D_new) {
    const int lim = LIM >= 0 ? LIM : lim_rt;
    const int local_iters = ROUNDS > 0 ? ROUNDS : rounds_rt;
    const FFTerms T = ff_terms(p0, p0lo, ps, ls, Ds, ah, jj);
    const DPoint pt = D_point(grad_floor_f(T.gx, T.gy, T.gz, inv2h, floor_), s_);
    float delta = 0.0f, Dp = 0.0f;
#pragma unroll(ROUNDS > 0 ? ROUNDS : 1)
    for (int r = 0; r < (ROUNDS > 0 ? ROUNDS : local_iters); ++r) {
        Dp = D_of_f(pt, __fadd_rn(p0, delta), floor_, lim, larsen_n);
        const ff S = ff_S(T, Dp);
        // delta is a correction: its rounding does not move the fixed point
        delta = __fdividef(__fadd_rn(S.hi, S.lo), ff_den(T, ah, Dp));
    }
    const ff nw = ff_add_f(ff{p0, p0lo}, __fmul_rn(omega, delta));
    hi_new = nw.hi;
    lo_new = nw.lo;
    D_new = Dp;
}

// ---------------------------------------------------------------------------
// cell_ff of two unknowns, one in each half of packed FP32 instructions (add /
// fma .f32x2).  The correction pass is bound by issue: 592 instructions per
// update, 390 of them on the FMA pipe.  A packed instruction keeps that pipe
// busy as long as the two it replaces (measured 63 against 126 per clock and
// SM) but takes one issue slot.  Each half rounds like the scalar instruction
// and every sum keeps its operands and order, so both unknowns get cell_ff's bits.
//
// Two rules keep it so.  The assembler contracts a packed product followed by a packed
// sum into an FMA even with explicit rounding, so products are FMAs with +0
// (mul2), which it leaves alone.  And a difference is an FMA with -1 (sub2): the
// product is exact.  Negated quantities (n...) save the sign changes.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long pack2(float2 a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(v));
    return a;
}
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)), "l"(pack2(c)));
    return unpack2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return fma2(a, b, both(0.0f)); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, both(-1.0f), a); }

struct ff2 {
    float2 hi, lo;
};
__device__ __forceinline__ ff2 two_sum2(float2 a, float2 b) {
    const float2 s = add2(a, b);
    const float2 bb = sub2(s, a);
    return {s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ ff2 fast_two_sum2(float2 a, float2 b) {
    const float2 s = add2(a, b);
    return {s, sub2(b, sub2(s, a))};
}

// FFTerms and S of two unknowns.
struct FFTerms2 {
    ff2 base;
    float2 A, nA, nAlo, C;       // A.hi, and both words of A negated
};

// |grad phi|, floored (grad_floor_f of ff_terms' differences).  Without LO the low
// words are zero, here and below.
template <bool LO = true>
__device__ __forceinline__ float2 grad_pair(const float2 ps[6], const float2 ls[6], float inv2h, float floor_) {
    const float2 dx = sub2(ps[1], ps[0]), dy = sub2(ps[3], ps[2]), dz = sub2(ps[5], ps[4]);
    const float2 gx = mul2(LO ? add2(dx, sub2(ls[1], ls[0])) : dx, both(inv2h));
    const float2 gy = mul2(LO ? add2(dy, sub2(ls[3], ls[2])) : dy, both(inv2h));
    const float2 gz = mul2(LO ? add2(dz, sub2(ls[5], ls[4])) : dz, both(inv2h));
    const float2 g2 = fma2(gx, gx, fma2(gy, gy, mul2(gz, gz)));
    return make_float2(fmaxf(sqrtf(g2.x), floor_), fmaxf(sqrtf(g2.y), floor_));
}

template <bool LO = true>
__device__ __forceinline__ FFTerms2 ff_terms_pair(float2 p0, float2 p0lo, const float2 ps[6], const float2 ls[6],
                                                  const float2 Ds[6], float2 ah, float2 jj) {
    FFTerms2 T;
    // A = sum d_s, B = sum D_s d_s (its low word negated), C = sum D_s
    const float2 np0 = neg2(p0), half = both(0.5f);
    float2 Ah, Al, Bh, nBl;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        const ff2 dh = two_sum2(ps[s], np0);
        const float2 dl = LO ? add2(sub2(ls[s], p0lo), dh.lo) : dh.lo;
        const float2 nD = neg2(Ds[s]);
        const float2 p = mul2(Ds[s], dh.hi);
        const float2 npe = fma2(nD, dl, fma2(nD, dh.hi, p));
        if (s == 0) {
            Ah = dh.hi; Al = dl;
            Bh = p; nBl = npe;
            T.C = Ds[0];
            continue;
        }
        const ff2 a = two_sum2(Ah, dh.hi);
        Ah = a.hi;
        Al = add2(Al, add2(dl, a.lo));
        const ff2 b = two_sum2(Bh, p);
        Bh = b.hi;
        nBl = add2(nBl, sub2(npe, b.lo));
        T.C = add2(T.C, Ds[s]);
    }
    const float2 B = sub2(Bh, nBl);
    const float2 nBlo = add2(nBl, sub2(B, Bh));
    // base = j h^2 - sigma_a' h^2 phi + B / 2
    const float2 P = mul2(p0, ah);
    const float2 pl = fma2(np0, ah, P);
    const float2 e = LO ? fma2(neg2(p0lo), ah, pl) : pl;
    const float2 mh = sub2(e, P);
    const float2 ml = sub2(e, add2(mh, P));
    const ff2 t = two_sum2(mh, jj);
    const ff2 u = fast_two_sum2(t.hi, add2(t.lo, ml));
    const ff2 v = two_sum2(u.hi, mul2(B, half));
    T.base = fast_two_sum2(v.hi, add2(v.lo, sub2(u.lo, mul2(nBlo, half))));
    const ff2 A = fast_two_sum2(Ah, Al);
    T.A = A.hi;
    T.nA = neg2(A.hi);
    T.nAlo = neg2(A.lo);
    return T;
}

__device__ __forceinline__ ff2 ff_S_pair(const FFTerms2 &T, float2 Dp) {
    const float2 hd = mul2(Dp, both(0.5f));
    const float2 p = mul2(T.A, hd);
    const float2 ne = fma2(T.nAlo, hd, fma2(T.nA, hd, p));
    const float2 m = sub2(p, ne);
    const float2 nml = add2(ne, sub2(m, p));
    const ff2 t = two_sum2(T.base.hi, m);
    return fast_two_sum2(t.hi, add2(t.lo, sub2(T.base.lo, nml)));
}

template <int LIM, int ROUNDS>
__device__ __forceinline__ void cell_ff_pair(float2 p0, float2 p0lo, const float2 ps[6], const float2 ls[6],
                                             const float2 Ds[6], float2 s_, float2 ah, float2 jj, int lim_rt,
                                             float larsen_n, float omega, float inv2h, float floor_, int rounds_rt,
                                             float2 &hi_new, float2 &lo_new, float2 &D_new) {
    const int lim = LIM >= 0 ? LIM : lim_rt;
    const int local_iters = ROUNDS > 0 ? ROUNDS : rounds_rt;
    const float2 gmax = grad_pair(ps, ls, inv2h, floor_);
    const DPoint ptx = D_point(gmax.x, s_.x), pty = D_point(gmax.y, s_.y);
    const FFTerms2 T = ff_terms_pair(p0, p0lo, ps, ls, Ds, ah, jj);
    const float2 hC = mul2(T.C, both(0.5f));
    float2 delta = both(0.0f), Dp = both(0.0f);
#pragma unroll(ROUNDS > 0 ? ROUNDS : 1)
    for (int r = 0; r < (ROUNDS > 0 ? ROUNDS : local_iters); ++r) {
        Dp.x = D_of_f(ptx, __fadd_rn(p0.x, delta.x), floor_, lim, larsen_n);
        Dp.y = D_of_f(pty, __fadd_rn(p0.y, delta.y), floor_, lim, larsen_n);
        const ff2 S = ff_S_pair(T, Dp);
        const float2 num = add2(S.hi, S.lo);
        const float2 den = add2(add2(ah, mul2(Dp, both(3.0f))), hC);
        delta = make_float2(__fdividef(num.x, den.x), __fdividef(num.y, den.y));
    }
    const ff2 t = two_sum2(p0, mul2(both(omega), delta));
    const ff2 nw = fast_two_sum2(t.hi, add2(t.lo, p0lo));
    hi_new = nw.hi;
    lo_new = nw.lo;
    D_new = Dp;
}

// Programmatic dependent launch (PTX griddepcontrol): a pass lets the next
// grid in its stream be scheduled as soon as all of its own CTAs are running,
// and waits for the preceding grid to complete (with its writes visible)
// before it reads phi, phi_lo or D.  The medium (sigma', sigma_a' h^2, j h^2)
// is written only by earlier, fully completed kernels and is loaded before
// the wait.  Without the launch attribute both instructions are no-ops.
__device__ __forceinline__ void pdl_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace cell
}  // namespace fld
