// ff_pair.cuh -- one pair of bodies in float expansions, two pairs per instruction:
// the pieces that the mixed kicks (kick_ff.cu, kick_tile.cu), the FP64 kick
// (kick_tile.cu) and the energy report (energy.cu) are made of.
#pragma once

#include "ff2.cuh"
#include "kick_sym.cuh"

namespace genga {

// A sum of terms as a double: f64_of_f32_any, but NaN for an infinite or NaN sum (whose
// bits as they stand would read as 2^128 and 1.5 2^128).
__device__ __forceinline__ double ff_sum_f64(float v) {
    const double d = f64_of_f32_any(v);
    return (__float_as_uint(v) & 0x7f800000u) == 0x7f800000u ? __hiloint2double(0x7ff80000, 0) : d;
}

// One coordinate's displacement as two floats.
__device__ __forceinline__ void ff_disp(f2 hj, f2 mj, f2 lj, f2 nhi, f2 nmi, f2 nli, f2 &H, f2 &L) {
    f2 e;
    f2_fast_two_sum(f2_add(hj, nhi), f2_add(mj, nmi), H, e);
    L = f2_add(e, f2_add(lj, nli));
}
// An FP64 displacement times 2^-es as three floats by integer operations: h truncated, l
// and t (|l| < 2^-23 |v|) the other bits.  With v scaled: |v| < 2^-74: l = t = 0, |v| <
// 2^-126 also h = 0; |v| >= 2^100, infinite or NaN: h = NaN.
__device__ __forceinline__ void f64_split3(double v, int es, float &h, float &l, float &t) {
    const unsigned hw = (unsigned)__double2hiint(v), lw = (unsigned)__double2loint(v);
    const unsigned mag = hw & 0x7fffffffu, sgn = hw & 0x80000000u;
    const int e = mag < 0x00100000u ? 0 : (int)(mag >> 20) - es;           // exponent field of the scaled value
    const unsigned top = ((mag - ((unsigned)es << 20) - 0x38000000u) << 3) | (lw >> 29);
    h = __uint_as_float(e >= 1123 ? 0x7fc00000u : e >= 897 ? sgn | top : sgn);
    const unsigned unit = e >= 949 ? sgn | ((unsigned)(e - 948) << 23) : 0u;       // 2^(e - 1075), the last place
    const unsigned unit14 = e >= 949 ? sgn | ((unsigned)(e - 934) << 23) : 0u;
    l = (__uint_as_float(0x4b000000u | (lw >> 14 & 0x7fffu)) - 8388608.0f) * __uint_as_float(unit14);
    t = (__uint_as_float(0x4b000000u | (lw & 0x3fffu)) - 8388608.0f) * __uint_as_float(unit);
}
// The displacements from body i to bodies jx and jy, two floats per component.
__device__ __forceinline__ void ff_disp_f64(const SymArgs &A, int i, int jx, int jy, int es, f2 (&H)[3], f2 (&L)[3]) {
    const double *P[3] = {A.x, A.y, A.z};
#pragma unroll
    for (int c = 0; c < 3; c++) {
        float hx, lx, tx, hy, ly, ty;
        f64_split3(P[c][jx] - P[c][i], es, hx, lx, tx);
        f64_split3(P[c][jy] - P[c][i], es, hy, ly, ty);
        f2_fast_two_sum(f2_make(hx, hy), f2_add(f2_make(lx, ly), f2_make(tx, ty)), H[c], L[c]);
    }
}

// g w as two floats (g = gh + gl, w + wl)
__device__ __forceinline__ void ff_coeff(f2 gh, f2 gl, f2 w, f2 wl, f2 &ch, f2 &cl) {
    ch = f2_mul(gh, w);
    cl = f2_fma(gh, wl, f2_fma(gl, w, f2_fma(gh, w, f2_neg(ch))));
}
// (ch + cl) d as two floats
__device__ __forceinline__ void ff_term(f2 ch, f2 cl, const f2 (&H)[3], const f2 (&L)[3], f2 (&th)[3], f2 (&te)[3]) {
#pragma unroll
    for (int c = 0; c < 3; c++) th[c] = f2_mul(ch, H[c]);
#pragma unroll
    for (int c = 0; c < 3; c++) te[c] = f2_fma(ch, H[c], f2_neg(th[c]));
#pragma unroll
    for (int c = 0; c < 3; c++) te[c] = f2_fma(ch, L[c], te[c]);
#pragma unroll
    for (int c = 0; c < 3; c++) te[c] = f2_fma(cl, H[c], te[c]);
}

// The changeover function at r^2 = s2 + tail, 1/rc_ij = ih + il: r as two floats
// from a fresh seed on the normalised r^2 (a small residual, so that r is good
// to 2^-47), then changeover_ff.
__device__ __forceinline__ void ff_changeover(float s2, float tail, float ih, float il, float &Kh, float &Kl) {
    ff_fast2sum(s2, tail);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(s2));
    y = fmaf(0.5f * y, fmaf(-(s2 * y), y, 1.0f), y);
    const float u = s2 * y, ue = fmaf(s2, y, -u);
    const float e = fmaf(-u, y, 1.0f) - fmaf(tail, y * y, ue * y);
    changeover_ff(u, ue, tail, y, e, ih, il, Kh, Kl);
}

// A pair that the packed coordinates do not give (a body that is not held, or r below
// kFfClose2): FP64 from the positions, K included.  The unit vector d / r as H + L
// and K / r^2 = w + wl: K r^-3 alone would leave the floats' range for a far body.
struct FfOne { float H[3], L[3], w, wl; };
__device__ __forceinline__ void ff_one(const SymArgs &A, int i, int j, float ih, float il, FfOne &o) {
    double d[3] = {0.0, 0.0, 0.0}, w = 0.0;
    if (i < A.n && j < A.n) {                      // not a padding body
        const double xs = scalbn(1.0, -A.ff_header[2]);
        d[0] = (A.x[j] - A.x[i]) * xs; d[1] = (A.y[j] - A.y[i]) * xs; d[2] = (A.z[j] - A.z[i]) * xs;
        const double r2 = fma(d[2], d[2], fma(d[1], d[1], d[0] * d[0])), y = rsqrt(r2);
        w = (r2 < 1e300 ? changeover_fast(r2 * y, (double)ih + (double)il) : 1.0) * (y * y);
        for (int c = 0; c < 3; c++) d[c] *= y;
    }
    for (int c = 0; c < 3; c++) {
        o.H[c] = __double2float_rn(d[c]);
        o.L[c] = __double2float_rn(d[c] - (double)o.H[c]);
    }
    o.w = __double2float_rn(w);
    o.wl = __double2float_rn(w - (double)o.w);
}

// r^2 = s2 + tail (two floats, 2^-48) of a displacement in two floats.
__device__ __forceinline__ void ff_r2(const f2 (&H)[3], const f2 (&L)[3], f2 &s2, f2 &tail) {
    s2 = f2_mul(H[0], H[0]);
    tail = f2_fma(H[0], H[0], f2_neg(s2));
    f2_acc_mul_pos(s2, tail, H[1], H[1]);
    f2_acc_mul_pos(s2, tail, H[2], H[2]);
    tail = f2_fma(f2_dup(2.0f), f2_fma(H[2], L[2], f2_fma(H[1], L[1], f2_mul(H[0], L[0]))), tail);
    f2_fast_two_sum(s2, tail, s2, tail);
}
// r^-3 = w + wl (2^-46) from it.
__device__ __forceinline__ void ff_inv_r3(f2 s2, f2 tail, f2 &w, f2 &wl) {
    const f2 y = f2_rsqrt(s2);
    const f2 u = f2_mul(s2, y), ue = f2_fma(s2, y, f2_neg(u));          // s2 y exactly
    const f2 p = f2_mul(y, y), pe = f2_fma(y, y, f2_neg(p));
    w = f2_mul(p, y);
    const f2 qe = f2_fma(pe, y, f2_fma(p, y, f2_neg(w)));
    const f2 ef = f2_sub(f2_fma(f2_neg(u), y, f2_dup(1.0f)), f2_fma(tail, p, f2_mul(ue, y)));
    wl = f2_fma(w, f2_mul(f2_fma(f2_dup(1.875f), ef, f2_dup(1.5f)), ef), qe);
    f2_fast_two_sum(w, wl, w, wl);
}

// v rounded to a multiple of a power of two g; c = 1.5 2^23 g, |v| < 2^22 g.
__device__ __forceinline__ f2 f2_round(f2 v, f2 c) { return f2_sub(f2_add(v, c), c); }

// A displacement as three floats, exactly: h, m and l are multiples of 2^-23, 2^-47 and
// 2^-71 S below 1, 2^-24 and 2^-48 S, so that each difference fits a float, and e, where
// it is not 0, is a multiple of 2^-47 S and so not below l's.
__device__ __forceinline__ void ff_disp3(f2 hj, f2 mj, f2 lj, f2 nhi, f2 nmi, f2 nli, f2 &H, f2 &L, f2 &T) {
    f2 e;
    f2_fast_two_sum(f2_add(hj, nhi), f2_add(mj, nmi), H, e);
    f2_fast_two_sum(e, f2_add(lj, nli), L, T);
}

// The residual e = 1 - |d y|^2 = eh + el of a displacement d = H + L + T and the
// FP32 seed y ~ 1/|d|, |e| < 2^-20.5, to 2^-56.  q = d y is cut into digits on the
// fixed grids 2^-11, 2^-22 and 2^-34 (|q| <= 1); the sums are of whole multiples
// that fit a float at every step -- 1 - sum Q0^2 (2^-22), - 2 sum Q0 Q1 (2^-32);
// - sum Q1^2 - 2 sum Q0 r0 (2^-44) -- and only the last digits' products round.
__device__ __forceinline__ void ff_residual(const f2 (&H)[3], const f2 (&L)[3], const f2 (&T)[3], f2 y, f2 &eh,
                                            f2 &el) {
    const f2 c0 = f2_dup(6144.0f), c1 = f2_dup(3.0f), c2 = f2_dup(7.32421875e-4f);   // 1.5 2^(23 - 11, - 22, - 34)
    const f2 two = f2_dup(2.0f);
    f2 E0 = f2_dup(1.0f), E1 = 0ull, E2 = 0ull, a1[3], D0[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const f2 q = f2_mul(H[c], y), Q0 = f2_round(q, c0);
        a1[c] = f2_sub(q, Q0);
        E0 = f2_fma(f2_neg(Q0), Q0, E0);
        D0[c] = f2_add(Q0, Q0);
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const f2 q = f2_mul(H[c], y), qe = f2_fma(H[c], y, f2_neg(q));     // H y = q + qe
        const f2 b1 = f2_mul(L[c], y), be = f2_fma(T[c], y, f2_fma(L[c], y, f2_neg(b1)));
        const f2 Q1 = f2_round(a1[c], c1), a2 = f2_sub(a1[c], Q1);
        // a2 + b1 + qe: digit r0 (multiple of 2^-34) and remainder r1
        const f2 t1 = f2_add(c2, a2), t2 = f2_add(t1, b1), t3 = f2_add(t2, qe), r0 = f2_sub(t3, c2);
        f2 r1 = f2_add(f2_sub(a2, f2_sub(t1, c2)), f2_sub(b1, f2_sub(t2, t1)));
        r1 = f2_add(r1, f2_add(f2_sub(qe, f2_sub(t3, t2)), be));
        const f2 r = f2_add(r0, r1);
        E0 = f2_fma(f2_neg(D0[c]), Q1, E0);
        E1 = f2_fma(f2_neg(Q1), Q1, E1);
        E1 = f2_fma(f2_neg(D0[c]), r0, E1);
        E2 = f2_fma(f2_neg(D0[c]), r1, E2);
        E2 = f2_fma(f2_neg(f2_fma(two, Q1, r)), r, E2);
    }
    eh = f2_add(E0, E1);                                                   // exact
    el = E2;
}

// A positive float v + small corrections as a double: v's bits as a double plus a
// whole number of units of 2^(exponent of v - 52), the last place of that double.
// The corrections a_k b_k (b_k scaled by ff_ulp_scale, so that products are in
// units) are summed exactly: t collects multiples of 2^12 units (its bits count
// them above 1.5 2^35), lo what is left.  sum |a_k b_k| < 2^34, lo + u < 2^22.
__device__ __forceinline__ float ff_ulp_scale(float v) {      // 2^(52 - exponent of v), 2^-75 <= v
    return __uint_as_float((306u << 23) - (__float_as_uint(v) & 0x7f800000u));
}
__device__ __forceinline__ void ff_units(f2 a, f2 b, f2 &t, f2 &lo) {
    const f2 m = f2_dup(51539607552.0f);                       // 1.5 2^35
    t = f2_fma(a, b, m);
    lo = f2_fma(a, b, f2_sub(m, t));
}
__device__ __forceinline__ void ff_units_add(f2 a, f2 b, f2 &t, f2 &lo) {
    const f2 s = f2_fma(a, b, t);
    lo = f2_add(lo, f2_fma(a, b, f2_sub(t, s)));
    t = s;
}
__device__ __forceinline__ f2 ff_units_end(f2 lo) { return f2_add(lo, f2_dup(12582912.0f)); }     // 1.5 2^23
// One of the two, times 2^EXP (v not within a few last places of a power of two).
template <int EXP = 0>
__device__ __forceinline__ double ff_add_units(float v, float t, float u) {
    const unsigned b = __float_as_uint(v);
    constexpr unsigned long long K = ((unsigned long long)(0x38000000u + ((unsigned)EXP << 20)) << 32) -
                                     4096ull * 0x51400000ull - 0x4b400000ull;
    return __longlong_as_double((long long)((((unsigned long long)(b >> 3) << 32) | (unsigned)(b << 29)) +
                                            4096ull * __float_as_uint(t) + __float_as_uint(u) + K));
}
// v 2^-896 as a double by its bits alone (v = 0 or a normal float).
__device__ __forceinline__ double ff_bits_down896(float v) {
    const unsigned b = __float_as_uint(v);
    return __hiloint2double((int)((unsigned)((int)b >> 3) & 0x8fffffffu), (int)(b << 29));
}
// within PLACES last places of a power of two (or not a positive normal float)
template <unsigned PLACES>
__device__ __forceinline__ bool ff_near_binade(float v) {
    return ((__float_as_uint(v) + PLACES) & 0x7fffffu) < 2u * PLACES;
}

}  // namespace genga
