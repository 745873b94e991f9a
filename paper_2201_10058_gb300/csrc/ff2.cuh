// ff2.cuh -- packed pairs of floats (the sm_100+ f32x2 instructions) and the
// float expansions of the mixed pair kicks.
//
// GB300 executes 128 FP32 lanes per clock and SM against 1.7-1.8 FP64 ones, and
// an f32x2 instruction does two lanes' work in one issue slot (2 cycles of the
// pipe; measured).  The kicks therefore carry coordinates, terms and sums as
// unevaluated sums of floats and process two pairs per instruction; the other
// half of the issue slots is left for the integer, shared-memory and shuffle
// work.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace genga {

typedef unsigned long long f2;     // two floats, x in the low word

__device__ __forceinline__ f2 f2_make(float x, float y) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ float2 f2_get(f2 p) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(p));
    return r;
}
__device__ __forceinline__ f2 f2_dup(float v) { return f2_make(v, v); }
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 f2_neg(f2 a) {       // folded into the consumer
    const float2 v = f2_get(a);
    return f2_make(-v.x, -v.y);
}
__device__ __forceinline__ f2 f2_shfl(f2 a, int src) {
    const float2 v = f2_get(a);
    return f2_make(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ f2 f2_select(bool px, bool py, f2 a, f2 b) {
    const float2 u = f2_get(a), v = f2_get(b);
    return f2_make(px ? u.x : v.x, py ? u.y : v.y);
}
__device__ __forceinline__ f2 f2_rsqrt(f2 a) {
    float2 v = f2_get(a);
    asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(v.x));
    asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(v.y));
    return f2_make(v.x, v.y);
}
// s + e = a + b exactly for |a| >= |b| (or a = 0).
__device__ __forceinline__ void f2_fast_two_sum(f2 a, f2 b, f2 &s, f2 &e) {
    s = f2_add(a, b);
    e = f2_sub(b, f2_sub(s, a));
}
__device__ __forceinline__ void f2_two_sum(f2 a, f2 b, f2 &s, f2 &e) {
    s = f2_add(a, b);
    const f2 bb = f2_sub(s, a);
    e = f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb));
}
// (hi, lo) += h + l resp. -= h + l, l of the order of h's last place.
__device__ __forceinline__ void f2_acc(f2 &hi, f2 &lo, f2 h, f2 l) {
    f2 e;
    f2_two_sum(hi, h, hi, e);
    lo = f2_add(lo, f2_add(l, e));
}
__device__ __forceinline__ void f2_acc_neg(f2 &hi, f2 &lo, f2 h, f2 l) {
    const f2 s = f2_sub(hi, h), bb = f2_sub(s, hi);
    lo = f2_add(lo, f2_sub(f2_sub(f2_sub(hi, f2_sub(s, bb)), f2_add(h, bb)), l));
    hi = s;
}
// (hi, lo) += a b for hi >= 0, a b >= 0: TwoSum of hi and the unrounded product
// by FMA, its error (the product's low part included) into lo.  (With terms of
// either sign the sum could end below hi's last place, where s - hi rounds.)
__device__ __forceinline__ void f2_acc_mul_pos(f2 &hi, f2 &lo, f2 a, f2 b) {
    const f2 s = f2_fma(a, b, hi), z = f2_sub(s, hi);
    lo = f2_add(lo, f2_add(f2_sub(hi, f2_sub(s, z)), f2_fma(a, b, f2_neg(z))));
    hi = s;
}

}  // namespace genga
