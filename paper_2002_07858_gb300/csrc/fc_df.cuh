// fc_df.cuh -- double-float arithmetic (a value is hi + lo, two binary32
// numbers with |lo| <= ulp(hi)/2) for the binary64-accuracy residual chi2 of
// the mixed path.  GB300 runs binary32 about 60 times faster than binary64,
// and a double-float multiply-add costs about a dozen binary32 operations:
//   - the product of two binary32 numbers is split exactly by one fma
//     (Dekker's TwoProduct with a fused multiply-add);
//   - sums use Knuth's TwoSum (six operations, exact error term);
//   - the lo * lo cross term is dropped (below 2^-48 relative).
// The relative error of a dot product of n terms is about n 2^-47 of the sum
// of the absolute terms, far below what the certified decisions and the
// output tolerances need.  Every function here is a fixed sequence of IEEE
// binary32 operations, so a value is the same bits wherever it is computed.
#pragma once

#include <cuda_runtime.h>

namespace fcdev {

// binary64 -> hi + lo (exact for |x| within the binary32 range up to 2^-48 |x|)
__device__ __forceinline__ float2 df_from(double x) {
    const float h = (float)x;
    const float l = (float)(x - (double)h);
    return make_float2(h, l);
}

__device__ __forceinline__ double df_to(float2 a) { return (double)a.x + (double)a.y; }

// s + e = a + b exactly (Knuth)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// renormalise hi + lo (requires |hi| >= |lo| or hi == 0)
__device__ __forceinline__ float2 df_norm(float hi, float lo) {
    const float s = __fadd_rn(hi, lo);
    return make_float2(s, __fsub_rn(lo, __fsub_rn(s, hi)));
}

// acc + a * b, a and b double-float
__device__ __forceinline__ float2 df_fma(float2 acc, float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);
    float e = __fmaf_rn(a.x, b.x, -p);
    e = __fmaf_rn(a.x, b.y, e);
    e = __fmaf_rn(a.y, b.x, e);
    float s, err;
    two_sum(acc.x, p, s, err);
    return make_float2(s, __fadd_rn(acc.y, __fadd_rn(err, e)));
}

// a + b, both double-float
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
    float s, e;
    two_sum(a.x, b.x, s, e);
    return df_norm(s, __fadd_rn(e, __fadd_rn(a.y, b.y)));
}

// a - b for a double-float a and a binary32 b (exact up to the lo rounding)
__device__ __forceinline__ float2 df_sub_f(float2 a, float b) {
    float s, e;
    two_sum(a.x, -b, s, e);
    return df_norm(s, __fadd_rn(e, a.y));
}

// ---- two double-floats side by side ----
// Two independent values packed as (hi0, hi1), (lo0, lo1) in 64-bit register
// pairs, worked by the packed binary32 instructions (f32x2): one issue slot
// does both, and each half is the IEEE operation of the scalar form, so every
// value has the bits df_fma / df_norm / df_add give it.
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 x2_add(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 x2_sub(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 x2_mul(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 x2_fma(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 x2_neg(f32x2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f32x2 x2_pack(float a, float b) {
    return (f32x2)__float_as_uint(a) | ((f32x2)__float_as_uint(b) << 32);
}
__device__ __forceinline__ float x2_lo(f32x2 a) { return __uint_as_float((uint32_t)a); }
__device__ __forceinline__ float x2_hi(f32x2 a) { return __uint_as_float((uint32_t)(a >> 32)); }

struct df2x {
    f32x2 x, y;  // (hi0, hi1), (lo0, lo1)
};

// acc + a * b (df_fma in both halves)
__device__ __forceinline__ df2x df2_fma(df2x acc, f32x2 ax, f32x2 ay, f32x2 bx, f32x2 by) {
    const f32x2 p = x2_mul(ax, bx);
    f32x2 e = x2_fma(ax, bx, x2_neg(p));
    e = x2_fma(ax, by, e);
    e = x2_fma(ay, bx, e);
    const f32x2 s = x2_add(acc.x, p);
    const f32x2 bb = x2_sub(s, acc.x);
    const f32x2 err = x2_add(x2_sub(acc.x, x2_sub(s, bb)), x2_sub(p, bb));
    return df2x{s, x2_add(acc.y, x2_add(err, e))};
}

__device__ __forceinline__ df2x df2_norm(df2x a) {
    const f32x2 s = x2_add(a.x, a.y);
    return df2x{s, x2_sub(a.y, x2_sub(s, a.x))};
}

// a + b (df_add in both halves)
__device__ __forceinline__ df2x df2_add(df2x a, df2x b) {
    const f32x2 s = x2_add(a.x, b.x);
    const f32x2 bb = x2_sub(s, a.x);
    const f32x2 e = x2_add(x2_sub(a.x, x2_sub(s, bb)), x2_sub(b.x, bb));
    return df2_norm(df2x{s, x2_add(e, x2_add(a.y, b.y))});
}

}  // namespace fcdev
