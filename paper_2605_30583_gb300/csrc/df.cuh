// Double-float ("df") arithmetic: a value is the unevaluated sum hi + lo of two FP32
// numbers with |lo| <= ulp(hi) / 2, about 48 significant bits, from FP32 operations only
// (Dekker, "A floating-point technique for extending the available precision", 1971;
// Knuth's TwoSum; the exact product by FMA).  On this GPU FP64 runs at 1/64 of the FP32
// rate, so the one quantity of the mixed form that needs more than FP32 -- the
// reprojection residual f s p - u, whose ~500 px terms cancel to ~1 px -- is computed
// this way.  The error-free transformations use the _rn intrinsics so the compiler
// neither contracts nor reassociates them.
#pragma once

#include <cuda_runtime.h>

#include "device_common.cuh"

namespace gbba {

struct DF {
    float hi, lo;
};

__device__ __forceinline__ DF df_from(float a) { return {a, 0.0f}; }

// hi + lo of a double, rounded twice (conversions on the integer units: narrow, widen).
__device__ __forceinline__ DF df_from_double(double a) {
    const float hi = narrow(a);
    return {hi, narrow(a - widen(hi))};
}

__device__ __forceinline__ float df_to_float(DF a) { return __fadd_rn(a.hi, a.lo); }

// s + e = a + b exactly (Knuth's TwoSum, no condition on the operands).
__device__ __forceinline__ DF two_sum_f(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}

// s + e = a + b exactly when |a| >= |b| (or a = 0).
__device__ __forceinline__ DF fast_two_sum_f(float a, float b) {
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// a b as the exact product of the high parts (fma gives its error) plus the cross terms; not
// renormalised: |lo| may reach a few ulp of hi, which the sums and products below take.
__device__ __forceinline__ DF df_mul(DF a, DF b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    return {p, __fmaf_rn(a.lo, b.hi, e)};
}

// a + b: the high parts' sum and its error exactly, the low parts added (not renormalised).
__device__ __forceinline__ DF df_add(DF a, DF b) {
    const DF s = two_sum_f(a.hi, b.hi);
    return {s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo))};
}

__device__ __forceinline__ DF df_add_f(DF a, float b) {
    const DF s = two_sum_f(a.hi, b);
    return {s.hi, __fadd_rn(s.lo, a.lo)};
}

__device__ __forceinline__ DF df_norm(DF a) { return fast_two_sum_f(a.hi, a.lo); }

__device__ __forceinline__ DF df_square(DF a) {
    const float p = __fmul_rn(a.hi, a.hi);
    return {p, __fmaf_rn(__fadd_rn(a.hi, a.hi), a.lo, __fmaf_rn(a.hi, a.hi, -p))};
}

// acc + a b for the row products of a rotation: as df_mul and df_add, the low parts gathered.
__device__ __forceinline__ DF df_mul_add(DF a, DF b, DF acc) {
    const float p = __fmul_rn(a.hi, b.hi);
    const DF s = two_sum_f(acc.hi, p);
    float e = __fadd_rn(__fmaf_rn(a.hi, b.hi, -p), __fadd_rn(acc.lo, s.lo));
    e = __fmaf_rn(a.hi, b.lo, e);
    return {s.hi, __fmaf_rn(a.lo, b.hi, e)};
}

// 1 / b: the FP32 reciprocal approximation x of b.hi, then x + x (e + e^2) with
// e = 1 - b x (fma: exact to 2^-48, |e| < 2^-22).
__device__ __forceinline__ DF df_rcp(DF b) {
    const float x = rcp_approx(b.hi);
    const float e = __fmaf_rn(-b.lo, x, __fmaf_rn(-b.hi, x, 1.0f));
    const float xe = __fmul_rn(x, e);
    return {x, __fmaf_rn(xe, e, xe)};
}

// Camera of a df residual: FP32 record plus its low-order record.
struct CamDF {
    DF R[9], t[3], f, k1, k2;
};

__device__ __forceinline__ CamDF load_cam_df(const float* __restrict__ rec, const float* __restrict__ lo) {
    const float4* r4 = reinterpret_cast<const float4*>(rec);
    const float4* l4 = reinterpret_cast<const float4*>(lo);
    float h[16], l[16];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 a = __ldg(r4 + k), b = __ldg(l4 + k);
        h[4 * k] = a.x; h[4 * k + 1] = a.y; h[4 * k + 2] = a.z; h[4 * k + 3] = a.w;
        l[4 * k] = b.x; l[4 * k + 1] = b.y; l[4 * k + 2] = b.z; l[4 * k + 3] = b.w;
    }
    CamDF c;
#pragma unroll
    for (int i = 0; i < 9; ++i) c.R[i] = {h[CP_R + i], l[CP_R + i]};
#pragma unroll
    for (int i = 0; i < 3; ++i) c.t[i] = {h[CP_T + i], l[CP_T + i]};
    c.f = {h[CP_F], l[CP_F]};
    c.k1 = {h[CP_K1], l[CP_K1]};
    c.k2 = {h[CP_K2], l[CP_K2]};
    return c;
}

// The Snavely residual of Sec. VI-A in df arithmetic: P = R X + t, d = P.z -+ eps
// (d_safe), p = -P.xy / d, s = 1 + k1 |p|^2 + k2 |p|^4, r = f s p - u.  Its error is a
// few units of 2^-46 of the ~500 px terms, so rounded to FP32 it is the exact residual
// to within an ulp of itself.  Low parts are gathered and renormalised only where a
// cancellation (R X + t, f s p - u) or a division follows: 210 FP32 operations, where
// renormalising every sum and product took 305
// (28.8M residuals: 475 -> 381 us).
__device__ __forceinline__ void residual_df(const CamDF& c, const DF (&X)[3], float eps, float u0, float u1,
                                            DF& r0, DF& r1) {
    DF P[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        DF a = df_mul(c.R[3 * i], X[0]);
        a = df_mul_add(c.R[3 * i + 1], X[1], a);
        a = df_mul_add(c.R[3 * i + 2], X[2], a);
        P[i] = df_norm(df_add(a, c.t[i]));
    }
    DF d = P[2];
    if (eps != 0.0f) d = df_norm(df_add_f(d, P[2].hi >= 0.0f ? eps : -eps));
    const DF iz = df_rcp(d);
    const DF q0 = df_norm(df_mul(P[0], iz)), q1 = df_norm(df_mul(P[1], iz));   // -p
    const DF n2 = df_add(df_square(q0), df_square(q1));
    const DF s = df_norm(df_add_f(df_mul(n2, df_add(c.k1, df_mul(c.k2, n2))), 1.0f));
    const DF fs = df_mul(c.f, s);
    // r = -(f s q + u)
    const DF a0 = df_norm(df_add_f(df_mul(fs, q0), u0)), a1 = df_norm(df_add_f(df_mul(fs, q1), u1));
    r0 = {-a0.hi, -a0.lo};
    r1 = {-a1.hi, -a1.lo};
}

}  // namespace gbba
