// Double-float ("df") arithmetic: a value is the unevaluated sum hi + lo of two FP32
// numbers with |lo| <= ulp(hi) / 2 (results of the _raw operations excepted), about 48
// significant bits, from FP32 operations only
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

// The operations ending in _raw leave out the last renormalisation: |lo| may reach a few ulp of
// hi, which the operations that take the result allow for; df_norm makes up for it.
__device__ __forceinline__ DF df_norm(DF a) { return fast_two_sum_f(a.hi, a.lo); }

// a b as the exact product of the high parts (fma gives its error) plus the cross terms.
__device__ __forceinline__ DF df_mul_raw(DF a, DF b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    return {p, __fmaf_rn(a.lo, b.hi, e)};
}

__device__ __forceinline__ DF df_mul(DF a, DF b) { return df_norm(df_mul_raw(a, b)); }

// a + b: the high parts' sum and its error exactly, the low parts added.
__device__ __forceinline__ DF df_add_raw(DF a, DF b) {
    const DF s = two_sum_f(a.hi, b.hi);
    return {s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo))};
}

__device__ __forceinline__ DF df_add(DF a, DF b) { return df_norm(df_add_raw(a, b)); }

__device__ __forceinline__ DF df_add_f(DF a, float b) {
    const DF s = two_sum_f(a.hi, b);
    return df_norm({s.hi, __fadd_rn(s.lo, a.lo)});
}

__device__ __forceinline__ DF df_square_raw(DF a) {
    const float p = __fmul_rn(a.hi, a.hi);
    return {p, __fmaf_rn(__fadd_rn(a.hi, a.hi), a.lo, __fmaf_rn(a.hi, a.hi, -p))};
}

// 1 / b: the FP32 reciprocal x of b.hi, then x + x (e + e^2) with e = 1 - b x
// (fma: exact to 2^-48, |e| < 2^-23).
__device__ __forceinline__ DF df_rcp_raw(DF b) {
    const float x = __frcp_rn(b.hi);
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
// few units of 2^-48 of the ~500 px terms, so rounded to FP32 it is the exact residual
// to within an ulp of itself.  R X + t, where the terms cancel, is renormalised after every
// product and sum; the polynomial of the distortion, whose terms do not, only where a product
// with p or a cancellation follows.  28.8M residuals: 475 us with every operation renormalised,
// 437 us so, with no larger an error (200 cameras: 3.26e-13 px rms against 3.28e-13; R X + t of
// 65-unit coordinates: 7.8e-12 against 7.7e-12); with R X + t left raw as well 381 us, but
// 3.7e-13 and 9.3e-12.
__device__ __forceinline__ void residual_df(const CamDF& c, const DF (&X)[3], float eps, float u0, float u1,
                                            DF& r0, DF& r1) {
    DF P[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        DF a = df_mul(c.R[3 * i], X[0]);
        a = df_add(a, df_mul(c.R[3 * i + 1], X[1]));
        a = df_add(a, df_mul(c.R[3 * i + 2], X[2]));
        P[i] = df_add(a, c.t[i]);
    }
    DF d = P[2];
    if (eps != 0.0f) d = df_add_f(d, P[2].hi >= 0.0f ? eps : -eps);
    const DF iz = df_rcp_raw(d);
    const DF q0 = df_mul(P[0], iz), q1 = df_mul(P[1], iz);   // -p
    const DF n2 = df_add_raw(df_square_raw(q0), df_square_raw(q1));
    const DF s = df_add_f(df_mul_raw(n2, df_add_raw(c.k1, df_mul_raw(c.k2, n2))), 1.0f);
    const DF fs = df_mul(c.f, s);
    // r = -(f s q + u)
    const DF a0 = df_add_f(df_mul_raw(fs, q0), u0), a1 = df_add_f(df_mul_raw(fs, q1), u1);
    r0 = {-a0.hi, -a0.lo};
    r1 = {-a1.hi, -a1.lo};
}

}  // namespace gbba
