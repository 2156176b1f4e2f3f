// Per-observation building blocks of the mixed-precision normal operator, shared by
// the multi-kernel path and the persistent PCG kernel.
#pragma once

#include "device_common.cuh"

namespace gbba {

constexpr uint32_t FULL = 0xffffffffu;
constexpr uint32_t NO_CAM = 0xffffffffu;

// Warp-segmented suffix sum: lanes with equal `key` in consecutive positions form a
// segment; afterwards the first lane of each segment holds the segment's sum.
template <int V>
__device__ __forceinline__ bool seg_reduce(uint32_t key, float (&acc)[V]) {
    const int lane = threadIdx.x & 31;
    const uint32_t prev = __shfl_up_sync(FULL, key, 1);
    const bool head = (lane == 0) || (prev != key);
    const uint32_t hm = __ballot_sync(FULL, head);
    const uint32_t after = hm & ~((2u << lane) - 1u);
    const int end = after ? (__ffs(after) - 1) : 32;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const float o = __shfl_down_sync(FULL, acc[k], d);
            if (lane + d < end) acc[k] += o;
        }
    }
    return head;
}

// Warp sum of N per-lane values by recursive halving: at each of the five levels the two
// lanes of a pair (lane, lane ^ o) split the values they still carry, each keeping one
// half and adding the partner's copy of it (about 4 N + 10 instructions, where a
// butterfly of every value takes 10 N).  Every lane ends with split_sum_slots(N) values;
// the first `returned` of them are complete sums, v[k] of value idx + k, and together
// the lanes hold each of the N sums exactly once.
__host__ __device__ constexpr int split_sum_slots(int n) {
    return ((((((n + 1) / 2 + 1) / 2 + 1) / 2 + 1) / 2) + 1) / 2;
}

template <int N>
__device__ __forceinline__ int warp_split_sum(float (&v)[N], int lane, int& idx) {
    int m = N;    // values every lane carries (the same in all lanes)
    int rc = N;   // of which real (the rest pad the upper halves of odd splits)
    idx = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int h = (m + 1) / 2;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < (N + 1) / 2; ++k) {
            if (k < h) {
                const float hi = (k + h < m) ? v[k + h] : 0.0f;
                const float send = up ? v[k] : hi;
                const float keep = up ? hi : v[k];
                v[k] = keep + __shfl_xor_sync(FULL, send, o);
            }
        }
        if (up) {
            idx += h;
            rc = rc > h ? rc - h : 0;
        } else {
            rc = rc < h ? rc : h;
        }
        m = h;
    }
    return rc;
}

// A thread's finished camera sums (op_finish) into the global accumulators, then cleared.
__device__ __forceinline__ void flush_matvec(float* __restrict__ dst, float (&a)[9]) {
    atomicAdd(reinterpret_cast<float4*>(dst), make_float4(a[0], a[1], a[2], a[3]));
    atomicAdd(reinterpret_cast<float4*>(dst + 4), make_float4(a[4], a[5], a[6], a[7]));
    atomicAdd(dst + 8, a[8]);
#pragma unroll
    for (int k = 0; k < 9; ++k) a[k] = 0.0f;
}

__device__ __forceinline__ void load_dir(const float* __restrict__ rec, float (&d)[9]) {
    const float4* r4 = reinterpret_cast<const float4*>(rec);
    const float4 a = __ldg(r4), b = __ldg(r4 + 1), c = __ldg(r4 + 2);
    d[0] = a.x; d[1] = a.y; d[2] = a.z; d[3] = a.w;
    d[4] = b.x; d[5] = b.y; d[6] = b.z; d[7] = b.w; d[8] = c.x;
}

// t = J d for one observation: J d = A (phi x RX + d_t + R d_X) + c_i p with
// phi = J_l d_w (precomputed per camera) and c_i = s d_f + f n2 d_k1 + f n2^2 d_k2.
__device__ __forceinline__ void jdir(const Geo& g, const Cam& c, const float (&dir)[9],
                                     float dX0, float dX1, float dX2, float& t0, float& t1) {
    const float* phi = dir + CD_PHI;
    float dP0 = fmaf(phi[1], g.RX[2], -phi[2] * g.RX[1]) + dir[CD_T + 0];
    float dP1 = fmaf(phi[2], g.RX[0], -phi[0] * g.RX[2]) + dir[CD_T + 1];
    float dP2 = fmaf(phi[0], g.RX[1], -phi[1] * g.RX[0]) + dir[CD_T + 2];
    dP0 = fmaf(c.R[0], dX0, fmaf(c.R[1], dX1, fmaf(c.R[2], dX2, dP0)));
    dP1 = fmaf(c.R[3], dX0, fmaf(c.R[4], dX1, fmaf(c.R[5], dX2, dP1)));
    dP2 = fmaf(c.R[6], dX0, fmaf(c.R[7], dX1, fmaf(c.R[8], dX2, dP2)));
    const float fn2 = c.f * g.n2;
    const float ci = fmaf(g.s, dir[CD_I + 0], fmaf(fn2, dir[CD_I + 1], fn2 * g.n2 * dir[CD_I + 2]));
    t0 = fmaf(g.A[0], dP0, fmaf(g.A[1], dP1, fmaf(g.A[2], dP2, ci * g.p[0])));
    t1 = fmaf(g.A[3], dP0, fmaf(g.A[4], dP1, fmaf(g.A[5], dP2, ci * g.p[1])));
}

// One observation's 2 x 12 Jacobian (camera columns, then point columns; 96 bytes) to `out`:
// six 16-byte stores when the address allows, since the rows of neighbouring lanes go to
// unrelated places and each store instruction costs a transaction per lane (1.2M observations:
// 301 us with scalar stores, 172 us so).
__device__ __forceinline__ void store_jacobian(float* out, const float (&j0)[9], const float (&jx0)[3],
                                               const float (&j1)[9], const float (&jx1)[3]) {
    if ((reinterpret_cast<uintptr_t>(out) & 15u) == 0) {
        float4* o = reinterpret_cast<float4*>(out);
        o[0] = make_float4(j0[0], j0[1], j0[2], j0[3]);
        o[1] = make_float4(j0[4], j0[5], j0[6], j0[7]);
        o[2] = make_float4(j0[8], jx0[0], jx0[1], jx0[2]);
        o[3] = make_float4(j1[0], j1[1], j1[2], j1[3]);
        o[4] = make_float4(j1[4], j1[5], j1[6], j1[7]);
        o[5] = make_float4(j1[8], jx1[0], jx1[1], jx1[2]);
    } else {
#pragma unroll
        for (int k = 0; k < 9; ++k) { out[k] = j0[k]; out[12 + k] = j1[k]; }
#pragma unroll
        for (int q = 0; q < 3; ++q) { out[9 + q] = jx0[q]; out[21 + q] = jx1[q]; }
    }
}

__device__ __forceinline__ void store_residual(float* out, float r0, float r1) {
    if ((reinterpret_cast<uintptr_t>(out) & 7u) == 0) {
        *reinterpret_cast<float2*>(out) = make_float2(r0, r1);
    } else {
        out[0] = r0;
        out[1] = r1;
    }
}

// Block-Jacobi inverse of one point block H + mu D (H packed xx, xy, xz, yy, yz, zz; D its
// diagonal clamped to [lo, hi]) in FP64 by the adjugate, M = adj(A) / det(A); the inverse of
// the diagonal where A is not positive definite.  lo_f, hi_f: the bounds as floats on the inner
// side, so that h >= lo exactly when h >= lo_f.  Writes M (packed) and D in FP32.  FP64 runs
// at 1/64 of the FP32 rate here (a warp instruction holds the SM's FP64 pipe for 16 cycles):
// only the 28 instructions of the inverse itself are FP64; clamping, comparisons and
// conversions run on the integer and FP32 units (the 28.8M-observation workload's
// preconditioner took 688 us with them in FP64).
__device__ __forceinline__ void point_inverse(const float (&H)[6], double mu, double lo, double hi, float lo_f,
                                              float hi_f, float (&m)[6], float (&D)[3]) {
    const float hd[3] = {H[0], H[3], H[5]};
    double a[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a[k] = widen(hd[k]);
        D[k] = hd[k];
        double d = a[k];
        if (!(hd[k] >= lo_f && hd[k] <= hi_f)) {   // clamped
            d = fmin(fmax(a[k], lo), hi);
            D[k] = (float)d;
        }
        a[k] = fma(mu, d, a[k]);
    }
    const double a00 = a[0], a11 = a[1], a22 = a[2], a01 = widen(H[1]), a02 = widen(H[2]), a12 = widen(H[4]);
    const double c00 = fma(a11, a22, -(a12 * a12)), c01 = fma(a02, a12, -(a01 * a22));
    const double c02 = fma(a01, a12, -(a02 * a11)), c11 = fma(a00, a22, -(a02 * a02));
    const double c12 = fma(a01, a02, -(a00 * a12)), c22 = fma(a00, a11, -(a01 * a01));
    const double det = fma(a00, c00, fma(a01, c01, a02 * c02));
    // positive and finite, from the high words (those of infinities and NaN are above)
    const int dh = __double2hiint(det);
    if (dh > 0 && dh < 0x7ff00000 && __double2hiint(a00) > 0 && __double2hiint(c22) > 0) {
        const double id = rcp64(det);
        m[0] = narrow(c00 * id); m[1] = narrow(c01 * id); m[2] = narrow(c02 * id);
        m[3] = narrow(c11 * id); m[4] = narrow(c12 * id); m[5] = narrow(c22 * id);
    } else {   // not SPD in FP64: inverse diagonal
        m[0] = a00 > 0 ? (float)(1.0 / a00) : 0.0f; m[1] = 0.0f; m[2] = 0.0f;
        m[3] = a11 > 0 ? (float)(1.0 / a11) : 0.0f; m[4] = 0.0f;
        m[5] = a22 > 0 ? (float)(1.0 / a22) : 0.0f;
    }
}

// Observations per thread when a CTA of `threads` threads splits `n` of them into
// contiguous chunks, rounded up to an odd count.  A camera's run covers consecutive
// tile slots, so lanes inside one run sit `chunk` slots apart: an odd stride sends
// their float4 point loads to distinct bank groups and their three-float point
// accumulations to distinct banks, where an even one (16 is the worst) serialises
// up to 16 of them.
template <typename T>
__host__ __device__ __forceinline__ T odd_chunk(T n, T threads) {
    return ((n + threads - 1) / threads) | (T)1;
}

__device__ __forceinline__ bool gated_off(const int32_t* gate) { return gate != nullptr && *gate == 0; }


// Camera direction record of camera c for p_c = zs_c + beta p_prev_c: phi = J_l p_w,
// then p_t and the intrinsic part.  zs and p_prev may change between launches or
// grid-wide phases, so they are read through L2 (never stale in L1).
__device__ __forceinline__ void camera_dir(const Views<float>& v, uint32_t c, const float* __restrict__ zs,
                                           const float* __restrict__ pc_old, float beta, float (&dir)[9]) {
    float pcv[9];
    const size_t e = 9 * (size_t)c;
#pragma unroll
    for (int k = 0; k < 9; ++k) pcv[k] = beta != 0.0f ? fmaf(beta, __ldcg(pc_old + e + k), __ldcg(zs + e + k)) : __ldcg(zs + e + k);
    const float4* j4 = reinterpret_cast<const float4*>(v.cam_pre + (size_t)c * CP_STRIDE + CP_JL);
    const float4 a = __ldg(j4), b = __ldg(j4 + 1), cc = __ldg(j4 + 2);
    const float JL[9] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, cc.x};
#pragma unroll
    for (int i = 0; i < 3; ++i) dir[CD_PHI + i] = fmaf(JL[3 * i], pcv[0], fmaf(JL[3 * i + 1], pcv[1], JL[3 * i + 2] * pcv[2]));
#pragma unroll
    for (int k = 3; k < 9; ++k) dir[k] = pcv[k];
}

// ---- one observation of the normal operator ---------------------------------------------
// J d and J^T t in camera coordinates.  With P~ = P + (0, 0, se), se = +-eps (the depth
// guard), p = -P~.xy / P~.z and v = (-p0, -p1, 1) = P~ / P~.z:
//   d(P)/P~.z = phi x v + (w + R dX) / P~.z,  w = d_t - phi x t  (se enters w),
//   e = dp = -(d(P).xy + p d(P).z) / P~.z,   J d = M e + c_i p,   M = a I + b p p^T,
//   c_i = d_f + n2 (c1 + n2 c2),  c1 = k1 d_f + f d_k1,  c2 = k2 d_f + f d_k2,
// and the adjoint of t: y = M t, u = -(y, p.y) / P~.z, P x u from y and p alone, and the
// intrinsic part as the three moments p.t, n2 p.t, n2^2 p.t.  The camera-constant factors
// (fk1 = f k1, w, c1, c2) are formed once per camera run and the camera sums brought to
// the record's form once per run (op_finish): 88 operations per observation, where the same
// products written per observation with R X, t and the intrinsics apart took 115.
struct OpCam {
    float R[9], t[3], f, fk1, fk2, b1, b2;   // a = f + n2 (fk1 + n2 fk2), b = b1 + n2 b2
};
struct OpDir {
    float ph[3], w[3], d6, c1, c2;
};

__device__ __forceinline__ OpCam op_cam(const Cam& m) {
    OpCam c;
#pragma unroll
    for (int k = 0; k < 9; ++k) c.R[k] = m.R[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) c.t[k] = m.t[k];
    c.f = m.f;
    c.fk1 = m.f * m.k1;
    c.fk2 = m.f * m.k2;
    c.b1 = 2.0f * c.fk1;
    c.b2 = 4.0f * c.fk2;
    return c;
}

// From a camera's direction record (phi, d_t, d_f, d_k1, d_k2).
__device__ __forceinline__ OpDir op_dir(const Cam& m, const float (&dir)[9]) {
    OpDir d;
#pragma unroll
    for (int k = 0; k < 3; ++k) d.ph[k] = dir[CD_PHI + k];
    d.w[0] = dir[CD_T + 0] - fmaf(dir[1], m.t[2], -dir[2] * m.t[1]);
    d.w[1] = dir[CD_T + 1] - fmaf(dir[2], m.t[0], -dir[0] * m.t[2]);
    d.w[2] = dir[CD_T + 2] - fmaf(dir[0], m.t[1], -dir[1] * m.t[0]);
    d.d6 = dir[CD_I];
    d.c1 = fmaf(m.k1, dir[CD_I], m.f * dir[CD_I + 1]);
    d.c2 = fmaf(m.k2, dir[CD_I], m.f * dir[CD_I + 2]);
    return d;
}

struct OpGeo {
    float iz, p0, p1, n2, a, b, se;
};

// EPS: the depth guard may be non-zero.
template <bool EPS>
__device__ __forceinline__ OpGeo op_geo(const OpCam& c, float X0, float X1, float X2, float eps) {
    OpGeo g;
    // P rounded as the linearisation rounds it (project_geo): a point close to a camera has few
    // bits left in P, and a Jacobian whose last bits differ from those in g = J^T r costs a digit
    // of the step there (t as the start of the FMA chain, three operations less: on 13,000
    // cameras a solve's error against 64 bits rose from 2.8e-8 to 4.1e-8 and, on a scene with such
    // points, from 2e-6 to 2e-5)
    const float P0 = fmaf(c.R[0], X0, fmaf(c.R[1], X1, c.R[2] * X2)) + c.t[0];
    const float P1 = fmaf(c.R[3], X0, fmaf(c.R[4], X1, c.R[5] * X2)) + c.t[1];
    const float P2 = fmaf(c.R[6], X0, fmaf(c.R[7], X1, c.R[8] * X2)) + c.t[2];
    g.se = EPS ? (P2 >= 0.0f ? eps : -eps) : 0.0f;
    g.iz = rcp_approx(EPS ? P2 + g.se : P2);
    g.p0 = -P0 * g.iz;
    g.p1 = -P1 * g.iz;
    g.n2 = fmaf(g.p0, g.p0, g.p1 * g.p1);
    g.a = fmaf(g.n2, fmaf(g.n2, c.fk2, c.fk1), c.f);
    g.b = fmaf(g.n2, c.b2, c.b1);
    return g;
}

// t = J d (the point's direction dx).
template <bool EPS>
__device__ __forceinline__ void op_forward(const OpCam& c, const OpDir& d, const OpGeo& g, float dx0, float dx1,
                                           float dx2, float& t0, float& t1) {
    float W0 = d.w[0], W1 = d.w[1];
    if (EPS) {
        W0 = fmaf(-d.ph[1], g.se, W0);
        W1 = fmaf(d.ph[0], g.se, W1);
    }
    const float w0 = fmaf(c.R[0], dx0, fmaf(c.R[1], dx1, fmaf(c.R[2], dx2, W0)));
    const float w1 = fmaf(c.R[3], dx0, fmaf(c.R[4], dx1, fmaf(c.R[5], dx2, W1)));
    const float w2 = fmaf(c.R[6], dx0, fmaf(c.R[7], dx1, fmaf(c.R[8], dx2, d.w[2])));
    const float ka = fmaf(d.ph[1], g.p0, -d.ph[0] * g.p1);
    // -e
    const float e0 = fmaf(g.iz, fmaf(g.p0, w2, w0), fmaf(g.p0, ka, fmaf(d.ph[2], g.p1, d.ph[1])));
    const float e1 = fmaf(g.iz, fmaf(g.p1, w2, w1), fmaf(g.p1, ka, fmaf(-d.ph[2], g.p0, -d.ph[0])));
    const float ci = fmaf(g.n2, fmaf(g.n2, d.c2, d.c1), d.d6);
    const float m = fmaf(-g.b, fmaf(g.p0, e0, g.p1 * e1), ci);
    t0 = fmaf(m, g.p0, -g.a * e0);
    t1 = fmaf(m, g.p1, -g.a * e1);
}

// J^T t: camera moments into acc, and v = -u with u = A^T t (the point part is R^T u).
template <bool EPS>
__device__ __forceinline__ void op_adjoint(const OpGeo& g, float t0, float t1, float (&acc)[9], float& v0, float& v1,
                                           float& v2) {
    const float pt = fmaf(g.p0, t0, g.p1 * t1);
    const float bp = g.b * pt;
    const float y0 = fmaf(g.a, t0, bp * g.p0), y1 = fmaf(g.a, t1, bp * g.p1);
    const float py = fmaf(g.p0, y0, g.p1 * y1);
    v0 = g.iz * y0;
    v1 = g.iz * y1;
    v2 = g.iz * py;
    acc[0] += fmaf(g.p1, py, y1);
    acc[1] -= fmaf(g.p0, py, y0);
    acc[2] = fmaf(g.p0, y1, fmaf(-g.p1, y0, acc[2]));
    if (EPS) {
        acc[0] = fmaf(-g.se, v1, acc[0]);
        acc[1] = fmaf(g.se, v0, acc[1]);
    }
    acc[3] += v0;
    acc[4] += v1;
    acc[5] += v2;
    const float np = g.n2 * pt;
    acc[6] += pt;
    acc[7] += np;
    acc[8] = fmaf(g.n2, np, acc[8]);
}

// q += R^T u = -R^T v.
__device__ __forceinline__ void op_point(const OpCam& c, float v0, float v1, float v2, float& q0, float& q1, float& q2) {
    q0 = fmaf(-c.R[0], v0, fmaf(-c.R[3], v1, fmaf(-c.R[6], v2, q0)));
    q1 = fmaf(-c.R[1], v0, fmaf(-c.R[4], v1, fmaf(-c.R[7], v2, q1)));
    q2 = fmaf(-c.R[2], v0, fmaf(-c.R[5], v1, fmaf(-c.R[8], v2, q2)));
}

// Camera moments of a run -> the camera sums of the accumulators (sum R X x u, sum u, intrinsic
// part): R X = P - t.  Linear, so it may be applied to partial sums.
__device__ __forceinline__ void op_finish(const OpCam& c, float k1, float k2, float (&acc)[9]) {
    const float u0 = -acc[3], u1 = -acc[4], u2 = -acc[5];
    acc[0] -= fmaf(c.t[1], u2, -c.t[2] * u1);
    acc[1] -= fmaf(c.t[2], u0, -c.t[0] * u2);
    acc[2] -= fmaf(c.t[0], u1, -c.t[1] * u0);
    acc[3] = u0;
    acc[4] = u1;
    acc[5] = u2;
    const float s1 = acc[7], s2 = acc[8];
    acc[6] = fmaf(k2, s2, fmaf(k1, s1, acc[6]));
    acc[7] = c.f * s1;
    acc[8] = c.f * s2;
}

// Contribution of one observation to the normal operator: t = J d (returns |t|^2), the camera
// moments into acc, the point part R^T u into qs (shared).  GEN: the depth guard may be
// non-zero, and the robust loss's IRLS weight w scales the observation's rows of J^T J
// (u = A^T (w t), returns w |t|^2).  PLAIN_Q: qs belongs to the calling warp alone and
// no other lane of it touches the same point in this step, so plain adds replace the
// shared-memory atomics.
template <bool GEN, bool PLAIN_Q = false>
__device__ __forceinline__ float obs_normal(const OpCam& cam, const OpDir& dir, const float4 x, const float4 dx,
                                            float eps, float w, float (&acc)[9], float* qs) {
    const OpGeo g = op_geo<GEN>(cam, x.x, x.y, x.z, eps);
    float t0, t1;
    op_forward<GEN>(cam, dir, g, dx.x, dx.y, dx.z, t0, t1);
    float tt = fmaf(t0, t0, t1 * t1);
    if (GEN) {
        tt *= w;
        t0 *= w;
        t1 *= w;
    }
    float v0, v1, v2;
    op_adjoint<GEN>(g, t0, t1, acc, v0, v1, v2);
    if (PLAIN_Q) {
        op_point(cam, v0, v1, v2, qs[0], qs[1], qs[2]);
    } else {
        float q0 = 0.0f, q1 = 0.0f, q2 = 0.0f;
        op_point(cam, v0, v1, v2, q0, q1, q2);
        atomicAdd(qs + 0, q0);
        atomicAdd(qs + 1, q1);
        atomicAdd(qs + 2, q2);
    }
    return tt;
}

// One pose factor in the normal operator: t = J_f (d_a; d_b) over the (phi, t) parts of
// the two cameras' direction records, J_f^T t added to their camera sums (phi part to
// entries 0-2, translation part to 3-5, as the observations' sums); returns |t|^2.
__device__ __forceinline__ float factor_normal(const float* __restrict__ Jf, const float* da, const float* db,
                                               float* acc_a, float* acc_b) {
    const float x[12] = {da[CD_PHI], da[CD_PHI + 1], da[CD_PHI + 2], da[CD_T], da[CD_T + 1], da[CD_T + 2],
                         db[CD_PHI], db[CD_PHI + 1], db[CD_PHI + 2], db[CD_T], db[CD_T + 1], db[CD_T + 2]};
    float t[6], tt = 0.0f;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        float ti = 0.0f;
#pragma unroll
        for (int j = 0; j < 12; ++j) ti = fmaf(__ldg(Jf + 12 * i + j), x[j], ti);
        t[i] = ti;
        tt = fmaf(ti, ti, tt);
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        float ga = 0.0f, gb = 0.0f;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            ga = fmaf(__ldg(Jf + 12 * i + j), t[i], ga);
            gb = fmaf(__ldg(Jf + 12 * i + 6 + j), t[i], gb);
        }
        atomicAdd(acc_a + j, ga);
        atomicAdd(acc_b + j, gb);
    }
    return tt;
}

}  // namespace gbba
