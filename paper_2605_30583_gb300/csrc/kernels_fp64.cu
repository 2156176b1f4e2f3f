// Plain all-FP64 form of the LM + PCGNR solver (the comparison baseline): the same
// algorithm as the mixed-precision path (Sec. V of arXiv 2605.30583) written the
// straightforward way -- FP64 everywhere, the Jacobian computed once per
// linearisation and stored (24 doubles per observation).  A CTA takes a tile: observations
// in their camera-sorted order a thread (or warp) each, camera sums in registers along a
// camera's run with one FP64 atomic per entry and run (one per entry and observation, all of a
// camera's on the same few addresses, bound these kernels before), then a thread per point
// (the point-major index), so point sums need no atomics.
#include <cuda_runtime.h>

#include <algorithm>

#include "device_common.cuh"
#include "kernels.h"

namespace gbba {

using V64 = Views<double>;

namespace {

// Camera record in FP64, same field order as the FP32 record (CP_*).
// With `retract` the rotation Jacobian is taken w.r.t. the tangent step d of
// R <- Exp(d) R(w) at d = 0: J_l is replaced by I.
__device__ void camera_record64(const double* c, double* out, bool retract = false) {
    const double w0 = c[0], w1 = c[1], w2 = c[2];
    const double th2 = w0 * w0 + w1 * w1 + w2 * w2;
    double A, B, C;
    rodrigues_coeffs(th2, A, B, C);
    const double K[9] = {0.0, -w2, w1, w2, 0.0, -w0, -w1, w0, 0.0};
    const double K2[9] = {w0 * w0 - th2, w0 * w1, w0 * w2, w1 * w0, w1 * w1 - th2, w1 * w2,
                          w2 * w0, w2 * w1, w2 * w2 - th2};
    for (int i = 0; i < 9; ++i) {
        const double I = (i % 4 == 0) ? 1.0 : 0.0;
        out[CP_R + i] = I + A * K[i] + B * K2[i];
        out[CP_JL + i] = retract ? I : I + B * K[i] + C * K2[i];
    }
    for (int k = 0; k < 3; ++k) out[CP_T + k] = c[3 + k];
    out[CP_F] = c[6];
    out[CP_K1] = c[7];
    out[CP_K2] = c[8];
    out[CP_PAD] = 0.0;
}

// Residual and the 2x12 Jacobian (camera 9 columns, point 3) of one observation.
__device__ void obs_jacobian64(const double* cam, double X0, double X1, double X2, double eps, double u0,
                               double u1, double& r0, double& r1, double* J /* [2][12] */) {
    const double* R = cam + CP_R;
    const double* JL = cam + CP_JL;
    const double RX0 = R[0] * X0 + R[1] * X1 + R[2] * X2;
    const double RX1 = R[3] * X0 + R[4] * X1 + R[5] * X2;
    const double RX2 = R[6] * X0 + R[7] * X1 + R[8] * X2;
    const double P0 = RX0 + cam[CP_T], P1 = RX1 + cam[CP_T + 1], P2 = RX2 + cam[CP_T + 2];
    const double d = P2 + (P2 >= 0.0 ? eps : -eps);
    const double iz = 1.0 / d;
    const double p0 = -P0 * iz, p1 = -P1 * iz;
    const double n2 = p0 * p0 + p1 * p1;
    const double f = cam[CP_F], k1 = cam[CP_K1], k2 = cam[CP_K2];
    const double s = 1.0 + n2 * (k1 + k2 * n2);
    const double sp = k1 + 2.0 * k2 * n2;
    r0 = f * s * p0 - u0;
    r1 = f * s * p1 - u1;
    if (!J) return;
    // A = d(pixel)/dP = M dp/dP, M = f (s I + 2 s' p p^T), dp/dP = -iz [[1,0,p0],[0,1,p1]]
    const double a = f * s, b = 2.0 * f * sp;
    const double m00 = a + b * p0 * p0, m01 = b * p0 * p1, m11 = a + b * p1 * p1;
    const double A0 = -iz * m00, A1 = -iz * m01, A2 = -iz * (m00 * p0 + m01 * p1);
    const double A3 = -iz * m01, A4 = -iz * m11, A5 = -iz * (m01 * p0 + m11 * p1);
    for (int k = 0; k < 3; ++k) {
        const double wa = JL[k], wb = JL[3 + k], wc = JL[6 + k];   // column k of J_l
        const double c0 = wb * RX2 - wc * RX1, c1 = wc * RX0 - wa * RX2, c2 = wa * RX1 - wb * RX0;
        J[k] = A0 * c0 + A1 * c1 + A2 * c2;
        J[12 + k] = A3 * c0 + A4 * c1 + A5 * c2;
    }
    J[3] = A0; J[4] = A1; J[5] = A2;
    J[15] = A3; J[16] = A4; J[17] = A5;
    J[6] = s * p0; J[7] = f * n2 * p0; J[8] = f * n2 * n2 * p0;
    J[18] = s * p1; J[19] = f * n2 * p1; J[20] = f * n2 * n2 * p1;
    for (int k = 0; k < 3; ++k) {
        J[9 + k] = A0 * R[k] + A1 * R[3 + k] + A2 * R[6 + k];
        J[21 + k] = A3 * R[k] + A4 * R[3 + k] + A5 * R[6 + k];
    }
}

__device__ __forceinline__ int grid_threads() { return gridDim.x * blockDim.x; }
__device__ __forceinline__ int gtid() { return blockIdx.x * blockDim.x + threadIdx.x; }

}  // namespace

__global__ void k64_camera_precompute(V64 v) {
    for (int c = gtid(); c < v.n_cams; c += grid_threads()) {
        camera_record64(v.x + 9 * (size_t)c, v.cam64 + (size_t)c * CP_STRIDE, v.st->opt.retract != 0);
        for (int k = 0; k < CL_STRIDE; ++k) v.cam_lin[(size_t)c * CL_STRIDE + k] = 0.0;
        for (int k = 0; k < CH_STRIDE; ++k) v.cam_H64[(size_t)c * CH_STRIDE + k] = 0.0;
    }
}

// Linearisation, a CTA of TILE_PTS threads per tile.  First a thread per observation: r and J
// stored.  Then the tile's observations in order, a contiguous part to a warp: lane l holds the
// entries l and l + 32 of a camera's 54 sums (g and the J_c^T J_c triangle), so every lane works
// on one observation's row at a time and nothing has to be reduced.  Then a thread per point.
// Bound by the FP64 pipe.  (A thread per point over its scattered observations, with 54 atomics
// each, and the operator below in the same form: 11.4 ms for a solve of 3 x 15 iterations of 200
// cameras and 50,000 points, 5.3 ms so.)
constexpr int T64 = TILE_PTS;

__global__ void __launch_bounds__(T64) k64_linearize(V64 v, int mode, double* res_out, double* jac_out,
                                                     CondHandle lm_cond, int use_cond) {
    if (mode == 1 && v.st->relin == 0) return;
    const double eps = v.st->opt.eps;
    // robust loss (evaluation, mode 2, is always the squared loss)
    const int loss = mode == 2 ? 0 : v.st->opt.loss;
    const double lscale = v.st->opt.loss_scale;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the row and column of this lane's two entries; entries below 9 are g (column = residual)
    int ra[2], ca[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int t = lane + 32 * q;
        ra[q] = ca[q] = 0;
        if (t < 9) {
            ra[q] = t;
            ca[q] = -1;
        } else {
            for (int i = 0; i < 9; ++i)
                if (t - 9 >= tri_index(9, i, i) && t - 9 < tri_index(9, i, i) + 9 - i) {
                    ra[q] = i;
                    ca[q] = i + (t - 9 - tri_index(9, i, i));
                }
        }
    }
    double cost = 0.0;
    for (int tile = blockIdx.x; tile < v.n_tiles; tile += gridDim.x) {
        const uint32_t lo = v.tile_off[tile], n = v.tile_off[tile + 1] - lo;
        const double* Xt = v.x + v.pt_off + 3 * (size_t)tile * v.tile_pts;
        for (uint32_t j = lo + threadIdx.x; j < lo + n; j += T64) {
            const uint32_t key = v.obs_key[j], c = key >> 8;
            const double* X = Xt + 3 * (key & 0xffu);
            double J[24], r0, r1;
            obs_jacobian64(v.cam64 + (size_t)c * CP_STRIDE, X[0], X[1], X[2], eps, v.obs_uv[2 * (size_t)j],
                           v.obs_uv[2 * (size_t)j + 1], r0, r1, J);
            if (mode == 2) {   // evaluation output: the unweighted residual and Jacobian
                const uint32_t o = v.obs_user[j];
                if (res_out) { res_out[2 * (size_t)o] = r0; res_out[2 * (size_t)o + 1] = r1; }
                if (jac_out) for (int q = 0; q < 24; ++q) jac_out[24 * (size_t)o + q] = J[q];
            }
            if (loss) {   // IRLS: the stored rows are scaled by sqrt(rho'(|r|^2))
                const double s2 = r0 * r0 + r1 * r1;
                cost += loss_rho64(s2, loss, lscale);
                const double sw = sqrt(loss_weight64(s2, loss, lscale));
                r0 *= sw;
                r1 *= sw;
                for (int q = 0; q < 24; ++q) J[q] *= sw;
            } else {
                cost += r0 * r0 + r1 * r1;
            }
            double2* Jo = reinterpret_cast<double2*>(v.jac + 24 * (size_t)j);
#pragma unroll
            for (int q = 0; q < 12; ++q) Jo[q] = make_double2(J[2 * q], J[2 * q + 1]);
            reinterpret_cast<double2*>(v.res)[j] = make_double2(r0, r1);
        }
        __syncthreads();   // the tile's rows are written
        const uint32_t chunk = (n + T64 / 32 - 1) / (T64 / 32);
        const uint32_t a = lo + min(warp * chunk, n), b = lo + min(warp * chunk + chunk, n);
        double acc[2] = {0.0, 0.0};
        for (uint32_t j = a; j < b; ++j) {
            const uint32_t c = v.obs_key[j] >> 8;
            const double* J = v.jac + 24 * (size_t)j;
            const double* r = v.res + 2 * (size_t)j;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const double y0 = ca[q] < 0 ? r[0] : J[ca[q]], y1 = ca[q] < 0 ? r[1] : J[12 + ca[q]];
                acc[q] = fma(J[ra[q]], y0, fma(J[12 + ra[q]], y1, acc[q]));
            }
            if (j + 1 == b || (v.obs_key[j + 1] >> 8) != c) {   // the run ends
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int t = lane + 32 * q;
                    if (t < 9) atomicAdd(v.cam_lin + (size_t)c * CL_STRIDE + t, acc[q]);
                    else if (t < 54) atomicAdd(v.cam_H64 + (size_t)c * CH_STRIDE + (t - 9), acc[q]);
                    acc[q] = 0.0;
                }
            }
        }
        const int ip = tile * v.tile_pts + (int)threadIdx.x;
        if ((int)threadIdx.x < v.tile_pts && ip < v.n_pts) {
            double gp[3] = {0, 0, 0}, hp[6] = {0, 0, 0, 0, 0, 0};
            for (uint32_t k = v.pt_obs_off[ip]; k < v.pt_obs_off[ip + 1]; ++k) {
                const uint32_t j = v.obs_pm[k];
                const double* J = v.jac + 24 * (size_t)j;
                const double r0 = v.res[2 * (size_t)j], r1 = v.res[2 * (size_t)j + 1];
                for (int a = 0; a < 3; ++a) {
                    gp[a] += J[9 + a] * r0 + J[21 + a] * r1;
                    for (int b = a; b < 3; ++b) hp[tri_index(3, a, b)] += J[9 + a] * J[9 + b] + J[21 + a] * J[21 + b];
                }
            }
            for (int a = 0; a < 3; ++a) v.g[v.pt_off + 3 * (size_t)ip + a] = gp[a];
            for (int a = 0; a < 6; ++a) v.pt_H[(size_t)ip * PH_STRIDE + a] = hp[a];
        }
    }
    double in[1] = {cost}, out[1];
    if (grid_reduce<1>(in, v.partials, &v.st->tickets[TK_LIN], out) && threadIdx.x == 0) {
        DevState* st = v.st;
        const double F = 0.5 * out[0];
        st->cost_out = F;
        if (mode == 0) {
            st->F = F;
            st->F0 = F;
            const bool ok = isfinite(F);
            if (!ok) st->status = 4;
            st->lm_active = (ok && F > 0.0 && st->opt.max_lm > 0) ? 1 : 0;
            if (use_cond) cudaGraphSetConditional(lm_cond, st->lm_active ? 1u : 0u);
        } else if (mode == 1) {
            st->F = F;
        }
    }
}

// Block-Jacobi inverses (FP64, camera blocks by warp Gauss-Jordan, points by adjugate)
// and the PCGNR start: r = -g, z = M^-1 r, p = 0, h = 0.
__global__ void k64_precond(V64 v, CondHandle pcg_cond, int use_cond) {
    DevState* st = v.st;
    if (st->lm_active == 0) {
        if (use_cond && blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(pcg_cond, 0u);
        return;
    }
    const double mu = st->mu, lo = st->opt.min_diag, hi = st->opt.max_diag;
    double rz = 0.0, rr = 0.0;
    const int warps = gridDim.x * (blockDim.x >> 5);
    for (int c0 = 3 * (int)(gtid() >> 5); c0 < v.n_cams; c0 += 3 * warps) {
        const CamLane L = cam_lane(c0, v.n_cams);
        const int c = L.cam;
        double col[9], D, diag;
        const bool ok = camera_inverse9(v.cam_H64 + (size_t)c * CH_STRIDE, mu, lo, hi, L, col, D, diag);
        double* Mo = v.Minv_c + (size_t)c * MC_STRIDE;
        if (L.live)
            for (int i = 0; i < 9; ++i)
                Mo[i * 9 + L.i] = ok ? col[i] : (i == L.i && diag > 0.0) ? 1.0 / diag : 0.0;
        __syncwarp();
        if (L.live) {
            const size_t e = 9 * (size_t)c + L.i;
            v.D[e] = D;
            const double* gc = v.cam_lin + (size_t)c * CL_STRIDE;
            const double ri = -gc[L.i];
            double z = 0.0;
            for (int k = 0; k < 9; ++k) z += Mo[L.i * 9 + k] * (-gc[k]);
            v.r[e] = ri;
            v.z[e] = z;
            v.p[e] = 0.0;
            v.h[e] = 0.0;
            rz += ri * z;
            rr += ri * ri;
        }
    }
    for (int i = gtid(); i < v.n_pts; i += grid_threads()) {
        const double* H = v.pt_H + (size_t)i * PH_STRIDE;
        const size_t e = v.pt_off + 3 * (size_t)i;
        double a00 = H[0], a01 = H[1], a02 = H[2], a11 = H[3], a12 = H[4], a22 = H[5];
        const double d0 = fmin(fmax(a00, lo), hi), d1 = fmin(fmax(a11, lo), hi), d2 = fmin(fmax(a22, lo), hi);
        a00 += mu * d0; a11 += mu * d1; a22 += mu * d2;
        const double c00 = a11 * a22 - a12 * a12, c01 = a02 * a12 - a01 * a22, c02 = a01 * a12 - a02 * a11;
        const double c11 = a00 * a22 - a02 * a02, c12 = a01 * a02 - a00 * a12, c22 = a00 * a11 - a01 * a01;
        const double det = a00 * c00 + a01 * c01 + a02 * c02;
        double m[6];
        if (det > 0.0 && isfinite(det) && a00 > 0.0 && c22 > 0.0) {
            const double id = 1.0 / det;
            m[0] = c00 * id; m[1] = c01 * id; m[2] = c02 * id; m[3] = c11 * id; m[4] = c12 * id; m[5] = c22 * id;
        } else {
            m[0] = a00 > 0 ? 1.0 / a00 : 0.0; m[1] = 0.0; m[2] = 0.0;
            m[3] = a11 > 0 ? 1.0 / a11 : 0.0; m[4] = 0.0; m[5] = a22 > 0 ? 1.0 / a22 : 0.0;
        }
        for (int k = 0; k < 6; ++k) v.Minv_p[(size_t)i * MP_STRIDE + k] = m[k];
        v.D[e] = d0; v.D[e + 1] = d1; v.D[e + 2] = d2;
        const double r0 = -v.g[e], r1 = -v.g[e + 1], r2 = -v.g[e + 2];
        const double z0 = m[0] * r0 + m[1] * r1 + m[2] * r2;
        const double z1 = m[1] * r0 + m[3] * r1 + m[4] * r2;
        const double z2 = m[2] * r0 + m[4] * r1 + m[5] * r2;
        v.r[e] = r0; v.r[e + 1] = r1; v.r[e + 2] = r2;
        v.z[e] = z0; v.z[e + 1] = z1; v.z[e + 2] = z2;
        v.p[e] = v.p[e + 1] = v.p[e + 2] = 0.0;
        v.h[e] = v.h[e + 1] = v.h[e + 2] = 0.0;
        rz += r0 * z0 + r1 * z1 + r2 * z2;
        rr += r0 * r0 + r1 * r1 + r2 * r2;
    }
    double in[2] = {rz, rr}, out[2];
    if (grid_reduce<2>(in, v.partials, &st->tickets[TK_PRE], out) && threadIdx.x == 0) {
        st->rz = out[0];
        st->rr0 = out[1];
        st->rr = out[1];
        st->beta = 0.0;
        st->pcg_iter = 0;
        // a non-finite r^T z means a non-finite gradient or block (a Jacobian that
        // overflowed, e.g. a point at a camera centre): a numeric failure, not a stall
        if (!isfinite(out[0]) || !isfinite(out[1])) st->status = 4;
        st->pcg_active = (out[1] > 0.0 && isfinite(out[0]) && st->opt.max_pcg > 0) ? 1 : 0;
        if (use_cond) cudaGraphSetConditional(pcg_cond, st->pcg_active ? 1u : 0u);
    }
}

// p = zs + beta p (beta = 0 for a given direction zs = p); q = mu D p, the start of
// the atomically accumulated normal product; p^T D p.
__global__ void k64_direction(V64 v, const double* zs, int use_beta, const int32_t* gate) {
    if (gate && *gate == 0) return;
    DevState* st = v.st;
    const double beta = use_beta ? st->beta : 0.0, mu = st->mu;
    double pdp = 0.0;
    for (size_t e = gtid(); e < (size_t)v.n_vec; e += grid_threads()) {
        const double pk = beta != 0.0 ? zs[e] + beta * v.p[e] : zs[e];
        v.p[e] = pk;
        v.q[e] = mu * v.D[e] * pk;
        pdp += v.D[e] * pk * pk;
    }
    double in[1] = {pdp}, out[1];
    if (grid_reduce<1>(in, v.partials, &st->tickets[TK_DIR], out) && threadIdx.x == 0) st->pDp = out[0];
}

// q += J^T J p with the stored Jacobian, a CTA per tile: first the tile's observations in
// order, a contiguous part to a thread: t = J_o p (kept in the residuals' place, which nothing
// reads after the linearisation) and the camera sums in registers along a run; then a thread per
// point over its observations' t.
__global__ void __launch_bounds__(T64) k64_matvec(V64 v, const int32_t* gate) {
    if (gate && *gate == 0) return;
    DevState* st = v.st;
    double jp2 = 0.0;
    for (int tile = blockIdx.x; tile < v.n_tiles; tile += gridDim.x) {
        const uint32_t lo = v.tile_off[tile], n = v.tile_off[tile + 1] - lo;
        const uint32_t chunk = (n + T64 - 1) / T64;
        const uint32_t a = lo + min(threadIdx.x * chunk, n), b = lo + min(threadIdx.x * chunk + chunk, n);
        const double* Pt = v.p + v.pt_off + 3 * (size_t)tile * v.tile_pts;
        double acc[9], pc[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) acc[k] = pc[k] = 0.0;
        uint32_t cur = 0xffffffffu;
        for (uint32_t j = a; j < b; ++j) {
            const uint32_t key = v.obs_key[j], c = key >> 8;
            if (c != cur) {
                if (cur != 0xffffffffu)
#pragma unroll
                    for (int k = 0; k < 9; ++k) {
                        atomicAdd(v.q + 9 * (size_t)cur + k, acc[k]);
                        acc[k] = 0.0;
                    }
                cur = c;
#pragma unroll
                for (int k = 0; k < 9; ++k) pc[k] = v.p[9 * (size_t)c + k];
            }
            const double2* J2 = reinterpret_cast<const double2*>(v.jac + 24 * (size_t)j);
            double J[24];
#pragma unroll
            for (int q = 0; q < 12; ++q) {
                const double2 d = J2[q];
                J[2 * q] = d.x;
                J[2 * q + 1] = d.y;
            }
            const double* pp = Pt + 3 * (key & 0xffu);
            const double p0 = pp[0], p1 = pp[1], p2 = pp[2];
            double t0 = J[9] * p0 + J[10] * p1 + J[11] * p2;
            double t1 = J[21] * p0 + J[22] * p1 + J[23] * p2;
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                t0 += J[k] * pc[k];
                t1 += J[12 + k] * pc[k];
            }
            jp2 += t0 * t0 + t1 * t1;
            reinterpret_cast<double2*>(v.res)[j] = make_double2(t0, t1);
#pragma unroll
            for (int k = 0; k < 9; ++k) acc[k] = fma(J[k], t0, fma(J[12 + k], t1, acc[k]));
        }
        if (cur != 0xffffffffu)
#pragma unroll
            for (int k = 0; k < 9; ++k) atomicAdd(v.q + 9 * (size_t)cur + k, acc[k]);
        __syncthreads();   // the tile's t
        const int ip = tile * v.tile_pts + (int)threadIdx.x;
        if ((int)threadIdx.x < v.tile_pts && ip < v.n_pts) {
            const size_t ep = v.pt_off + 3 * (size_t)ip;
            double q0 = 0.0, q1 = 0.0, q2 = 0.0;
            for (uint32_t k = v.pt_obs_off[ip]; k < v.pt_obs_off[ip + 1]; ++k) {
                const uint32_t j = v.obs_pm[k];
                const double* J = v.jac + 24 * (size_t)j;
                const double2 t = reinterpret_cast<const double2*>(v.res)[j];
                q0 += J[9] * t.x + J[21] * t.y;
                q1 += J[10] * t.x + J[22] * t.y;
                q2 += J[11] * t.x + J[23] * t.y;
            }
            v.q[ep] += q0;
            v.q[ep + 1] += q1;
            v.q[ep + 2] += q2;
        }
    }
    double in[1] = {jp2}, out[1];
    if (grid_reduce<1>(in, v.partials, &st->tickets[TK_MV], out) && threadIdx.x == 0) {
        st->jp2 = out[0];
        const double denom = out[0] + st->mu * st->pDp;
        if (denom > 0.0 && isfinite(denom)) {
            st->alpha = st->rz / denom;
        } else {
            st->alpha = 0.0;
            if (st->pcg_active) {
                st->pcg_active = 0;
                if (!isfinite(denom)) st->status = 4;
            }
        }
    }
}

// h += alpha p; r -= alpha q; z = M^-1 r; r^T z, |r|^2; the last block takes the PCG
// stop decision and sets the loop flag.  Never gated.
__global__ void k64_update(V64 v, CondHandle pcg_cond, int use_cond) {
    DevState* st = v.st;
    const int active = st->pcg_active;
    double rz = 0.0, rr = 0.0;
    if (active) {
        const double alpha = st->alpha;
        // cameras: nine lanes each, three to a warp
        const int lane = threadIdx.x & 31;
        for (int cw = 3 * (gtid() >> 5); cw < v.n_cams; cw += 3 * (grid_threads() >> 5)) {
            const int sub = lane / 9, base = 9 * sub;
            const bool live = lane < 27 && cw + sub < v.n_cams;
            const int c = live ? cw + sub : cw, i = live ? lane - base : 0;
            const size_t e = 9 * (size_t)c + i;
            const double* M = v.Minv_c + (size_t)c * MC_STRIDE + 9 * i;
            const double rn = v.r[e] - alpha * v.q[e];
            double z = 0.0;
#pragma unroll
            for (int k = 0; k < 9; ++k) z += M[k] * __shfl_sync(0xffffffffu, rn, base + k);
            if (live) {
                v.h[e] += alpha * v.p[e];
                v.r[e] = rn;
                v.z[e] = z;
                rz += rn * z;
                rr += rn * rn;
            }
        }
        for (int i = gtid(); i < v.n_pts; i += grid_threads()) {
            const size_t e = v.pt_off + 3 * (size_t)i;
            double rn[3];
            for (int k = 0; k < 3; ++k) {
                v.h[e + k] += alpha * v.p[e + k];
                rn[k] = v.r[e + k] - alpha * v.q[e + k];
                v.r[e + k] = rn[k];
            }
            const double* m = v.Minv_p + (size_t)i * MP_STRIDE;
            const double z0 = m[0] * rn[0] + m[1] * rn[1] + m[2] * rn[2];
            const double z1 = m[1] * rn[0] + m[3] * rn[1] + m[4] * rn[2];
            const double z2 = m[2] * rn[0] + m[4] * rn[1] + m[5] * rn[2];
            v.z[e] = z0; v.z[e + 1] = z1; v.z[e + 2] = z2;
            rz += rn[0] * z0 + rn[1] * z1 + rn[2] * z2;
            rr += rn[0] * rn[0] + rn[1] * rn[1] + rn[2] * rn[2];
        }
    }
    double in[2] = {rz, rr}, out[2];
    if (grid_reduce<2>(in, v.partials, &st->tickets[TK_UPD], out) && threadIdx.x == 0) {
        if (active) {
            st->pcg_iter += 1;
            st->pcg_total += 1;
            st->rr = out[1];
            const double tol = st->opt.tol;
            if (!isfinite(out[0]) || !isfinite(out[1])) {
                st->status = 4;
                st->pcg_active = 0;
            } else if (out[1] <= tol * tol * st->rr0 || st->pcg_iter >= st->opt.max_pcg) {
                st->pcg_active = 0;
            } else {
                st->beta = out[0] / st->rz;
                st->rz = out[0];
            }
        }
        if (use_cond) cudaGraphSetConditional(pcg_cond, st->pcg_active ? 1u : 0u);
    }
}

// Candidate x' = x + h, g^T h, camera records at x'.
__global__ void k64_candidate(V64 v) {
    DevState* st = v.st;
    if (st->lm_active == 0) return;
    const bool retract = st->opt.retract != 0;
    double gh = 0.0;
    for (size_t e = gtid(); e < (size_t)v.n_vec; e += grid_threads()) {
        const bool cam = e < 9 * (size_t)v.n_cams;
        if (!(retract && cam && e % 9 < 3)) v.x_new[e] = v.x[e] + v.h[e];   // rotations: below
        const double ge = cam ? v.cam_lin[(e / 9) * CL_STRIDE + e % 9] : (e >= (size_t)v.pt_off ? v.g[e] : 0.0);
        gh += ge * v.h[e];
    }
    for (int c = gtid(); c < v.n_cams; c += grid_threads()) {
        double xn[9];
        for (int k = 0; k < 9; ++k) xn[k] = v.x[9 * (size_t)c + k] + v.h[9 * (size_t)c + k];
        if (retract) {   // R' = Exp(h_w) R(w)
            compose_rotvec(v.h + 9 * (size_t)c, v.x + 9 * (size_t)c, xn);
            for (int k = 0; k < 3; ++k) v.x_new[9 * (size_t)c + k] = xn[k];
        }
        camera_record64(xn, v.cam64_new + (size_t)c * CP_STRIDE, retract);
    }
    double in[1] = {gh}, out[1];
    if (grid_reduce<1>(in, v.partials, &st->tickets[TK_CAND], out) && threadIdx.x == 0) st->gh = out[0];
}

// F(x') and |J h|^2 with the stored Jacobian; the last block applies the LM rule.
__global__ void k64_eval_candidate(V64 v, CondHandle lm_cond, int use_cond) {
    DevState* st = v.st;
    const int active = st->lm_active;
    const double eps = st->opt.eps;
    const int loss = st->opt.loss;
    const double lscale = st->opt.loss_scale;
    double fnew = 0.0, jh2 = 0.0;
    if (active) {
        for (int tile = blockIdx.x; tile < v.n_tiles; tile += gridDim.x) {
            const size_t base = v.pt_off + 3 * (size_t)tile * v.tile_pts;
            for (uint32_t j = v.tile_off[tile] + threadIdx.x; j < v.tile_off[tile + 1]; j += blockDim.x) {
                const uint32_t key = v.obs_key[j], c = key >> 8;
                const double* Xn = v.x_new + base + 3 * (key & 0xffu);
                const double* hp = v.h + base + 3 * (key & 0xffu);
                double r0, r1;
                obs_jacobian64(v.cam64_new + (size_t)c * CP_STRIDE, Xn[0], Xn[1], Xn[2], eps, v.obs_uv[2 * (size_t)j],
                               v.obs_uv[2 * (size_t)j + 1], r0, r1, nullptr);
                fnew += loss ? loss_rho64(r0 * r0 + r1 * r1, loss, lscale) : r0 * r0 + r1 * r1;
                const double* J = v.jac + 24 * (size_t)j;   // sqrt(w)-scaled: |J h|^2 is weighted
                const double* hc = v.h + 9 * (size_t)c;
                double t0 = J[9] * hp[0] + J[10] * hp[1] + J[11] * hp[2];
                double t1 = J[21] * hp[0] + J[22] * hp[1] + J[23] * hp[2];
                for (int a = 0; a < 9; ++a) {
                    t0 += J[a] * hc[a];
                    t1 += J[12 + a] * hc[a];
                }
                jh2 += t0 * t0 + t1 * t1;
            }
        }
    }
    double in[2] = {fnew, jh2}, out[2];
    if (grid_reduce<2>(in, v.partials, &st->tickets[TK_COST], out) && threadIdx.x == 0) {
        lm_decide(st, active, 0.5 * out[0], out[1]);
        if (use_cond) cudaGraphSetConditional(lm_cond, st->lm_active ? 1u : 0u);
    }
}

__global__ void k64_commit(V64 v) {
    if (v.st->accepted == 0) return;
    for (size_t e = gtid(); e < (size_t)v.n_vec; e += grid_threads()) v.x[e] = v.x_new[e];
    for (int c = gtid(); c < v.n_cams; c += grid_threads()) {
        for (int k = 0; k < CP_STRIDE; ++k) v.cam64[(size_t)c * CP_STRIDE + k] = v.cam64_new[(size_t)c * CP_STRIDE + k];
        for (int k = 0; k < CL_STRIDE; ++k) v.cam_lin[(size_t)c * CL_STRIDE + k] = 0.0;
        for (int k = 0; k < CH_STRIDE; ++k) v.cam_H64[(size_t)c * CH_STRIDE + k] = 0.0;
    }
}

template <typename S>
__global__ void k64_pack(V64 v, const S* cams, const S* pts) {
    for (int c = gtid(); c < v.n_cams; c += grid_threads())
        for (int k = 0; k < 9; ++k) v.x[9 * (size_t)c + k] = (double)cams[9 * (size_t)c + k];
    for (int u = gtid(); u < v.n_pts; u += grid_threads()) {
        const size_t e = v.pt_off + 3 * (size_t)v.pt_internal[u];
        for (int k = 0; k < 3; ++k) v.x[e + k] = (double)pts[3 * (size_t)u + k];
    }
}

template <typename S>
__global__ void k64_unpack(V64 v, S* cams, S* pts) {
    for (int c = gtid(); c < v.n_cams; c += grid_threads())
        for (int k = 0; k < 9; ++k) cams[9 * (size_t)c + k] = (S)v.x[9 * (size_t)c + k];
    for (int u = gtid(); u < v.n_pts; u += grid_threads()) {
        const size_t e = v.pt_off + 3 * (size_t)v.pt_internal[u];
        for (int k = 0; k < 3; ++k) pts[3 * (size_t)u + k] = (S)v.x[e + k];
    }
}

// user-layout vector <-> internal p / q
__global__ void k64_set_vec(V64 v, const double* src, double* dst) {
    for (int c = gtid(); c < v.n_cams; c += grid_threads())
        for (int k = 0; k < 9; ++k) dst[9 * (size_t)c + k] = src[9 * (size_t)c + k];
    for (int u = gtid(); u < v.n_pts; u += grid_threads()) {
        const size_t e = v.pt_off + 3 * (size_t)v.pt_internal[u];
        for (int k = 0; k < 3; ++k) dst[e + k] = src[9 * (size_t)v.n_cams + 3 * (size_t)u + k];
    }
}

__global__ void k64_get_vec(V64 v, const double* src, double* dst) {
    for (int c = gtid(); c < v.n_cams; c += grid_threads())
        for (int k = 0; k < 9; ++k) dst[9 * (size_t)c + k] = src[9 * (size_t)c + k];
    for (int u = gtid(); u < v.n_pts; u += grid_threads()) {
        const size_t e = v.pt_off + 3 * (size_t)v.pt_internal[u];
        for (int k = 0; k < 3; ++k) dst[9 * (size_t)v.n_cams + 3 * (size_t)u + k] = src[e + k];
    }
}

// ------------------------------------------------------------- autograd ------
template <typename S>
__global__ void k64_pack_to(V64 v, const S* cams, const S* pts, double* dst) {
    for (int c = gtid(); c < v.n_cams; c += grid_threads())
        for (int k = 0; k < 9; ++k) dst[9 * (size_t)c + k] = (double)cams[9 * (size_t)c + k];
    for (int u = gtid(); u < v.n_pts; u += grid_threads()) {
        const size_t e = v.pt_off + 3 * (size_t)v.pt_internal[u];
        for (int k = 0; k < 3; ++k) dst[e + k] = (double)pts[3 * (size_t)u + k];
    }
}

__global__ void k64_records_from(V64 v, const double* src, double* dst) {
    for (int c = gtid(); c < v.n_cams; c += grid_threads()) {
        camera_record64(src + 9 * (size_t)c, dst + (size_t)c * CP_STRIDE);
        for (int k = 0; k < CL_STRIDE; ++k) v.cam_lin[(size_t)c * CL_STRIDE + k] = 0.0;
    }
}

// F = 1/2 |r|^2 and, if want_grad, J^T r (cameras by FP64 atomics, points in registers).
__global__ void k64_cost_grad(V64 v, const double* xs, const double* crec, int want_grad, double* cost_dev) {
    const double eps = v.st->opt.eps;
    double cost = 0.0;
    for (int ip = gtid(); ip < v.n_pts; ip += grid_threads()) {
        const double* X = xs + v.pt_off + 3 * (size_t)ip;
        double gp[3] = {0, 0, 0};
        for (uint32_t k = v.pt_obs_off[ip]; k < v.pt_obs_off[ip + 1]; ++k) {
            const uint32_t j = v.obs_pm[k];
            const uint32_t c = v.obs_key[j] >> 8;
            double J[24], r0, r1;
            obs_jacobian64(crec + (size_t)c * CP_STRIDE, X[0], X[1], X[2], eps, v.obs_uv[2 * (size_t)j],
                           v.obs_uv[2 * (size_t)j + 1], r0, r1, want_grad ? J : nullptr);
            cost += r0 * r0 + r1 * r1;
            if (want_grad) {
                for (int a = 0; a < 9; ++a) atomicAdd(v.cam_lin + (size_t)c * CL_STRIDE + a, J[a] * r0 + J[12 + a] * r1);
                for (int a = 0; a < 3; ++a) gp[a] += J[9 + a] * r0 + J[21 + a] * r1;
            }
        }
        if (want_grad)
            for (int a = 0; a < 3; ++a) v.g[v.pt_off + 3 * (size_t)ip + a] = gp[a];
    }
    double in[1] = {cost}, out[1];
    if (grid_reduce<1>(in, v.partials, &v.st->tickets[TK_MISC], out) && threadIdx.x == 0) {
        v.st->cost_out = 0.5 * out[0];
        if (cost_dev) *cost_dev = 0.5 * out[0];
    }
}

template <typename S>
__global__ void k64_grad_out(V64 v, const double* grad_out, S* gc, S* gp) {
    const double s = *grad_out;
    for (int c = gtid(); c < v.n_cams; c += grid_threads())
        for (int k = 0; k < 9; ++k) gc[9 * (size_t)c + k] = (S)(s * v.cam_lin[(size_t)c * CL_STRIDE + k]);
    for (int u = gtid(); u < v.n_pts; u += grid_threads()) {
        const size_t e = v.pt_off + 3 * (size_t)v.pt_internal[u];
        for (int k = 0; k < 3; ++k) gp[3 * (size_t)u + k] = (S)(s * v.g[e + k]);
    }
}

// ------------------------------------------------------------------ launchers --

namespace {
inline int g64(const LaunchCfg& L, size_t items) {
    size_t g = (items + L.item_block - 1) / L.item_block;
    return (int)std::max<size_t>(1, std::min<size_t>(g, (size_t)L.item_grid));
}
// A CTA per tile, capped by the partial sums' room.
inline int tiles64(const V64& v) { return std::max(1, std::min(v.n_tiles, MAX_GRID)); }
}  // namespace

void launch64_camera_precompute(const V64& v, const LaunchCfg& L, cudaStream_t s) {
    k64_camera_precompute<<<g64(L, v.n_cams), L.item_block, 0, s>>>(v);
}
void launch64_linearize(const V64& v, const LaunchCfg& L, cudaStream_t s, int mode, double* r, double* J,
                        CondHandle c, int use) {
    k64_linearize<<<tiles64(v), T64, 0, s>>>(v, mode, r, J, c, use);
}
void launch64_precond(const V64& v, const LaunchCfg& L, cudaStream_t s, CondHandle c, int use) {
    k64_precond<<<g64(L, std::max((size_t)v.n_pts, 11 * (size_t)v.n_cams)), L.item_block, 0, s>>>(v, c, use);
}
void launch64_direction(const V64& v, const LaunchCfg& L, cudaStream_t s, const double* zs, int use_beta,
                        const int32_t* gate) {
    k64_direction<<<g64(L, v.n_vec), L.item_block, 0, s>>>(v, zs, use_beta, gate);
}
void launch64_matvec(const V64& v, const LaunchCfg& L, cudaStream_t s, const int32_t* gate) {
    k64_matvec<<<tiles64(v), T64, 0, s>>>(v, gate);
}
void launch64_update(const V64& v, const LaunchCfg& L, cudaStream_t s, CondHandle c, int use) {
    k64_update<<<g64(L, std::max((size_t)v.n_pts, 11 * (size_t)v.n_cams)), L.item_block, 0, s>>>(v, c, use);
}
void launch64_candidate(const V64& v, const LaunchCfg& L, cudaStream_t s) {
    k64_candidate<<<g64(L, v.n_vec), L.item_block, 0, s>>>(v);
}
void launch64_eval_candidate(const V64& v, const LaunchCfg& L, cudaStream_t s, CondHandle c, int use) {
    k64_eval_candidate<<<tiles64(v), T64, 0, s>>>(v, c, use);
}
void launch64_commit(const V64& v, const LaunchCfg& L, cudaStream_t s) {
    k64_commit<<<g64(L, v.n_vec), L.item_block, 0, s>>>(v);
}
void launch64_pack(const V64& v, const LaunchCfg& L, cudaStream_t s, const void* cams, const void* pts, int dtype) {
    const int g = g64(L, std::max(v.n_cams, v.n_pts));
    if (dtype == 1) k64_pack<double><<<g, L.item_block, 0, s>>>(v, (const double*)cams, (const double*)pts);
    else k64_pack<float><<<g, L.item_block, 0, s>>>(v, (const float*)cams, (const float*)pts);
}
void launch64_unpack(const V64& v, const LaunchCfg& L, cudaStream_t s, void* cams, void* pts, int dtype) {
    const int g = g64(L, std::max(v.n_cams, v.n_pts));
    if (dtype == 1) k64_unpack<double><<<g, L.item_block, 0, s>>>(v, (double*)cams, (double*)pts);
    else k64_unpack<float><<<g, L.item_block, 0, s>>>(v, (float*)cams, (float*)pts);
}
void launch64_set_vec(const V64& v, const LaunchCfg& L, cudaStream_t s, const double* src, double* dst) {
    k64_set_vec<<<g64(L, std::max(v.n_cams, v.n_pts)), L.item_block, 0, s>>>(v, src, dst);
}
void launch64_cost_grad(const V64& v, const LaunchCfg& L, cudaStream_t s, const void* cams, const void* pts, int dtype,
                        int want_grad, double* cost_dev) {
    const int g = g64(L, std::max(v.n_cams, v.n_pts));
    if (dtype == 1) k64_pack_to<double><<<g, L.item_block, 0, s>>>(v, (const double*)cams, (const double*)pts, v.x_new);
    else k64_pack_to<float><<<g, L.item_block, 0, s>>>(v, (const float*)cams, (const float*)pts, v.x_new);
    k64_records_from<<<g64(L, v.n_cams), L.item_block, 0, s>>>(v, v.x_new, v.cam64_new);
    k64_cost_grad<<<g64(L, v.n_pts), L.item_block, 0, s>>>(v, v.x_new, v.cam64_new, want_grad, cost_dev);
}
void launch64_grad_out(const V64& v, const LaunchCfg& L, cudaStream_t s, const double* grad_out, void* gc, void* gp,
                       int dtype) {
    const int g = g64(L, std::max(v.n_cams, v.n_pts));
    if (dtype == 1) k64_grad_out<double><<<g, L.item_block, 0, s>>>(v, grad_out, (double*)gc, (double*)gp);
    else k64_grad_out<float><<<g, L.item_block, 0, s>>>(v, grad_out, (float*)gc, (float*)gp);
}
void launch64_get_vec(const V64& v, const LaunchCfg& L, cudaStream_t s, const double* src, double* dst) {
    k64_get_vec<<<g64(L, std::max(v.n_cams, v.n_pts)), L.item_block, 0, s>>>(v, src, dst);
}

}  // namespace gbba
