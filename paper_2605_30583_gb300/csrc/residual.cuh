// The residual pass over tiles (residual.cu says what it computes and why), for the kernels that
// run it.
#pragma once

#include "device_common.cuh"
#include "df.cuh"

namespace gbba {

// Residuals of tiles first, first + stride, ... to v.rbuf; returns this thread's part of twice the
// cost.  sXh, sXl: TILE_PTS entries of shared memory each (the tile's points, double-float).
template <int TB>
__device__ __forceinline__ double residual_tiles(const Views<float>& v, int at_candidate, int squared, int first, int stride,
                                                 float4* sXh, float4* sXl) {
    DevState* st = v.st;
    const double* xm = at_candidate ? v.xm_new : v.xm;
    const float* rec = at_candidate ? v.cam_pre_new : v.cam_pre;
    const float* lor = at_candidate ? v.cam_lo_new : v.cam_lo;
    const float eps = (float)st->opt.eps;
    const int loss = squared ? 0 : st->opt.loss;
    const float lscale = (float)st->opt.loss_scale;
    const bool dfp = st->opt.res_df != 0;
    // the cost: Kahan pair of the high parts of |r|^2 (double-float |r|^2 before any
    // rounding, so F resolves steps far below an FP32 ulp of the residuals) and the sum
    // of their low parts
    float cs = 0.0f, cc = 0.0f, cl = 0.0f;
    for (int tile = first; tile < v.n_tiles; tile += stride) {
        const uint32_t lo = v.tile_off[tile], hi = v.tile_off[tile + 1];
        const int pt0 = tile * v.tile_pts;
        const int npt = min(v.tile_pts, v.n_pts - pt0);
        const size_t base = v.pt_off + 3 * (size_t)pt0;
        for (int i = threadIdx.x; i < npt; i += TB) {
            const DF a = df_from_double(xm[base + 3 * i]), b = df_from_double(xm[base + 3 * i + 1]),
                     c = df_from_double(xm[base + 3 * i + 2]);
            sXh[i] = make_float4(a.hi, b.hi, c.hi, 0.0f);
            sXl[i] = make_float4(a.lo, b.lo, c.lo, 0.0f);
        }
        __syncthreads();
        for (uint32_t j = lo + threadIdx.x; j < hi; j += TB) {
            const uint32_t key = __ldg(v.obs_key + j);
            const uint32_t c = key >> 8, slot = key & 0xffu;
            const float2 uv = __ldg(reinterpret_cast<const float2*>(v.obs_uv) + j);
            const float4 xh = sXh[slot];
            float r0, r1;
            DF s2 = {0.0f, 0.0f};
            if (dfp) {
                const float4 xl = sXl[slot];
                const CamDF cam = load_cam_df(rec + (size_t)c * CP_STRIDE, lor + (size_t)c * CLO_STRIDE);
                const DF X[3] = {{xh.x, xl.x}, {xh.y, xl.y}, {xh.z, xl.z}};
                DF d0, d1;
                residual_df(cam, X, eps, uv.x, uv.y, d0, d1);
                r0 = df_to_float(d0);
                r1 = df_to_float(d1);
                s2 = df_add(df_mul(d0, d0), df_mul(d1, d1));
            } else {
                const Cam cam = load_cam(rec + (size_t)c * CP_STRIDE);
                project_residual(cam, xh.x, xh.y, xh.z, eps, uv.x, uv.y, r0, r1);
                s2.hi = fmaf(r0, r0, r1 * r1);
            }
            reinterpret_cast<float2*>(v.rbuf)[j] = make_float2(r0, r1);
            if (loss) {   // robust loss: rho of the FP32-rounded |r|^2
                kahan_add(cs, cc, loss_rho(df_to_float(s2), loss, lscale));
            } else {
                kahan_add(cs, cc, s2.hi);
                cl += s2.lo;
            }
        }
        __syncthreads();   // the next tile's staging overwrites the points
    }
    return pair_sum(cs, cc) + widen(cl);
}

}  // namespace gbba
