// Persistent PCGNR (Sec. V-A of arXiv 2605.30583) for problems whose tiles fit in the
// GPU's aggregate shared memory.
//
// One cooperative launch runs every PCG iteration of one LM step.  The grid is one
// CTA per SM; CTA b owns a contiguous run of tiles (balanced by observation count)
// and keeps, for the whole solve, its observation keys and its points' X, D, M^-1
// and PCG vectors in shared memory.  Grid-wide sums travel through an exchange: every CTA
// publishes its sums and waits for those of all others, which it adds up in the same
// order and so takes the same stop decision.  Every wait is time-bounded: on a
// time-out the CTA sets an error flag, every CTA leaves, and the solve reports
// BA_ERR_TIMEOUT.
//
// Two forms of the same Krylov iteration:
//
// k_pcg_persistent (pcg_kernel 0): the textbook recurrences, two exchanges per iteration:
//   A  p = z + beta p (points in smem; cameras double-buffered in global), then
//      q = J^T J p + mu D p with |J p|^2 and p^T D p;            -> exchange
//   B  alpha = r^T z / (|J p|^2 + mu p^T D p); h += alpha p; r -= alpha q; z = M^-1 r;
//      r^T z, |r|^2                                              -> exchange
//   C  stop test (|r| <= tol |r_0| or the iteration cap), beta.
//
// k_pcg_persistent_1x (the default): one exchange per iteration.  The recurrences are arranged as in
// the CG of Chronopoulos and Gear (J. Comput. Appl. Math. 25, 1989): with u = M^-1 r,
// w = A u and s = A p carried by s = w + beta s,
//   gamma = r^T u,  delta = u^T A u = |J u|^2 + mu u^T D u,
//   beta = gamma / gamma_prev,  alpha = gamma / (delta - beta gamma / alpha_prev),
// so both inner products of an iteration come out of the one exchange that follows
// the operator.  Each CTA keeps its own copy of the camera vectors it touches and
// updates them from the assembled camera sums of the operator, so no second exchange
// publishes them; the one CTA that owns a camera adds it to the inner products and
// writes its step.  Same iterates in exact arithmetic; in FP32 the recurrence for s
// lets the updated residual drift from the true one sooner.
//   M  w = J^T W J u: point part in shared memory, camera part into one of three
//      rotating accumulator sets; |J u|^2 with the partials of the previous update;
//   X  exchange: gamma, |r|^2, u^T D u, |J u|^2 over the grid; stop test, alpha, beta;
//   U  p = u + beta p, s = w + beta s, h += alpha p, r -= alpha s, u = M^-1 r.
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "kernels.h"
#include "mixed_common.cuh"

namespace gbba {

namespace {

// The limit of a wait for other CTAs, asked by one thread after each poll that found something
// missing: true when the wait is over because it ran out of time (the shared error word is then
// set) or another CTA's did.  Limits below 1 ms are checked at every poll (0: give up at the first
// one), longer ones every 64th; the limit counts from the first check, so a wait that ends
// sooner never reads the (slow) timer.
struct WaitLimit {
    int* err;
    long long limit_ns, t0 = -1;
    unsigned spins = 0;
    __device__ __forceinline__ bool over() {
        if (limit_ns >= 1000000LL && (++spins & 63u) != 0u) return false;
        if (*reinterpret_cast<volatile int*>(err)) return true;
        const long long now = global_ns();
        if (t0 < 0) t0 = now;
        if (now - t0 < limit_ns) return false;
        atomicExch(err, 1);
        return true;
    }
};

// One published FP64 sum: each half of it in a 64-bit word with the exchange's number in the upper
// 32 bits (64-bit accesses are not torn, so a reader needs no order between the words).
__device__ __forceinline__ void publish(ulonglong2* to, double x, uint32_t epoch) {
    const unsigned long long e = (unsigned long long)epoch << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(to), "l"(e | (uint32_t)__double2hiint(x)),
                 "l"(e | (uint32_t)__double2loint(x))
                 : "memory");
}

// Waits until the sums of `n` <= MAX_PBLOCKS CTAs at `from` carry `epoch` and adds them up, in the
// same order in every CTA; one warp, the total in every lane.  False when the wait's limit ran out.
__device__ __forceinline__ bool gather(const ulonglong2* from, int n, uint32_t epoch, WaitLimit limit, double& sum) {
    constexpr int PER = MAX_PBLOCKS / 32;
    const int lane = threadIdx.x & 31;
    double x[PER];
    unsigned missing = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        x[i] = 0.0;
        if (lane + 32 * i < n) missing |= 1u << i;
    }
    for (;;) {
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (missing >> i & 1u) {
                unsigned long long a, b;
                asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(from + lane + 32 * i) : "memory");
                if ((uint32_t)(a >> 32) == epoch && (uint32_t)(b >> 32) == epoch) {
                    x[i] = __hiloint2double((int)(uint32_t)a, (int)(uint32_t)b);
                    missing &= ~(1u << i);
                }
            }
        if (__all_sync(FULL, missing == 0u)) break;
        int over = 0;
        if (lane == 0) over = limit.over() ? 1 : 0;
        if (__shfl_sync(FULL, over, 0)) return false;
    }
    // a tree over the lane's values, then over the lanes; an FP64 addition is ~130 cycles, so none
    // for values that the grid does not have
#pragma unroll
    for (int o = 1; o < PER; o <<= 1)
#pragma unroll
        for (int i = 0; i + o < PER; i += 2 * o)
            if (32 * (i + o) < n) x[i] += x[i + o];
    sum = x[0];
    for (int o = 1; o < 32 && o < n; o <<= 1) sum += __shfl_xor_sync(FULL, sum, o);
    return true;
}

// What the CTA does after an exchange, decided by one thread for all.  FP64 runs at 1/64 of
// the FP32 rate on this GPU: a warp instruction holds its pipe for 16 cycles, so scalar
// recurrences repeated by all 16 warps cost 4-5 us per iteration; here one lane runs them.
enum : int { ACT_STOP = 0, ACT_UPDATE, ACT_VERIFY, ACT_TIMEOUT };
struct PcgStep {
    int act;
    float alpha, beta;
};

// Grid-wide sums of XCH_NV per-warp values, the grid barrier, and the decision.  red holds the
// CTA's compensated partials, value k of warp w at red[NW k + w]; with `last_only` the values
// before the last count as zero.  Warp k adds up the CTA's value k and publishes it with the
// number of the exchange, then gathers the value k of every CTA: there is no counter to arrive
// at and no second read, the sums themselves say that their CTA has arrived.  (Slot-spread FP64
// atomics, a release on a counter, the wait and the read of the slots: ~5.5 us.)  Two sets of
// words alternate: a CTA that publishes exchange e + 2 has seen every CTA's e + 1, which each
// published after reading all of e.  What the CTAs wrote before (camera sums) is visible after:
// the last value's publisher and readers carry the fences.  The sums are FP64 from the warps on:
// float pairs took 0.64 us less an exchange (the solve of 16 cameras and 1,000 points 1,062 us, so
// 1,130), but the squares of a residual can add up beyond FP32 although no warp's part does.
// Thread 0 calls decide(totals), which
// writes the shared step.  Call with the partials published (a barrier before); returns after
// a barrier.
template <int NW, typename F>
__device__ __forceinline__ void exchange(DevState* st, ulonglong2* words, uint32_t epoch, const float2* red,
                                         bool last_only, PcgStep* step, F&& decide) {
    static_assert(NW >= XCH_NV && NW <= 32 && (NW & (NW - 1)) == 0, "a warp per value, a lane per warp");
    __shared__ double s_tot[XCH_NV];
    __shared__ int s_ok[XCH_NV];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w < XCH_NV) {
        const bool last = w == XCH_NV - 1;
        ulonglong2* cur = words + (size_t)((epoch & 1u) * XCH_NV + w) * MAX_PBLOCKS;
        double x = 0.0;
        if (lane < NW && (last || !last_only)) {
            const float2 p = red[NW * w + lane];
            x = widen(p.x) + widen(p.y);
        }
#pragma unroll
        for (int o = NW / 2; o > 0; o >>= 1) x += __shfl_down_sync(FULL, x, o);
        if (lane == 0) {
            if (last) asm volatile("fence.acq_rel.gpu;" ::: "memory");
            publish(cur + blockIdx.x, x, epoch);
        }
        __syncwarp();
        const bool ok = gather(cur, gridDim.x, epoch, WaitLimit{&st->bar_err, st->opt.wait_ns}, x);
        if (last) asm volatile("fence.acq_rel.gpu;" ::: "memory");
        if (lane == 0) {
            s_tot[w] = x;
            s_ok[w] = ok;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * XCH_NV) : "memory");
        if (threadIdx.x == 0) {
            double tot[XCH_NV];
            bool all = true;
#pragma unroll
            for (int i = 0; i < XCH_NV; ++i) {
                tot[i] = s_tot[i];
                all = all && s_ok[i] != 0;
            }
            if (all) decide(tot);
            else step->act = ACT_TIMEOUT;
        }
    }
    __syncthreads();
}

// Tests on the high word, off the chain of FP64 operations.
__device__ __forceinline__ bool finite64(double x) { return ((uint32_t)__double2hiint(x) & 0x7fffffffu) < 0x7ff00000u; }
__device__ __forceinline__ bool positive_finite64(double x) {
    return (uint32_t)__double2hiint(x) - 1u < 0x7ff00000u - 1u;
}

// Local index of camera c in the CTA's sorted camera list (c must be listed).
__device__ __forceinline__ uint32_t local_cam(const uint32_t* sCid, uint32_t ncb, uint32_t c) {
    uint32_t lo = 0, hi = ncb;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (sCid[mid] <= c) lo = mid; else hi = mid;
    }
    return lo;
}

// CTA b's pose factors [f0, f1) through the operator (both cameras of each are in the CTA's
// list): returns this thread's part of |J_f d|^2.
__device__ __forceinline__ float factor_pass(const Views<float>& v, const uint32_t* sCid, uint32_t ncb,
                                          const float* sDir, float* acc, uint32_t f0, uint32_t f1) {
    float jj = 0.0f;
    for (uint32_t k = f0 + threadIdx.x; k < f1; k += blockDim.x) {
        const uint32_t ca = v.fac_cam[2 * (size_t)k], cb = v.fac_cam[2 * (size_t)k + 1];
        jj += factor_normal(v.fac_J + 72 * (size_t)k, sDir + 12 * local_cam(sCid, ncb, ca),
                            sDir + 12 * local_cam(sCid, ncb, cb), acc + (size_t)ca * CA_STRIDE,
                            acc + (size_t)cb * CA_STRIDE);
    }
    return jj;
}

// The CTA's tiles: block-local first observation, first short-run observation, and the number
// of long- and short-run observations in the tiles before.
struct TileTab {
    uint32_t lo[MAX_CTA_TILES + 1], ss[MAX_CTA_TILES], nl[MAX_CTA_TILES + 1], ns[MAX_CTA_TILES + 1];
};

__device__ __forceinline__ void make_tile_tab(const Views<float>& v, uint32_t t0, int tiles, uint32_t ob, TileTab& T) {
    if (threadIdx.x != 0) return;
    uint32_t nl = 0, ns = 0;
    for (int t = 0; t < tiles; ++t) {
        const uint32_t lo = v.tile_off[t0 + t], ss = v.short_start[t0 + t], hi = v.tile_off[t0 + t + 1];
        T.lo[t] = lo - ob;
        T.ss[t] = ss - ob;
        T.nl[t] = nl;
        T.ns[t] = ns;
        nl += ss - lo;
        ns += hi - ss;
        T.lo[t + 1] = hi - ob;
    }
    T.nl[tiles] = nl;
    T.ns[tiles] = ns;
}

// A camera's records from the CTA's tables (128-bit shared loads; both arrays are 16-byte
// aligned).
__device__ __forceinline__ void resident_cam(const float* sCam, const float* sDir, uint32_t lc, OpCam& oc, OpDir& od) {
    const float4* r4 = reinterpret_cast<const float4*>(sCam + 16 * lc);
    const float4 ra = r4[0], rb = r4[1], rc = r4[2], rd = r4[3];
    Cam cam;
    cam.R[0] = ra.x; cam.R[1] = ra.y; cam.R[2] = ra.z; cam.R[3] = ra.w;
    cam.R[4] = rb.x; cam.R[5] = rb.y; cam.R[6] = rb.z; cam.R[7] = rb.w;
    cam.R[8] = rc.x; cam.t[0] = rc.y; cam.t[1] = rc.z; cam.t[2] = rc.w;
    cam.f = rd.x; cam.k1 = rd.y; cam.k2 = rd.z;
    const float4* d4 = reinterpret_cast<const float4*>(sDir + 12 * lc);
    const float4 da = d4[0], db = d4[1], dc = d4[2];
    const float dir[9] = {da.x, da.y, da.z, da.w, db.x, db.y, db.z, db.w, dc.x};
    oc = op_cam(cam);
    od = op_dir(cam, dir);
}

// The normal operator over the CTA's observations (the keys carry CTA-local camera indices):
// points and directions from shared memory, point sums into sQ, camera sums into `cacc`.  Bound
// by latency: 16 warps, each a serial chain of keys, points and shared atomics.  Every thread
// takes an equal contiguous chunk of the long runs' observations (it meets few cameras there) and
// one of the short runs' (nearly every observation another camera): with one chunk over both, the
// two warps that held a tile's short runs took three times as long as the others (20k against
// 7k cycles on 200 cameras and 50,000 points) and the grid waited for them; 688 -> 667 us per 50
// iterations there.  One short-run observation per thread and step, neighbouring lanes of a camera
// combined by shuffles, took 961 us.
template <int TB>
__device__ __forceinline__ void resident_normal(const Views<float>& v, const uint32_t* skey, const float4* sX4,
                                                const float4* sD4, float* sQ, const TileTab& T, int tiles,
                                                const uint32_t* sCid, const float* sCam, const float* sDir, float* cacc,
                                                uint32_t ob, float eps, bool weighted, float& js, float& jc) {
    const bool general = weighted || eps != 0.0f;
    uint32_t cur = NO_CAM;
    float acc[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) acc[q] = 0.0f;
    OpCam oc;
    OpDir od;
    for (int part = 0; part < 2; ++part) {
        const uint32_t* cnt = part ? T.ns : T.nl;
        const uint32_t* first = part ? T.ss : T.lo;
        const uint32_t n = cnt[tiles], chunk = odd_chunk<uint32_t>(n, TB);
        const uint32_t a = min(threadIdx.x * chunk, n), b = min(a + chunk, n);
        int t = -1;
        uint32_t tend = 0, off = 0;
        for (uint32_t i = a; i < b; ++i) {
            while (i >= tend) {
                ++t;
                off = first[t] - cnt[t];
                tend = cnt[t + 1];
            }
            const uint32_t j = i + off;
            const uint32_t key = skey[j], lc = key >> 8;
            if (lc != cur) {
                if (cur != NO_CAM) {
                    op_finish(oc, sCam[16 * cur + CP_K1], sCam[16 * cur + CP_K2], acc);
                    flush_matvec(cacc + (size_t)sCid[cur] * CA_STRIDE, acc);
                }
                cur = lc;
                resident_cam(sCam, sDir, lc, oc, od);
            }
            const int lp = t * v.tile_pts + (int)(key & 0xffu);
            const float4 x = sX4[lp], dx = sD4[lp];
            const float tt = general ? obs_normal<true>(oc, od, x, dx, eps, weighted ? __ldg(v.obs_w + ob + j) : 1.0f,
                                                        acc, sQ + 3 * lp)
                                     : obs_normal<false>(oc, od, x, dx, 0.0f, 1.0f, acc, sQ + 3 * lp);
            kahan_add(js, jc, tt);
        }
    }
    if (cur != NO_CAM) op_finish(oc, sCam[16 * cur + CP_K1], sCam[16 * cur + CP_K2], acc);
    // every lane of the warp reaches this one collective
    const bool head = seg_reduce<9>(cur, acc);
    if (head && cur != NO_CAM) flush_matvec(cacc + (size_t)sCid[cur] * CA_STRIDE, acc);
}

}  // namespace

template <int TB>
__global__ void __launch_bounds__(TB, 1) k_pcg_persistent(Views<float> v, const uint32_t* __restrict__ blk_tile,
                                                         const uint32_t* __restrict__ blk_cam_off,
                                                         const uint32_t* __restrict__ blk_cams,
                                                         const uint32_t* __restrict__ blk_fac,
                                                         ulonglong2* __restrict__ words) {
    const uint32_t f0 = __ldg(blk_fac + blockIdx.x), f1 = __ldg(blk_fac + blockIdx.x + 1);
    DevState* st = v.st;
    if (st->pcg_active == 0) return;
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int CAMS_PER_PASS = TB / 9;
    constexpr int NW = TB / 32;
    __shared__ float2 red[XCH_NV * NW];
    __shared__ PcgStep step;
    __shared__ float s_cam_r[9 * CAMS_PER_PASS];
    const int tid = threadIdx.x;
    // cameras owned by this CTA: blockIdx.x + gridDim.x * j, j < n_own
    const int n_own = v.n_cams > (int)blockIdx.x ? (v.n_cams - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const uint32_t t0 = blk_tile[blockIdx.x], t1 = blk_tile[blockIdx.x + 1];
    const int tiles = (int)(t1 - t0);
    __shared__ TileTab tab;
    const uint32_t ob = v.tile_off[t0], oe = v.tile_off[t1];
    const uint32_t no = oe - ob;
    const int pb = (int)t0 * v.tile_pts;
    const int pe = min((int)t1 * v.tile_pts, v.n_pts);
    const int np = pe > pb ? pe - pb : 0;
    const int n3 = 3 * np;
    const int n3p = (n3 + 3) & ~3;
    uint32_t* skey = reinterpret_cast<uint32_t*>(smem);
    // X and p of the CTA's points as (x, y, z, 0) quadruples: one 128-bit load each
    float4* sX4 = reinterpret_cast<float4*>(smem + (((size_t)no * 4 + 15) & ~(size_t)15));
    float4* sP4 = sX4 + np;
    float* sD = reinterpret_cast<float*>(sP4 + np);
    float* sR = sD + n3p;
    float* sZ = sR + n3p;
    float* sH = sZ + n3p;
    float* sQ = sH + n3p;
    float* sM = sQ + n3p;   // 6 per point
    // cameras seen by this CTA (sorted): records (R, t, f, k1, k2) and direction records
    const uint32_t cb = blk_cam_off[blockIdx.x], ncb = blk_cam_off[blockIdx.x + 1] - cb;
    uint32_t* sCid = reinterpret_cast<uint32_t*>(sM + ((6 * np + 3) & ~3));
    float* sCam = reinterpret_cast<float*>(sCid + ((ncb + 3) & ~3u));   // 16 per camera
    float* sDir = sCam + 16 * (size_t)ncb;                              // 12 per camera
    const size_t g0 = v.pt_off + 3 * (size_t)pb;
    make_tile_tab(v, t0, tiles, ob, tab);
    for (uint32_t i = tid; i < ncb; i += TB) sCid[i] = __ldg(blk_cams + cb + i) & ~BLK_CAM_OWNER;
    for (uint32_t i = tid; i < 16 * ncb; i += TB)
        sCam[i] = __ldg(v.cam_pre + (size_t)(__ldg(blk_cams + cb + i / 16) & ~BLK_CAM_OWNER) * CP_STRIDE + i % 16);
    for (uint32_t i = tid; i < no; i += TB) skey[i] = __ldg(v.obs_key + ob + i);
    for (int i = tid; i < n3; i += TB) {
        sD[i] = v.D[g0 + i];
        sR[i] = v.r[g0 + i];
        sZ[i] = v.z[g0 + i];
        sH[i] = 0.0f;
    }
    for (int i = tid; i < np; i += TB) {
        sX4[i] = make_float4(v.x[g0 + 3 * i], v.x[g0 + 3 * i + 1], v.x[g0 + 3 * i + 2], 0.0f);
        sP4[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    for (int i = tid; i < 6 * np; i += TB) sM[i] = v.Minv_p[6 * (size_t)pb + i];
    __syncthreads();
    // keys carry the CTA-local camera index from here on (no search in the loop)
    for (uint32_t i = tid; i < no; i += TB) {
        const uint32_t key = skey[i];
        skey[i] = (local_cam(sCid, ncb, key >> 8) << 8) | (key & 0xffu);
    }
    __syncthreads();

    const double mu = st->mu;
    const float muf = (float)mu;
    const float eps = (float)st->opt.eps;
    const bool weighted = st->opt.loss != 0;   // robust loss: IRLS weights per observation
    const int max_pcg = st->opt.max_pcg;
    // the recurrences' scalars, kept by thread 0 (lane 0 of the deciding warp)
    double rz = st->rz, rr = st->rr0, alpha = 0.0, beta_d = 0.0;
    const double stop_rr = st->opt.tol * st->opt.tol * rr;
    bool numeric_fail = false;
    float beta = 0.0f;
    uint32_t epoch = 0u;
    int k = 0;
    bool ok = true;
    for (int i = tid; i < XCH_NV * NW; i += TB) red[i] = make_float2(0.0f, 0.0f);

    while (k < max_pcg) {
        const float* pc_old = v.pc + (size_t)(k & 1) * v.pc_stride;
        float* pc_new = v.pc + (size_t)((k & 1) ^ 1) * v.pc_stride;
        // ------------------------------------------------------------ phase A
        float pdp = 0.0f, pdpc = 0.0f, jp2 = 0.0f, jp2c = 0.0f;   // Kahan pairs
        // direction records of this CTA's cameras: p_c = z_c + beta p_prev_c, phi = J_l p_w
        // (global loads first, so their latency overlaps the point loop below)
        for (uint32_t i = tid; i < ncb; i += TB) {
            float dir[9];
            camera_dir(v, sCid[i], v.z, pc_old, beta, dir);
#pragma unroll
            for (int q = 0; q < 9; ++q) sDir[12 * i + q] = dir[q];
        }
        // owned cameras (b, b + G, ...): one thread per vector entry, all in parallel
        for (int idx = tid; idx < 9 * n_own; idx += TB) {
            const int c = blockIdx.x + (int)gridDim.x * (idx / 9);
            const size_t e = 9 * (size_t)c + idx % 9;
            const float zc = __ldcg(v.z + e);
            const float pk = beta != 0.0f ? fmaf(beta, __ldcg(pc_old + e), zc) : zc;
            pc_new[e] = pk;
            kahan_add(pdp, pdpc, __ldg(v.D + e) * pk * pk);
        }
        for (int i = tid; i < np; i += TB) {
            const float4 po = sP4[i];
            const float p0 = fmaf(beta, po.x, sZ[3 * i]);
            const float p1 = fmaf(beta, po.y, sZ[3 * i + 1]);
            const float p2 = fmaf(beta, po.z, sZ[3 * i + 2]);
            sP4[i] = make_float4(p0, p1, p2, 0.0f);
            sQ[3 * i] = 0.0f;
            sQ[3 * i + 1] = 0.0f;
            sQ[3 * i + 2] = 0.0f;
            kahan_add(pdp, pdpc, fmaf(sD[3 * i] * p0, p0, fmaf(sD[3 * i + 1] * p1, p1, sD[3 * i + 2] * p2 * p2)));
        }
        __syncthreads();
        resident_normal<TB>(v, skey, sX4, sP4, sQ, tab, tiles, sCid, sCam, sDir, v.cam_acc, ob, eps, weighted, jp2, jp2c);
        if (v.n_fac > 0) kahan_add(jp2, jp2c, factor_pass(v, sCid, ncb, sDir, v.cam_acc, f0, f1));
        {
            const float2 a = warp_pair(jp2, -jp2c), b = warp_pair(pdp, -pdpc);
            if ((tid & 31) == 0) {
                red[tid >> 5] = a;
                red[NW + (tid >> 5)] = b;
            }
        }
        __syncthreads();
        exchange<NW>(st, words, ++epoch, red, false, &step, [&](const double (&tot)[XCH_NV]) {
            const double denom = tot[0] + mu * tot[1];
            if (!positive_finite64(denom)) {
                numeric_fail = !finite64(denom);
                step.act = ACT_STOP;
            } else {
                alpha = rz * rcp64(denom);
                step.act = ACT_UPDATE;
                step.alpha = (float)alpha;
            }
        });
        // ------------------------------------------------------------ phase B
        if (step.act != ACT_UPDATE) {   // every CTA takes the same step
            ok = step.act != ACT_TIMEOUT;
            break;
        }
        const float af = step.alpha;
        float lrz = 0.0f, lrzc = 0.0f, lrr = 0.0f, lrrc = 0.0f;   // Kahan pairs
        // points: all of it in shared memory
        auto update_points = [&]() {
            for (int i = tid; i < np; i += TB) {
                const int e = 3 * i;
                const float4 p4 = sP4[i];
                const float pq[3] = {p4.x, p4.y, p4.z};
                float r3[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const float pk = pq[q];
                    sH[e + q] = fmaf(af, pk, sH[e + q]);
                    r3[q] = fmaf(-af, fmaf(muf, sD[e + q] * pk, sQ[e + q]), sR[e + q]);
                    sR[e + q] = r3[q];
                }
                const float* m = sM + 6 * i;
                const float z0 = fmaf(m[0], r3[0], fmaf(m[1], r3[1], m[2] * r3[2]));
                const float z1 = fmaf(m[1], r3[0], fmaf(m[3], r3[1], m[4] * r3[2]));
                const float z2 = fmaf(m[2], r3[0], fmaf(m[4], r3[1], m[5] * r3[2]));
                sZ[e] = z0; sZ[e + 1] = z1; sZ[e + 2] = z2;
                kahan_add(lrz, lrzc, fmaf(r3[0], z0, fmaf(r3[1], z1, r3[2] * z2)));
                kahan_add(lrr, lrrc, fmaf(r3[0], r3[0], fmaf(r3[1], r3[1], r3[2] * r3[2])));
            }
        };
        if (n_own <= CAMS_PER_PASS) {
            // owned cameras in one pass, nine threads per camera (one per row); their
            // global loads go out before the point update, which hides their latency
            const int j = tid / 9, i = tid - 9 * j;
            const bool mine = j < n_own;
            const int c = blockIdx.x + (int)gridDim.x * j;
            const size_t e = 9 * (size_t)c + i;
            float qi = 0.0f, pk = 0.0f, hk = 0.0f, rk = 0.0f, dk = 0.0f;
            if (mine) {
                const float* ca = v.cam_acc + (size_t)c * CA_STRIDE;
                if (i < 3) {
                    const float* JL = v.cam_pre + (size_t)c * CP_STRIDE + CP_JL;
                    qi = fmaf(__ldg(JL + i), __ldcg(ca + 0), fmaf(__ldg(JL + 3 + i), __ldcg(ca + 1),
                                                              __ldg(JL + 6 + i) * __ldcg(ca + 2)));
                } else {
                    qi = __ldcg(ca + i);
                }
                pk = pc_new[e];
                hk = v.h[e];
                rk = v.r[e];
                dk = __ldg(v.D + e);
            }
            update_points();
            float ri = 0.0f;
            if (mine) {
                v.p[e] = pk;
                v.h[e] = fmaf(af, pk, hk);
                ri = fmaf(-af, fmaf(muf, dk * pk, qi), rk);
                v.r[e] = ri;
                s_cam_r[tid] = ri;
            }
            __syncthreads();
            if (mine) {
                const float* M = v.Minv_c + (size_t)c * MC_STRIDE + 9 * i;
                const float* rr9 = s_cam_r + 9 * j;
                float z = 0.0f;
#pragma unroll
                for (int q = 0; q < 9; ++q) z = fmaf(__ldg(M + q), rr9[q], z);
                v.z[e] = z;
                kahan_add(lrz, lrzc, ri * z);
                kahan_add(lrr, lrrc, ri * ri);
                v.cam_acc[(size_t)c * CA_STRIDE + i] = 0.0f;
            }
        } else {
            // owned cameras: nine threads per camera (one per row), CAMS_PER_PASS per pass
            for (int j0 = 0; j0 < n_own; j0 += CAMS_PER_PASS) {
                const int idx = tid;
                const int j = j0 + idx / 9, i = idx % 9;
                const bool mine = idx < 9 * CAMS_PER_PASS && j < n_own;
                const int c = blockIdx.x + (int)gridDim.x * j;
                const size_t e = 9 * (size_t)c + i;
                float ri = 0.0f;
                if (mine) {
                    const float* ca = v.cam_acc + (size_t)c * CA_STRIDE;
                    float qi;
                    if (i < 3) {
                        const float* JL = v.cam_pre + (size_t)c * CP_STRIDE + CP_JL;
                        qi = fmaf(__ldg(JL + i), __ldcg(ca + 0), fmaf(__ldg(JL + 3 + i), __ldcg(ca + 1),
                                                                  __ldg(JL + 6 + i) * __ldcg(ca + 2)));
                    } else {
                        qi = __ldcg(ca + i);
                    }
                    const float pk = pc_new[e];
                    v.p[e] = pk;
                    v.h[e] = fmaf(af, pk, v.h[e]);
                    ri = fmaf(-af, fmaf(muf, __ldg(v.D + e) * pk, qi), v.r[e]);
                    v.r[e] = ri;
                    s_cam_r[idx] = ri;
                }
                __syncthreads();
                if (mine) {
                    const float* M = v.Minv_c + (size_t)c * MC_STRIDE + 9 * i;
                    const float* rr9 = s_cam_r + 9 * (idx / 9);
                    float z = 0.0f;
#pragma unroll
                    for (int q = 0; q < 9; ++q) z = fmaf(__ldg(M + q), rr9[q], z);
                    v.z[e] = z;
                    kahan_add(lrz, lrzc, ri * z);
                    kahan_add(lrr, lrrc, ri * ri);
                    v.cam_acc[(size_t)c * CA_STRIDE + i] = 0.0f;
                }
                __syncthreads();
            }
            update_points();
        }
        {
            const float2 a = warp_pair(lrz, -lrzc), b = warp_pair(lrr, -lrrc);
            if ((tid & 31) == 0) {
                red[tid >> 5] = a;
                red[NW + (tid >> 5)] = b;
            }
        }
        __syncthreads();
        ++k;
        exchange<NW>(st, words, ++epoch, red, false, &step, [&](const double (&tot)[XCH_NV]) {
            // ------------------------------------------------------------ phase C
            const double rzn = tot[0];
            rr = tot[1];
            step.act = ACT_UPDATE;
            if (!finite64(rzn) || !finite64(rr)) {
                numeric_fail = true;
                step.act = ACT_STOP;
            } else if (rr <= stop_rr) {
                step.act = ACT_STOP;
            } else {
                beta_d = rzn * rcp64(rz);
                rz = rzn;
                step.beta = (float)beta_d;
            }
        });
        if (step.act != ACT_UPDATE) {
            ok = step.act != ACT_TIMEOUT;
            if (!ok) --k;
            break;
        }
        beta = step.beta;
    }
    // points' h back to global for the candidate step
    for (int i = tid; i < n3; i += TB) v.h[g0 + i] = sH[i];
    if (blockIdx.x == 0 && tid == 0) {
        st->pcg_iter = k;
        st->pcg_total += k;
        st->rz = rz;
        st->rr = rr;
        st->alpha = alpha;
        st->beta = beta_d;
        st->pcg_active = 0;
        if (!ok) st->status = 5;
        else if (numeric_fail) st->status = 4;
    }
}


// ------------------------------------------------------------ one-exchange form ---

namespace {


__device__ __forceinline__ bool owns(const uint32_t* sOwn, int lc) { return (sOwn[lc >> 5] >> (lc & 31)) & 1u; }

// Camera direction records (phi = J_l u_w, u_t, u_intr) of the CTA's cameras from u.
template <int TB>
__device__ __forceinline__ void camera_dirs(const Views<float>& v, const uint32_t* sCid, const float* sCu,
                                            float* sDir, int ne) {
    for (int e = threadIdx.x; e < ne; e += TB) {
        const int lc = e / 9, i = e - 9 * lc;
        float d;
        if (i < 3) {
            const float* JL = v.cam_pre + (size_t)sCid[lc] * CP_STRIDE + CP_JL + 3 * i;
            const float* u = sCu + 9 * lc;
            d = fmaf(__ldg(JL), u[0], fmaf(__ldg(JL + 1), u[1], __ldg(JL + 2) * u[2]));
        } else {
            d = sCu[e];
        }
        sDir[12 * lc + i] = d;
    }
}

// The CTA's tables of the one-exchange form (shared memory).
struct Tables1x {
    const float4* sX4;   // (X, D_0)
    float4* sU4;         // (u, D_1)
    const float* sD2;
    float *sP, *sS, *sR, *sH, *sQ;
    const float* sM;
    const uint32_t *sCid, *sOwn;
    float *sDir, *sCu, *sCp, *sCs, *sCr, *sCh;
};

// Update phase of the one-exchange form, from the assembled operator sums (points in sQ,
// cameras in the accumulator set `cacc`): w = A u, then p, s, h, r and u = M^-1 r; with
// TRUE_R (residual replacement) the sums are A h instead, r = b - A h with b = -g, and p, s,
// h are kept.  The cameras' direction records follow, the owner of a camera clears the
// accumulator set `clear` (filled by the iteration after next: its last readers are past
// the exchange), and the warps' partials of r^T u, |r|^2 and u^T D u go to `red`.
// A camera is nine lanes, three cameras a warp: its sums, r and u travel by shuffles, so no
// block barrier separates the steps.  The last warps take the cameras, the first ones hold
// the most points.
template <int TB, bool TRUE_R>
__device__ __forceinline__ void update_1x(const Views<float>& v, const Tables1x& T, const float* cacc, float* clear,
                                          int ncb, int np, size_t g0, float muf, float af, float beta, float2* red) {
    constexpr int NW = TB / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float lg = 0.0f, lr = 0.0f, lu = 0.0f, lgc = 0.0f, lrc = 0.0f, luc = 0.0f;   // Kahan pairs
    for (int cw = 3 * (NW - 1 - warp); cw < ncb; cw += 3 * NW) {
        const int sub = lane / 9, i = lane - 9 * sub, base = 9 * sub;
        const bool live = lane < 27 && cw + sub < ncb;
        const int lc = live ? cw + sub : cw;
        const int ii = live ? i : 0;
        const int e = 9 * lc + ii;
        const uint32_t c = T.sCid[lc];
        const float* JL = v.cam_pre + (size_t)c * CP_STRIDE + CP_JL;
        const float* M = v.Minv_c + (size_t)c * MC_STRIDE + 9 * ii;
        const float ca = __ldcg(cacc + (size_t)c * CA_STRIDE + ii);
        const float Dc = __ldg(v.D + 9 * (size_t)c + ii);
        float m[9], jc[3], jr[3];
#pragma unroll
        for (int q = 0; q < 9; ++q) m[q] = __ldg(M + q);
        const int i3 = ii < 3 ? ii : 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            jc[q] = __ldg(JL + 3 * q + i3);
            jr[q] = __ldg(JL + 3 * i3 + q);
        }
        const float c0 = __shfl_sync(FULL, ca, base), c1 = __shfl_sync(FULL, ca, base + 1);
        const float c2 = __shfl_sync(FULL, ca, base + 2);
        const float q = ii < 3 ? fmaf(jc[0], c0, fmaf(jc[1], c1, jc[2] * c2)) : ca;
        float r;
        if (TRUE_R) {
            r = (float)(-v.cam_lin[(size_t)c * CL_STRIDE + CL_G + ii]) - fmaf(muf, Dc * T.sCh[e], q);
        } else {
            const float u = T.sCu[e];
            const float pk = fmaf(beta, T.sCp[e], u);
            const float sk = fmaf(beta, T.sCs[e], fmaf(muf, Dc * u, q));
            r = fmaf(-af, sk, T.sCr[e]);
            if (live) {
                T.sCp[e] = pk;
                T.sCs[e] = sk;
                T.sCh[e] = fmaf(af, pk, T.sCh[e]);
            }
        }
        float z = 0.0f;
#pragma unroll
        for (int k = 0; k < 9; ++k) z = fmaf(m[k], __shfl_sync(FULL, r, base + k), z);
        const float z0 = __shfl_sync(FULL, z, base), z1 = __shfl_sync(FULL, z, base + 1);
        const float z2 = __shfl_sync(FULL, z, base + 2);
        if (live) {
            T.sCr[e] = r;
            T.sCu[e] = z;
            T.sDir[12 * lc + ii] = ii < 3 ? fmaf(jr[0], z0, fmaf(jr[1], z1, jr[2] * z2)) : z;
            if (owns(T.sOwn, lc)) {
                kahan_add(lg, lgc, r * z);
                kahan_add(lr, lrc, r * r);
                kahan_add(lu, luc, Dc * z * z);
                clear[(size_t)c * CA_STRIDE + ii] = 0.0f;
            }
        }
    }
    // points: all of it in shared memory
    for (int i = tid; i < np; i += TB) {
        const float4 u4 = T.sU4[i];
        const float Dq[3] = {T.sX4[i].w, u4.w, T.sD2[i]};
        const float uq[3] = {u4.x, u4.y, u4.z};
        float r3[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int e = 3 * i + q;
            if (TRUE_R) {
                r3[q] = -v.g[g0 + e] - fmaf(muf, Dq[q] * T.sH[e], T.sQ[e]);
            } else {
                const float pk = fmaf(beta, T.sP[e], uq[q]);
                const float sk = fmaf(beta, T.sS[e], fmaf(muf, Dq[q] * uq[q], T.sQ[e]));
                T.sP[e] = pk;
                T.sS[e] = sk;
                T.sH[e] = fmaf(af, pk, T.sH[e]);
                r3[q] = fmaf(-af, sk, T.sR[e]);
            }
            T.sQ[e] = 0.0f;
            T.sR[e] = r3[q];
        }
        const float* m = T.sM + 6 * i;
        const float z0 = fmaf(m[0], r3[0], fmaf(m[1], r3[1], m[2] * r3[2]));
        const float z1 = fmaf(m[1], r3[0], fmaf(m[3], r3[1], m[4] * r3[2]));
        const float z2 = fmaf(m[2], r3[0], fmaf(m[4], r3[1], m[5] * r3[2]));
        T.sU4[i] = make_float4(z0, z1, z2, u4.w);
        kahan_add(lg, lgc, fmaf(r3[0], z0, fmaf(r3[1], z1, r3[2] * z2)));
        kahan_add(lr, lrc, fmaf(r3[0], r3[0], fmaf(r3[1], r3[1], r3[2] * r3[2])));
        kahan_add(lu, luc, fmaf(Dq[0] * z0, z0, fmaf(Dq[1] * z1, z1, Dq[2] * z2 * z2)));
    }
    const float2 a = warp_pair(lg, -lgc), b = warp_pair(lr, -lrc), d = warp_pair(lu, -luc);
    if (lane == 0) {
        red[warp] = a;
        red[NW + warp] = b;
        red[2 * NW + warp] = d;
    }
}

}  // namespace

template <int TB>
__global__ void __launch_bounds__(TB, 1) k_pcg_persistent_1x(Views<float> v, const uint32_t* __restrict__ blk_tile,
                                                         const uint32_t* __restrict__ blk_cam_off,
                                                         const uint32_t* __restrict__ blk_cams,
                                                         const uint32_t* __restrict__ blk_fac,
                                                         ulonglong2* __restrict__ words) {
    const uint32_t f0 = __ldg(blk_fac + blockIdx.x), f1 = __ldg(blk_fac + blockIdx.x + 1);
    DevState* st = v.st;
    if (st->pcg_active == 0) return;
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int NW = TB / 32;
    __shared__ float2 red[XCH_NV * NW];   // r^T u, |r|^2, u^T D u (update phase), |J u|^2 (operator)
    __shared__ PcgStep step;
    const int tid = threadIdx.x;
    const uint32_t t0 = blk_tile[blockIdx.x], t1 = blk_tile[blockIdx.x + 1];
    const int tiles = (int)(t1 - t0);
    __shared__ TileTab tab;
    const uint32_t ob = v.tile_off[t0], oe = v.tile_off[t1];
    const uint32_t no = oe - ob;
    const int pb = (int)t0 * v.tile_pts;
    const int pe = min((int)t1 * v.tile_pts, v.n_pts);
    const int np = pe > pb ? pe - pb : 0;
    const int n3p = (3 * np + 3) & ~3;
    const uint32_t cb = blk_cam_off[blockIdx.x], ncb = blk_cam_off[blockIdx.x + 1] - cb;
    const int ne = 9 * (int)ncb;   // camera vector entries of this CTA
    // shared memory, carved in the order pcg_smem_bytes counts it
    uint32_t* skey = reinterpret_cast<uint32_t*>(smem);
    float4* sX4 = reinterpret_cast<float4*>(smem + (((size_t)no * 4 + 15) & ~(size_t)15));   // (X, D_0)
    float4* sU4 = sX4 + np;                                                                  // (u, D_1)
    float* sD2 = reinterpret_cast<float*>(sU4 + np);
    float* sP = sD2 + ((np + 3) & ~3);
    float* sS = sP + n3p;
    float* sR = sS + n3p;
    float* sH = sR + n3p;
    float* sQ = sH + n3p;
    float* sM = sQ + n3p;
    uint32_t* sCid = reinterpret_cast<uint32_t*>(sM + ((6 * np + 3) & ~3));
    uint32_t* sOwn = sCid + ((ncb + 3) & ~3u);
    float* sCam = reinterpret_cast<float*>(sOwn + ((((ncb + 31) >> 5) + 3) & ~3u));
    float* sDir = sCam + 16 * (size_t)ncb;
    float* sCu = sDir + 12 * (size_t)ncb;
    float* sCp = sCu + ne;
    float* sCs = sCp + ne;
    float* sCr = sCs + ne;
    float* sCh = sCr + ne;
    const size_t g0 = v.pt_off + 3 * (size_t)pb;
    const size_t cas = (size_t)CA_STRIDE * v.n_cams;   // floats between accumulator sets

    make_tile_tab(v, t0, tiles, ob, tab);
    for (uint32_t i = tid; i < ncb; i += TB) sCid[i] = __ldg(blk_cams + cb + i) & ~BLK_CAM_OWNER;
    for (uint32_t w = tid; w < (ncb + 31) / 32; w += TB) {
        uint32_t m = 0u;
        for (uint32_t j = 0; j < 32u && 32u * w + j < ncb; ++j)
            if (__ldg(blk_cams + cb + 32u * w + j) & BLK_CAM_OWNER) m |= 1u << j;
        sOwn[w] = m;
    }
    for (uint32_t i = tid; i < no; i += TB) skey[i] = __ldg(v.obs_key + ob + i);
    // partials of r^T u, |r|^2, u^T D u (Kahan pairs)
    float lg = 0.0f, lr = 0.0f, lu = 0.0f, lgc = 0.0f, lrc = 0.0f, luc = 0.0f;
    for (int i = tid; i < np; i += TB) {
        const size_t e = g0 + 3 * (size_t)i;
        const float D0 = v.D[e], D1 = v.D[e + 1], D2 = v.D[e + 2];
        const float u0 = v.z[e], u1 = v.z[e + 1], u2 = v.z[e + 2];
        const float r0 = v.r[e], r1 = v.r[e + 1], r2 = v.r[e + 2];
        sX4[i] = make_float4(v.x[e], v.x[e + 1], v.x[e + 2], D0);
        sU4[i] = make_float4(u0, u1, u2, D1);
        sD2[i] = D2;
        sR[3 * i] = r0; sR[3 * i + 1] = r1; sR[3 * i + 2] = r2;
        kahan_add(lg, lgc, fmaf(r0, u0, fmaf(r1, u1, r2 * u2)));
        kahan_add(lr, lrc, fmaf(r0, r0, fmaf(r1, r1, r2 * r2)));
        kahan_add(lu, luc, fmaf(D0 * u0, u0, fmaf(D1 * u1, u1, D2 * u2 * u2)));
    }
    for (int i = tid; i < n3p; i += TB) {
        sP[i] = 0.0f;
        sS[i] = 0.0f;
        sH[i] = 0.0f;
        sQ[i] = 0.0f;
    }
    for (int i = tid; i < 6 * np; i += TB) sM[i] = v.Minv_p[6 * (size_t)pb + i];
    __syncthreads();   // camera ids and owner bits
    // keys carry the CTA-local camera index from here on (no search in the loop)
    for (uint32_t i = tid; i < no; i += TB) {
        const uint32_t key = skey[i];
        skey[i] = (local_cam(sCid, ncb, key >> 8) << 8) | (key & 0xffu);
    }
    for (uint32_t i = tid; i < 16 * ncb; i += TB)
        sCam[i] = __ldg(v.cam_pre + (size_t)sCid[i / 16] * CP_STRIDE + i % 16);
    for (int e = tid; e < ne; e += TB) {
        const int lc = e / 9, i = e - 9 * lc;
        const size_t ge = 9 * (size_t)sCid[lc] + i;
        const float u = v.z[ge], r = v.r[ge];
        sCu[e] = u;
        sCr[e] = r;
        sCp[e] = 0.0f;
        sCs[e] = 0.0f;
        sCh[e] = 0.0f;
        if (owns(sOwn, lc)) {
            kahan_add(lg, lgc, r * u);
            kahan_add(lr, lrc, r * r);
            kahan_add(lu, luc, __ldg(v.D + ge) * u * u);
        }
    }
    {
        const float2 a = warp_pair(lg, -lgc), b = warp_pair(lr, -lrc), d = warp_pair(lu, -luc);
        if ((tid & 31) == 0) {
            red[tid >> 5] = a;
            red[NW + (tid >> 5)] = b;
            red[2 * NW + (tid >> 5)] = d;
        }
    }
    __syncthreads();   // camera u
    camera_dirs<TB>(v, sCid, sCu, sDir, ne);
    __syncthreads();
    const Tables1x T{sX4, sU4, sD2, sP, sS, sR, sH, sQ, sM, sCid, sOwn, sDir, sCu, sCp, sCs, sCr, sCh};

    const double mu = st->mu;
    const float muf = (float)mu;
    const float eps = (float)st->opt.eps;
    const bool weighted = st->opt.loss != 0;   // robust loss: IRLS weights per observation
    const int max_pcg = st->opt.max_pcg;
    // the recurrences' scalars, kept by thread 0 (lane 0 of the deciding warp)
    double gam = st->rz, igam = 0.0, alpha = 0.0, ialpha = 0.0, beta_d = 0.0, dprev = 0.0, rr = st->rr0;
    const double stop_rr = st->opt.tol * st->opt.tol * rr;
    bool numeric_fail = false;
    int checks = 0;
    uint32_t epoch = 0u;
    int k = 0;    // PCG updates
    int it = 0;   // operator passes (they rotate the camera accumulator sets)
    // Residual replacement (van der Vorst and Ye, SIAM J. Sci. Comput. 22, 2000): when the
    // recursively updated residual meets the tolerance, one operator pass on h gives the
    // true residual r = b - A h (b = -g), which replaces r (and u = M^-1 r) while the
    // search directions p, s are kept; the solve stops only on a true residual that
    // meets the tolerance.  At most MAX_CHECKS such checks per solve; past them the
    // recursive residual decides.
    constexpr int MAX_CHECKS = 4;
    bool verify = false;   // the coming operator pass applies A to h
    bool true_r = false;   // r was just replaced by the true residual
    bool ok = true;

    while (k < max_pcg) {
        float* cacc = v.cam_acc + (size_t)(it % CA_SETS) * cas;
        // ------------------------------------------------------------ M: w = A u (A h when verifying)
        float jj = 0.0f, jjc = 0.0f;   // Kahan pair
        resident_normal<TB>(v, skey, sX4, sU4, sQ, tab, tiles, sCid, sCam, sDir, cacc, ob, eps, weighted, jj, jjc);
        if (v.n_fac > 0) kahan_add(jj, jjc, factor_pass(v, sCid, ncb, sDir, cacc, f0, f1));
        const float2 jw = warp_pair(jj, -jjc);
        if ((tid & 31) == 0) red[3 * NW + (tid >> 5)] = jw;
        __syncthreads();
        // ------------------------------------------------------------ X: exchange
        exchange<NW>(st, words, ++epoch, red, verify, &step, [&](const double (&tot)[XCH_NV]) {
            if (verify) {   // a verification pass only assembles A h
                step.act = ACT_UPDATE;
                return;
            }
            const double g_k = tot[0], udu = tot[2], jju = tot[3];
            if (!finite64(g_k) || !finite64(tot[1])) {
                numeric_fail = true;
                step.act = ACT_STOP;
                return;
            }
            rr = tot[1];
            if (k > 0 && rr <= stop_rr) {
                // a true residual (or no checks left) ends the solve; else the recursive one is
                // checked against the true one: the next pass applies A to h
                step.act = true_r || checks >= MAX_CHECKS ? ACT_STOP : ACT_VERIFY;
                ++checks;
                return;
            }
            beta_d = k > 0 ? g_k * igam : 0.0;
            const double delta = jju + mu * udu;                                     // u^T A u
            const double denom = k > 0 ? fma(-beta_d, g_k * ialpha, delta) : delta;   // p^T A p
            if (!positive_finite64(denom)) {
                numeric_fail = !finite64(denom);
                step.act = ACT_STOP;
                return;
            }
            gam = g_k;
            // alpha and beta are used in FP32: of 10^8 random quotients none differs there from
            // the IEEE one, which takes 0.25 us longer each
            alpha = g_k * rcp64(denom);
            step.act = ACT_UPDATE;
            step.alpha = narrow(alpha);
            step.beta = narrow(beta_d);
            dprev = denom;   // 1 / gamma and 1 / alpha: taken off the other warps' path, below
        });
        const int act = step.act;   // every CTA takes the same step
        if (act == ACT_STOP || act == ACT_TIMEOUT) {
            ok = act == ACT_STOP;
            break;
        }
        if (act == ACT_VERIFY) {
            verify = true;
            for (int i = tid; i < np; i += TB) {
                sU4[i] = make_float4(sH[3 * i], sH[3 * i + 1], sH[3 * i + 2], sU4[i].w);
                // w = A u of the pass that found the tolerance met is not applied
                sQ[3 * i] = sQ[3 * i + 1] = sQ[3 * i + 2] = 0.0f;
            }
            float* clear = v.cam_acc + (size_t)((it + 2) % CA_SETS) * cas;   // as the update would
            for (int e = tid; e < ne; e += TB) {
                sCu[e] = sCh[e];
                const int lc = e / 9;
                if (owns(sOwn, lc)) clear[(size_t)sCid[lc] * CA_STRIDE + (e - 9 * lc)] = 0.0f;
            }
            __syncthreads();
            camera_dirs<TB>(v, sCid, sCu, sDir, ne);
            __syncthreads();
            ++it;
            continue;
        }
        float* clear = v.cam_acc + (size_t)((it + 2) % CA_SETS) * cas;
        if (verify) {
            // ---------------------------------------------------- R: r = b - A h, restart
            update_1x<TB, true>(v, T, cacc, clear, (int)ncb, np, g0, muf, 0.0f, 0.0f, red);
            verify = false;
            true_r = true;
        } else {
            // ------------------------------------------------------------ U: update
            if (tid == 0) {
                igam = rcp64(gam);
                ialpha = dprev * igam;
            }
            update_1x<TB, false>(v, T, cacc, clear, (int)ncb, np, g0, muf, step.alpha, step.beta, red);
            true_r = false;
            ++k;
        }
        __syncthreads();   // u and the direction records
        ++it;
    }
    // closing exchange: past it no CTA reads an accumulator set any more, so the
    // owners leave all of them cleared
    if (ok) {
        __syncthreads();
        exchange<NW>(st, words, ++epoch, red, true, &step, [&](const double (&)[XCH_NV]) { step.act = ACT_STOP; });
        ok = step.act != ACT_TIMEOUT;
    }
    for (int e = tid; e < ne; e += TB) {
        const int lc = e / 9, i = e - 9 * lc;
        if (!owns(sOwn, lc)) continue;
        const uint32_t c = sCid[lc];
        v.h[9 * (size_t)c + i] = sCh[e];
        if (ok)
            for (int set = 0; set < CA_SETS; ++set) v.cam_acc[set * cas + (size_t)c * CA_STRIDE + i] = 0.0f;
    }
    for (int i = tid; i < 3 * np; i += TB) v.h[g0 + i] = sH[i];
    if (blockIdx.x == 0 && tid == 0) {
        st->pcg_iter = k;
        st->pcg_total += k;
        st->rz = gam;
        st->rr = rr;
        st->alpha = alpha;
        st->beta = beta_d;
        st->pcg_active = 0;
        if (!ok) st->status = 5;
        else if (numeric_fail) st->status = 4;
    }
}

// ------------------------------------------------------------------ host ----------

int persistent_max_smem() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return v;
}

cudaError_t persistent_prepare(int form, int smem_bytes, int* blocks_per_sm) {
    const void* f = form == PCG_TWO_EXCHANGE ? (const void*)k_pcg_persistent<PCG_TB>
                                            : (const void*)k_pcg_persistent_1x<PCG_TB>;
    cudaError_t e = ensure_dynamic_smem(f, smem_bytes);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, f, PCG_TB, smem_bytes);
}

cudaError_t launch_pcg_persistent(const Views<float>& v, const uint32_t* blk_tile, const uint32_t* blk_cam_off,
                                  const uint32_t* blk_cams, const uint32_t* blk_fac, ulonglong2* words, int grid,
                                  int smem_bytes, int form, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(PCG_TB);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (form == PCG_TWO_EXCHANGE)
        return cudaLaunchKernelEx(&cfg, k_pcg_persistent<PCG_TB>, v, blk_tile, blk_cam_off, blk_cams, blk_fac, words);
    return cudaLaunchKernelEx(&cfg, k_pcg_persistent_1x<PCG_TB>, v, blk_tile, blk_cam_off, blk_cams, blk_fac, words);
}

// Self-test of the bounded wait: every CTA of a cooperative grid waits for a sum that nothing will
// ever publish.  Every CTA must give up after `timeout_ns`, set the shared error word and
// return; scratch = {unused (u64), error word (i32), CTAs that gave up (u32)}.
__device__ ulonglong2 selftest_words[1];

__global__ void k_selftest_wait(unsigned long long* scratch, long long timeout_ns) {
    int* err = reinterpret_cast<int*>(scratch + 1);
    if (threadIdx.x >= 32) return;
    double sum;
    const bool ok = gather(selftest_words, 1, 1u, WaitLimit{err, timeout_ns}, sum);
    if (!ok && threadIdx.x == 0) atomicAdd(reinterpret_cast<unsigned int*>(err) + 1, 1u);
}

__global__ void k_selftest_rcp64(const double* __restrict__ x, double* __restrict__ y, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = rcp64(x[i]);
}

void launch_selftest_rcp64(const double* x, double* y, int64_t n, cudaStream_t s) {
    const int64_t b = (n + 255) / 256;
    k_selftest_rcp64<<<(unsigned int)(b < 1024 ? b : 1024), 256, 0, s>>>(x, y, n);
}

__global__ void k_selftest_conversions(const float* __restrict__ x32, double* __restrict__ wide,
                                       const double* __restrict__ x64, float* __restrict__ narrowed, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        wide[i] = widen(x32[i]);
        narrowed[i] = narrow(x64[i]);
    }
}

void launch_selftest_conversions(const float* x32, double* wide, const double* x64, float* narrowed, int64_t n,
                                 cudaStream_t s) {
    const int64_t b = (n + 255) / 256;
    k_selftest_conversions<<<(unsigned int)(b < 1024 ? b : 1024), 256, 0, s>>>(x32, wide, x64, narrowed, n);
}

cudaError_t launch_selftest_wait(void* scratch, int grid, long long timeout_ns, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(64);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_selftest_wait, (unsigned long long*)scratch, timeout_ns);
}

}  // namespace gbba
