// Residual pass of the mixed-precision form: r = f s p - u of every observation (the
// Snavely reprojection factor of Sec. VI-A), written to v.rbuf in solver order, and the
// cost 1/2 sum rho(|r|^2) into st->F_res: every cost of the mixed form (F at the start
// of a solve, F' of a candidate, the evaluation's cost) comes from this one sum.
//
// Precision.  Everything else in the mixed form is FP32 with FP64 reductions, but the
// residual is a difference of ~500 px terms that cancel to ~1 px, so FP32 leaves it with
// an error of ~1e-4 px that depends on the parameters' last bits.  On problems with flat
// directions (points seen along nearly parallel rays) LM walks along them into places
// where those errors happen to lower the FP32 cost, and stops at parameters whose true
// cost is higher than the plain FP64 solver's optimum.  With res_df (the default) the
// residual is computed in double-float arithmetic (df.cuh) from the FP64 master
// parameters (points) and the double-float camera records, and only then rounded to
// FP32: the cost LM sees is then the true cost to ~1e-7 px per residual.  The Jacobian,
// the normal operator and PCG stay FP32.
//
// One CTA per tile (grid-stride): the tile's points are staged in shared memory, then
// the threads walk the tile's observations in order (coalesced keys, pixels and
// results); consecutive observations share their camera, whose records come through L1.
#include <cuda_runtime.h>

#include <algorithm>

#include "device_common.cuh"
#include "kernels.h"
#include "residual.cuh"

namespace gbba {
namespace {

constexpr int RS_TB = 256;

template <int TB>
__global__ void __launch_bounds__(TB, 5) k_residual(Views<float> v, int at_candidate, int squared) {
    DevState* st = v.st;
    // a candidate is only evaluated while LM runs (the decision kernel reads F' then)
    if (at_candidate && st->lm_active == 0) return;
    __shared__ float4 sXh[TILE_PTS], sXl[TILE_PTS];
    const double cost2 = residual_tiles<TB>(v, at_candidate, squared, blockIdx.x, gridDim.x, sXh, sXl);
    __shared__ double red[TB / 32];
    double in[1], out[1];
    in[0] = block_sum(cost2, red);
    if (grid_reduce_block<1>(in, v.partials, &st->tickets[TK_RES], out) && threadIdx.x == 0) st->F_res = 0.5 * out[0];
}

}  // namespace

void launch_residual(const Views<float>& v, const LaunchCfg& L, cudaStream_t s, int at_candidate, int squared) {
    const int grid = std::max(1, std::min({v.n_tiles, L.res_grid, MAX_GRID}));
    k_residual<RS_TB><<<grid, RS_TB, 0, s>>>(v, at_candidate, squared);
}

int occupancy_blocks_residual() {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_residual<RS_TB>, RS_TB, 0) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return std::max(1, n);
}

}  // namespace gbba
