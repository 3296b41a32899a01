// nr_rhs_kernels.cuh -- k_rhs and k_rhs_spread, their launch shapes and the rule that chooses among them;
// instantiated once per coordinate family and finite-difference order (nr_rhs_{sph,cyl}{,8}.cu) so the four
// compile in parallel.
#pragma once

#include "nr_stage.cuh"

namespace nrk {

// One RK stage (or, MODE_RHS, the right-hand side alone), one point per thread: each block takes 32 x RHS_WARPS
// consecutive interior points (i0 fastest), so that no lane idles at the ends of rows that are no multiple of 32:
// 77x10x131, 8th order: 619 -> 548 us against tiles of 32 x 4 points, 35x2x700: 265 -> 178 us, 100x50x60: 1.24 -> 1.03
// ms; rows of a multiple of 32 take the same time.  oa.nblocks further blocks take the pure-outer points: the first
// ones with BPS = 4, the last ones with BPS = 2, whose tiles then fill whole SMs and leave the light outer blocks
// beside them.
//
// Bound: the FP64 pipe (2 lanes a cycle per SM: 16 to 20 cycles per warp instruction), 81 % active on 256x2x512, with
// the difference sums on the integer pipe beside it (fixed_sum.cuh).  A warp does its integer passes first and its
// FP64 part after them; four blocks per SM (128 registers, 3 to 5 KB of spills) keep one warp of each scheduler in its
// FP64 part nearly always: 640 us per right-hand side on 256x2x512 when that was chosen, against 664 us with three
// (168 registers); two (255 registers, no spills) were 10 % slower.  All in FP64 arithmetic, two per scheduler, 865
// us, now 636; 8th order on the same grid 1137 -> 744 us; 192x96x192 spherical 15.66 -> 10.47 ms (4th), 23.2 -> 12.9 ms
// (8th).  Where no scheduler gets more than two warps, the 255 registers are the faster ones (rhs_shape).
constexpr int RHS_WARPS = 4;
template <int FAM, int AX, int ORD, int BPS>
__global__ void __launch_bounds__(32 * RHS_WARPS, BPS)
    k_rhs(GridK G, const double* __restrict__ yin, const double* __restrict__ d1x, const double* __restrict__ d1y,
          double* out, const double* yn, double* acc, Stage st, OuterArgs oa)
{
    const int ntile = (int)gridDim.x - oa.nblocks, first = BPS == 2 ? ntile : 0, ob = (int)blockIdx.x - first;
    if (ob >= 0 && ob < oa.nblocks) {
        const int t = ob * (32 * RHS_WARPS) + threadIdx.x;
        if (t < oa.npts)
            outer_point_stage<FAM, ORD, ssp_first_short<AX>()>(G, oa.pts[t], yin, out, yn, acc, oa.finf, oa.wspeed, st);
        return;
    }
    const int p = (BPS == 2 ? (int)blockIdx.x : ob - oa.nblocks) * (32 * RHS_WARPS) + threadIdx.x;
    if (p < G.N0 * G.N1 * G.N2)
        rhs_point_stage<FAM, AX, ORD>(G, yin, d1x, d1y, out, yn, acc, st, p % G.N0, p / G.N0);
}

// The same for grids of few points, whose time is one warp's way through its tile: a block of SPREAD_WARPS warps
// takes 32 consecutive interior points (i0 fastest) and divides the integer passes among its warps.  64x16x2: 90
// -> 66 us; 72x12x24: 187 -> 156 us (with k_d1 and the launches; the all-FP64 kernel took 83 and 196 us).
// BPS blocks per SM: with three (168 registers) a step is 3 to 10 % faster than with four (128 registers) where both
// run in one round; two are 3 % faster on the smallest grids and 35 % slower on 72x12x24.
template <int FAM, int AX, int ORD, int BPS>
__global__ void __launch_bounds__(32 * SPREAD_WARPS, BPS)
    k_rhs_spread(GridK G, const double* __restrict__ yin, const double* __restrict__ d1x,
                 const double* __restrict__ d1y, double* out, const double* yn, double* acc, Stage st, OuterArgs oa)
{
    __shared__ double tab[RawIx<AX>::N + NGF][32];
    __shared__ int slot;
    if ((int)blockIdx.x < oa.nblocks) {
        const int t = blockIdx.x * (32 * SPREAD_WARPS) + threadIdx.x;
        if (t < oa.npts)
            outer_point_stage<FAM, ORD, ssp_first_short<AX>()>(G, oa.pts[t], yin, out, yn, acc, oa.finf, oa.wspeed, st);
        return;
    }
    spread_slot(&slot);
    const int n = G.N0 * G.N1 * G.N2, p = (blockIdx.x - oa.nblocks) * 32 + (threadIdx.x & 31), q = p < n ? p : n - 1;
    rhs_spread_stage<FAM, AX, ORD>(G, yin, d1x, d1y, out, yn, acc, st, q % G.N0, q / G.N0, p < n, threadIdx.x / 32,
                                   slot, tab);
}

template <int FAM, int AX, int ORD>
cudaError_t launch_k_rhs(cudaStream_t s, const GridK& G, const double* yin, double* d1x, double* d1y, double* out,
                         const double* yn, double* acc, const Stage& st, const RhsLoad& load, OuterArgs oa)
{
    static_assert(RHS_WARPS == SPREAD_WARPS, "outer blocks of the same size");
    oa.nblocks = (oa.npts + 32 * RHS_WARPS - 1) / (32 * RHS_WARPS);
    const long n = (long)G.N0 * G.N1 * G.N2, tiles = (n + 31) / 32, blocks = (n + 32 * RHS_WARPS - 1) / (32 * RHS_WARPS);
    const unsigned ng = (unsigned)(blocks + oa.nblocks), ns = (unsigned)(tiles + oa.nblocks);
    switch (rhs_shape(FAM, ORD, AX >= 0, load)) {
    case RHS_SPREAD3: k_rhs_spread<FAM, AX, ORD, 3><<<ns, 32 * SPREAD_WARPS, 0, s>>>(G, yin, d1x, d1y, out, yn, acc, st, oa); break;
    case RHS_SPREAD4: k_rhs_spread<FAM, AX, ORD, 4><<<ns, 32 * SPREAD_WARPS, 0, s>>>(G, yin, d1x, d1y, out, yn, acc, st, oa); break;
    case RHS_POINTS2: k_rhs<FAM, AX, ORD, 2><<<ng, 32 * RHS_WARPS, 0, s>>>(G, yin, d1x, d1y, out, yn, acc, st, oa); break;
    default: k_rhs<FAM, AX, ORD, 4><<<ng, 32 * RHS_WARPS, 0, s>>>(G, yin, d1x, d1y, out, yn, acc, st, oa);
    }
    return cudaGetLastError();
}

// one translation unit per family and order defines, through NRK_RHS_LAUNCH, the launch for grids whose azimuth
// holds two points (two) or more
#define NRK_RHS_ARGS                                                                                              \
    bool two, cudaStream_t s, const GridK &G, const double *yin, double *d1x, double *d1y, double *out,           \
        const double *yn, double *acc, const Stage &st, const RhsLoad &load, const OuterArgs &oa
cudaError_t rhs_sph4(NRK_RHS_ARGS);
cudaError_t rhs_sph8(NRK_RHS_ARGS);
cudaError_t rhs_cyl4(NRK_RHS_ARGS);
cudaError_t rhs_cyl8(NRK_RHS_ARGS);
#define NRK_RHS_LAUNCH(NAME, FAM_, AXTWO_, ORD_)                                                                  \
    cudaError_t rhs_##NAME(NRK_RHS_ARGS)                                                                          \
    {                                                                                                             \
        return two ? launch_k_rhs<FAM_, AXTWO_, ORD_>(s, G, yin, d1x, d1y, out, yn, acc, st, load, oa)            \
                   : launch_k_rhs<FAM_, -1, ORD_>(s, G, yin, d1x, d1y, out, yn, acc, st, load, oa);               \
    }

}  // namespace nrk
