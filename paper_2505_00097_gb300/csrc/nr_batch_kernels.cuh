// nr_batch_kernels.cuh -- the per-substage kernel of batched mode and its
// launch helpers, instantiated once per coordinate family and finite-difference
// order (nr_batch_{sph,cyl}{,8}.cu) so the four compile in parallel.
//
// A work item is a tx x ty tile of one grid's interior points, or, in the spread shapes of small batches, 32
// consecutive ones, or a chunk of its pure-outer ghost points.  One launch per RK substage covers the items of all
// grids, one block per item (tx * ty threads; spread: four warps, as k_rhs_spread): the block finds its grid
// by binary search over the items' start indices and stages that grid's
// record in shared memory.  Every
// point runs the same per-point code as the single-grid kernels
// (nr_stage.cuh, with the same two-point-azimuth specialisation AX; the grids
// of one batch share it), so a grid's state after n batched steps is bitwise
// the state after n single-grid steps, whatever the tile shape or the company.
#pragma once

#include <algorithm>

#include "nr_stage.cuh"

namespace nrk {

struct __align__(16) BGrid {
    GridK K;
    double *y, *ya, *yb, *acc;
    double *d1x, *d1y;         // the grid's stored first differences
    int d1_begin, d1_end;      // its items of the first-difference pass (256 points each)
    const OuterPt* outer;
    const double* finf;
    const double* wspeed;
    int n_outer;
    int tiles_x, tx;           // tiles of tx columns, blockDim.x points (not in the spread shapes)
    int w_begin, w_rhs_end, w_end;
    int ssp;                   // the table's integrator: 0 RK4 (st[0..3]), 1 SSPRK3 (st[0..2])
    Stage st[4];
};

constexpr int BATCH_MAX_THREADS = 128;

struct BInner {
    int grid, dst, src, negmask;
};

// the buffers of one substage, as the single-grid drivers use them: RK4 y -> ya -> yb -> ya
// -> y (the last stage from acc); SSPRK3 y -> ya -> yb -> y (in place, reading y_n)
__device__ __forceinline__ void stage_buffers(const BGrid& B, int stage, const double*& yin, double*& out,
                                              const double*& yn)
{
    switch (stage) {
    case 0: yin = B.y; out = B.ya; yn = B.y; break;
    case 1: yin = B.ya; out = B.yb; yn = B.y; break;
    case 2: yin = B.yb; out = B.ssp ? B.y : B.ya; yn = B.y; break;
    default: yin = B.ya; out = B.y; yn = nullptr; break;
    }
}

// the grid of work item w, its record staged in shared memory; ends with the block's barrier
__device__ __forceinline__ const BGrid& batch_grid(const BGrid* __restrict__ grids, int ngrids, int w,
                                                   unsigned long long* s_grid)
{
    int lo = 0, hi = ngrids - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (grids[mid].w_begin <= w) lo = mid;
        else hi = mid - 1;
    }
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(grids + lo);
    for (int q = threadIdx.x; q < (int)(sizeof(BGrid) / 8); q += blockDim.x) s_grid[q] = src[q];
    __syncthreads();
    return *reinterpret_cast<const BGrid*>(s_grid);
}
constexpr int BGRID_WORDS = (sizeof(BGrid) + 7) / 8;

// one block per work item; BPS blocks of BATCH_MAX_THREADS per SM (registers), two in batches that leave no scheduler more
// than two warps (rhs_shape), as k_rhs
template <int FAM, int AX, int ORD, int BPS>
__global__ void __launch_bounds__(BATCH_MAX_THREADS, BPS) k_batch_stage(const BGrid* __restrict__ grids, int ngrids,
                                                                        int total, int stage)
{
    __shared__ __align__(16) unsigned long long s_grid[BGRID_WORDS];
    const int tid = threadIdx.x;
    const int w = (int)blockIdx.x;
    if (w >= total) return;
    const BGrid& B = batch_grid(grids, ngrids, w, s_grid);
    const double* yin;
    const double* yn;
    double* out;
    stage_buffers(B, stage, yin, out, yn);
    if (w < B.w_rhs_end) {
        const int t = w - B.w_begin, ty = (int)blockDim.x / B.tx;
        const int i = (t % B.tiles_x) * B.tx + tid % B.tx;
        const int j = (t / B.tiles_x) * ty + tid / B.tx;
        if (i < B.K.N0 && j < B.K.N1 * B.K.N2)
            rhs_point_stage<FAM, AX, ORD>(B.K, yin, B.d1x, B.d1y, out, yn, B.acc, B.st[stage], i, j);
    } else {
        const int p = (w - B.w_rhs_end) * (int)blockDim.x + tid;
        if (p < B.n_outer)
            outer_point_stage<FAM, ORD, ssp_first_short<AX>()>(B.K, B.outer[p], yin, out, yn, B.acc, B.finf, B.wspeed,
                                                               B.st[stage]);
    }
}

// The same for batches of few points (rhs_shape), 32 consecutive points per block of four warps, as k_rhs_spread.  Per RK
// step: six 64x16x2 grids 382 -> 296 us (all-FP64: 341)
template <int FAM, int AX, int ORD, int BPS>
__global__ void __launch_bounds__(32 * SPREAD_WARPS, BPS) k_batch_spread(const BGrid* __restrict__ grids, int ngrids,
                                                                         int total, int stage)
{
    __shared__ __align__(16) unsigned long long s_grid[BGRID_WORDS];
    __shared__ double tab[RawIx<AX>::N + NGF][32];
    __shared__ int slot;
    const int w = (int)blockIdx.x;
    if (w >= total) return;
    const BGrid& B = batch_grid(grids, ngrids, w, s_grid);
    const double* yin;
    const double* yn;
    double* out;
    stage_buffers(B, stage, yin, out, yn);
    if (w >= B.w_rhs_end) {
        const int p = (w - B.w_rhs_end) * (32 * SPREAD_WARPS) + threadIdx.x;
        if (p < B.n_outer)
            outer_point_stage<FAM, ORD, ssp_first_short<AX>()>(B.K, B.outer[p], yin, out, yn, B.acc, B.finf, B.wspeed,
                                                               B.st[stage]);
        return;
    }
    spread_slot(&slot);
    const int n = B.K.N0 * B.K.N1 * B.K.N2, p = (w - B.w_begin) * 32 + (threadIdx.x & 31), q = p < n ? p : n - 1;
    rhs_spread_stage<FAM, AX, ORD>(B.K, yin, B.d1x, B.d1y, out, yn, B.acc, B.st[stage], q % B.K.N0, q / B.K.N0, p < n,
                                   threadIdx.x / 32, slot, tab);
}

// the stored first differences of every grid's stage input, 256 points per block
template <int AX, int ORD>
__global__ void __launch_bounds__(256) k_batch_d1(const BGrid* __restrict__ grids, int ngrids, int total, int stage)
{
    const int w = (int)blockIdx.x;
    if (w >= total) return;
    int lo = 0, hi = ngrids - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (grids[mid].d1_begin <= w) lo = mid;
        else hi = mid - 1;
    }
    const BGrid& B = grids[lo];
    const double* yin;
    const double* yn;
    double* out;
    stage_buffers(B, stage, yin, out, yn);
    d1_point<AX, ORD>(B.K, yin, B.d1x, B.d1y, (long)(w - B.d1_begin) * 256 + threadIdx.x);
}

// work-item shapes the autotuner tries: tiles, which nr_batch_set_tile can ask for too, and 32 points spread over four
// warps with three or four blocks per SM
struct TileShape {
    int tx, ty, spread;
};
constexpr TileShape kTiles[] = {{32, 4, 0}, {64, 2, 0}, {128, 1, 0}, {16, 8, 0}, {32, 2, 0},
                                {64, 1, 0}, {32, 1, 0}, {32, 1, 3},  {32, 1, 4}};
constexpr int kNumShapes = sizeof(kTiles) / sizeof(kTiles[0]), kNumTiles = kNumShapes - 2;

// few: the batch is small enough for two blocks per SM
template <int FAM, int AX, int ORD>
cudaError_t launch_bstage(int tile, bool few, const BGrid* g, int n, int total, int stage, cudaStream_t s)
{
    const TileShape t = kTiles[tile];
    if (total <= 0) return cudaSuccess;
    if (t.spread == 3) k_batch_spread<FAM, AX, ORD, 3><<<total, 32 * SPREAD_WARPS, 0, s>>>(g, n, total, stage);
    else if (t.spread == 4) k_batch_spread<FAM, AX, ORD, 4><<<total, 32 * SPREAD_WARPS, 0, s>>>(g, n, total, stage);
    else if (few) k_batch_stage<FAM, AX, ORD, 2><<<total, t.tx * t.ty, 0, s>>>(g, n, total, stage);
    else k_batch_stage<FAM, AX, ORD, 4><<<total, t.tx * t.ty, 0, s>>>(g, n, total, stage);
    return cudaGetLastError();
}

template <int AX, int ORD>
cudaError_t launch_batch_d1(const BGrid* g, int n, int total_d1, int stage, cudaStream_t s)
{
    if (total_d1 > 0) k_batch_d1<AX, ORD><<<total_d1, 256, 0, s>>>(g, n, total_d1, stage);
    return cudaGetLastError();
}

// one translation unit per family and order (nr_batch_{sph,cyl}{,8}.cu) defines, through
// NRK_BATCH_LAUNCH, the substage launch (tile shape `tile`) and the first-difference pass
// of all grids; two_point: the grids' azimuth holds two points (GridK::ax >= 0)
#define NRK_BATCH_DECL(NAME)                                                                                   \
    cudaError_t batch_stage_##NAME(bool two_point, int tile, bool few, const BGrid* g, int n, int total,       \
                                   int stage, cudaStream_t s);                                                 \
    cudaError_t batch_d1_##NAME(bool two_point, const BGrid* g, int n, int total_d1, int stage, cudaStream_t s);
NRK_BATCH_DECL(sph4)
NRK_BATCH_DECL(sph8)
NRK_BATCH_DECL(cyl4)
NRK_BATCH_DECL(cyl8)

#define NRK_BATCH_LAUNCH(NAME, FAM_, AXTWO_, ORD_)                                                             \
    cudaError_t batch_stage_##NAME(bool two_point, int tile, bool few, const BGrid* g, int n, int total,       \
                                   int stage, cudaStream_t s)                                                  \
    {                                                                                                          \
        return two_point ? launch_bstage<FAM_, AXTWO_, ORD_>(tile, few, g, n, total, stage, s)                 \
                         : launch_bstage<FAM_, -1, ORD_>(tile, few, g, n, total, stage, s);                    \
    }                                                                                                          \
    cudaError_t batch_d1_##NAME(bool two_point, const BGrid* g, int n, int total_d1, int stage, cudaStream_t s) \
    {                                                                                                          \
        return two_point ? launch_batch_d1<AXTWO_, ORD_>(g, n, total_d1, stage, s)                             \
                         : launch_batch_d1<-1, ORD_>(g, n, total_d1, stage, s);                                \
    }

}  // namespace nrk
