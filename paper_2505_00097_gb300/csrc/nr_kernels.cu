// nr_kernels.cu -- sm_103a FP64 kernels of the BSSN hot path.
//
//   k_d1      raw first differences along axes 0 (and 1) of the gridfunctions
//             with second derivatives, read by k_rhs for its mixed derivatives
//   k_rhs     (nr_rhs_kernels.cuh, launched from here) interior right-hand side
//             (Sec. 2.1 equations, upwinded advection, Kreiss-Oliger dissipation)
//             with the RK4 stage update and the det(gammabar) enforcement fused
//             into its epilogue; in an RK stage some of its blocks run the
//             radiation condition at the pure-outer ghosts (Sec. 3) with the same
//             epilogue
//   k_outer   the radiation condition alone (nr_apply_bcs)
//   k_inner   parity copies at inner ghosts (Sec. 3), one warp-coalesced gather
//             per gridfunction
//   k_bl      Brill-Lindquist data + SplitMix64 perturbation
//   k_ham     Hamiltonian constraint (Eq. Hconstraint) + per-block norm partials
//   k_mom     momentum constraint (Eq. Mconstraint) + per-block norm partials
//   k_ham_reduce  fixed-order reduction of the partials (both constraints)
//   k_finite  NaN/Inf guard on alpha and W
//   k_digest  64-bit digest of a state at the canonical points (bitwise comparisons)
#include <math.h>

#include <algorithm>

#include "bssn_point.cuh"
#include "nr_geo.cuh"
#include "nr_internal.h"
#include "nr_rhs_kernels.cuh"
#include "nr_stage.cuh"

namespace nrk {

// Raw first differences along axis 0 (and, on a general grid, axis 1) of the N_D1
// gridfunctions with second derivatives, at interior i0 and every row a mixed
// stencil of an interior point reads: i1 and i2 within two points of the interior,
// except along a two-point azimuth (no mixed derivatives there); the axis-1 set at
// interior i1 only.
template <int AX, int ORD>
__global__ void __launch_bounds__(256) k_d1(GridK G, const double* __restrict__ y, double* d1x, double* d1y)
{
    d1_point<AX, ORD>(G, y, d1x, d1y, (long)blockIdx.x * blockDim.x + threadIdx.x);
}

template <int FAM, int ORD>
__global__ void __launch_bounds__(128) k_outer(GridK G, const OuterPt* __restrict__ pts, int npts,
                                               const double* __restrict__ yin, double* out, const double* yn,
                                               double* acc, const double* __restrict__ finf,
                                               const double* __restrict__ wspeed, Stage st)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= npts) return;
    outer_point_stage<FAM, ORD>(G, pts[t], yin, out, yn, acc, finf, wspeed, st);
}

__global__ void __launch_bounds__(256) k_inner(long T, const InnerPt* __restrict__ pts, int npts, double* y)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= npts) return;
    inner_copy(T, pts[t], blockIdx.y, y);
}

// SplitMix64 (Steele, Lea & Flood 2014) first output for state x
__device__ __forceinline__ uint64_t splitmix64(uint64_t x)
{
    uint64_t z = x + 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// ctr (NULL: the flat index itself): the perturbation counter of each canonical point -- its flat
// index on the whole grid when G describes one partition of it
__global__ void k_bl(GridK G, const int* __restrict__ canon, const int* __restrict__ ctr, long ncanon, int np,
                     const double* __restrict__ mxyz, double amp, uint64_t seed, double* y)
{
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ncanon) return;
    const long idx = canon[t];
    const uint64_t key = ctr ? (uint64_t)ctr[t] : (uint64_t)idx;
    const int i0 = (int)(idx % G.n0), i1 = (int)((idx / G.n0) % G.n1), i2 = (int)(idx / ((long)G.n0 * G.n1));
    double x[3];
    cart_of(G, i0, i1, i2, x);
    double psi = 1.0;
    for (int q = 0; q < np; q++) {
        const double dx = x[0] - mxyz[4 * q + 1], dy = x[1] - mxyz[4 * q + 2], dz = x[2] - mxyz[4 * q + 3];
        psi += mxyz[4 * q] / (2.0 * sqrt(dx * dx + dy * dy + dz * dz));
    }
    const double w = 1.0 / (psi * psi);
    for (int g = 0; g < NGF; g++) y[(long)g * G.T + idx] = 0.0;
    y[(long)G_CF * G.T + idx] = w;
    y[(long)G_ALPHA * G.T + idx] = w;
    if (amp != 0.0) {
        for (int s = 0; s < 6; s++) {
            const uint64_t u = splitmix64(seed ^ (((uint64_t)(G_HDD + s) << 40) | key));
            y[(long)(G_HDD + s) * G.T + idx] = amp * (2.0 * ((double)(u >> 11) * 0x1.0p-53) - 1.0);
        }
    }
}

// The constraints, one point per thread: the first and mixed differences on the integer pipe into a table in local
// memory, then the FP64 part, which bounds them (as in k_rhs).  BPS blocks per SM: with six (80 registers) both
// constraints with their norms take 751 us on 256x2x512, against 792 / 876 / 1063 us with four, three, two, and 904 us
// with the differences in FP64 (no limit on the registers).  The Hamiltonian constraint takes three (168 registers, no
// spills to speak of) where one round holds them (ham_shape).
constexpr int HAM_THREADS = 128;

// per-block partial norms (sum of squares, max, count) of a constraint, in a fixed order
__device__ __forceinline__ void block_partials(double s2, double mx, double cnt, double* partials)
{
    __shared__ double sh[3][HAM_THREADS];
    sh[0][threadIdx.x] = s2;
    sh[1][threadIdx.x] = mx;
    sh[2][threadIdx.x] = cnt;
    __syncthreads();
    for (int w = HAM_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
            sh[1][threadIdx.x] = fmax(sh[1][threadIdx.x], sh[1][threadIdx.x + w]);
            sh[2][threadIdx.x] += sh[2][threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partials[3 * blockIdx.x + 0] = sh[0][0];
        partials[3 * blockIdx.x + 1] = sh[1][0];
        partials[3 * blockIdx.x + 2] = sh[2][0];
    }
}

// interior point t (i0 fastest) of a constraint: padded indices, and the inputs but geometry and differences
__device__ __forceinline__ PointIn constraint_point(const GridK& G, const double* __restrict__ y, long t, int p[3])
{
    const int i = (int)(t % G.N0), j = (int)(t / G.N0);
    p[0] = i + G.NG;
    p[1] = j % G.N1 + G.NG;
    p[2] = j / G.N1 + G.NG;
    return point_in<-1>(G, y, nullptr, nullptr, p[0], p[1], p[2]);
}

// the FP64 part of a constraint (MOM: momentum, Eq. Mconstraint, rescaled M^i; else Hamiltonian, Eq. Hconstraint) at one
// point from the table P.raw, into out (1 or 3 gridfunctions, or NULL), and its share of the norms (of |M|)
template <int FAM, int ORD, bool MOM, int S>
__device__ __forceinline__ void constraint_value(const GridK& G, PointIn& P, const double* y, const int p[3], double* out,
                                                 double rmin, double rmax, double& s2, double& mx, double& cnt)
{
    const long idx = P.y - y;
    P.g = make_geo<FAM>(G, p[0], p[1], p[2]);
    double v;
    if constexpr (MOM) {
        double Mv[3];
        v = mom_core<FAM, ORD, S>(P, Mv);
        if (out) {
            out[idx] = Mv[0];
            out[G.T + idx] = Mv[1];
            out[2 * G.T + idx] = Mv[2];
        }
    } else {
        v = ham_core<FAM, ORD, S>(P);
        if (out) out[idx] = v;
    }
    double x[3];
    cart_of(G, p[0], p[1], p[2], x);
    const double r = sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
    if (r >= rmin && r <= rmax) {
        s2 = v * v;
        mx = fabs(v);
        cnt = 1.0;
    }
}

template <int FAM, int ORD, bool MOM>
__device__ __forceinline__ void constraint_points(const GridK& G, const double* __restrict__ y, double* out, double rmin,
                                                  double rmax, double* partials)
{
    const long t = (long)blockIdx.x * HAM_THREADS + threadIdx.x;
    double s2 = 0.0, mx = 0.0, cnt = 0.0;
    if (t < (long)G.N0 * G.N1 * G.N2) {
        int p[3];
        PointIn P = constraint_point(G, y, t, p);
        double raw[DiagIx::N];
        if constexpr (MOM) mom_table<ORD>(P, raw);
        else ham_table<ORD>(P, raw);
        P.raw = raw;
        constraint_value<FAM, ORD, MOM, SRC_DIAG>(G, P, y, p, out, rmin, rmax, s2, mx, cnt);
    }
    block_partials(s2, mx, cnt, partials);
}
template <int FAM, int ORD, int BPS>
__global__ void __launch_bounds__(HAM_THREADS, BPS) k_ham(GridK G, const double* __restrict__ y, double* H, double rmin,
                                                                 double rmax, double* partials)
{
    constraint_points<FAM, ORD, false>(G, y, H, rmin, rmax, partials);
}
template <int FAM, int ORD>
__global__ void __launch_bounds__(HAM_THREADS, 6) k_mom(GridK G, const double* __restrict__ y, double* M, double rmin,
                                                                 double rmax, double* partials)
{
    constraint_points<FAM, ORD, true>(G, y, M, rmin, rmax, partials);
}

// The same on grids of few points, whose time is one warp's way through its tile: 32 consecutive points per block, the
// differences divided among its warps, as in k_rhs_spread, and the same arithmetic per point.  BPS blocks per SM (168,
// 128 or 80 registers).
template <int FAM, int ORD, bool MOM, int BPS>
__global__ void __launch_bounds__(32 * SPREAD_WARPS, BPS)
    k_constraint_spread(GridK G, const double* __restrict__ y, double* out, double rmin, double rmax, double* partials)
{
    static_assert(HAM_THREADS == 32 * SPREAD_WARPS, "block_partials");
    __shared__ double tab[DiagIx::N][32];
    __shared__ int slot;
    const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
    const long n = (long)G.N0 * G.N1 * G.N2, t = (long)blockIdx.x * 32 + lane;
    int p[3];
    PointIn P = constraint_point(G, y, t < n ? t : n - 1, p);
    if constexpr (MOM) mom_table<ORD>(P, &tab[0][lane], 32, warp, SPREAD_WARPS);
    else ham_table<ORD>(P, &tab[0][lane], 32, warp, SPREAD_WARPS);
    spread_slot(&slot);
    double s2 = 0.0, mx = 0.0, cnt = 0.0;
    if (warp == slot && t < n) {
        P.raw = &tab[0][lane];
        constraint_value<FAM, ORD, MOM, SRC_DIAG_SHARED>(G, P, y, p, out, rmin, rmax, s2, mx, cnt);
    }
    block_partials(s2, mx, cnt, partials);
}

// one block; fixed order: thread t sums partials t, t+256, ..., then a tree
__global__ void __launch_bounds__(256) k_ham_reduce(const double* __restrict__ partials, int nparts, double* result)
{
    __shared__ double sh[3][256];
    double s = 0.0, m = 0.0, c = 0.0;
    for (int p = threadIdx.x; p < nparts; p += 256) {
        s += partials[3 * p];
        m = fmax(m, partials[3 * p + 1]);
        c += partials[3 * p + 2];
    }
    sh[0][threadIdx.x] = s;
    sh[1][threadIdx.x] = m;
    sh[2][threadIdx.x] = c;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
            sh[1][threadIdx.x] = fmax(sh[1][threadIdx.x], sh[1][threadIdx.x + w]);
            sh[2][threadIdx.x] += sh[2][threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double cnt = sh[2][0];
        result[0] = cnt > 0.0 ? sqrt(sh[0][0] / cnt) : 0.0;
        result[1] = sh[1][0];
        result[2] = cnt;
    }
}

__global__ void k_finite(long T, const double* __restrict__ y, int* flag)
{
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const double w = y[(long)G_CF * T + t], a = y[(long)G_ALPHA * T + t];
    if (!isfinite(w) || !isfinite(a)) atomicOr(flag, 1);
}

// Digest of a 24-gridfunction set at the canonical points: the wrapping sum over (gf, point)
// of splitmix64(bits ^ splitmix64((gf << 40) | idx)).  A sum modulo 2^64 does not depend on
// the order of its terms, so the digest does not depend on the launch shape; each term is a
// bijective mix of its value's bits, so a change of one value always changes the digest.
// ctr (NULL: the flat index itself): the key of each canonical point -- its flat index on the
// whole grid when the set is one partition of it.
__global__ void __launch_bounds__(256) k_digest(long T, const int* __restrict__ canon, const int* __restrict__ ctr,
                                                long nc, const double* __restrict__ y, unsigned long long* out)
{
    const int g = blockIdx.y;
    unsigned long long acc = 0;
    for (long t = (long)blockIdx.x * 256 + threadIdx.x; t < nc; t += (long)gridDim.x * 256) {
        const long idx = canon[t];
        const uint64_t key = ctr ? (uint64_t)ctr[t] : (uint64_t)idx;
        const uint64_t v = (uint64_t)__double_as_longlong(y[(long)g * T + idx]);
        acc += splitmix64(v ^ splitmix64(((uint64_t)g << 40) | key));
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

// FP64 FMA throughput probe: 8 independent FMA chains per thread, a fixed
// number of iterations (no data-dependent trip count), one store per thread.
__global__ void __launch_bounds__(256) k_fp64_probe(int iters, double seed, double* sink)
{
    double a[8];
#pragma unroll
    for (int q = 0; q < 8; q++) a[q] = seed + (double)(threadIdx.x + q);
    const double m = 0.999999999, c = 1e-9;
    for (int it = 0; it < iters; it++) {
#pragma unroll
        for (int q = 0; q < 8; q++) a[q] = fma(a[q], m, c);
    }
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < 8; q++) s += a[q];
    sink[(long)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

cudaError_t launch_fp64_probe(int blocks, int iters, double* sink, cudaStream_t s)
{
    k_fp64_probe<<<blocks, 256, 0, s>>>(iters, 1.0, sink);
    return cudaGetLastError();
}

// ------------------------------------------------------------ launchers

template <int ORD>
cudaError_t launch_rhs_ord(const GridK& G, const double* yin, double* d1x, double* d1y, double* out,
                           const double* yn, double* acc, Stage st, cudaStream_t s, const RhsLoad& load, OuterArgs oa)
{
    // the stored first differences of yin
    {
        const unsigned b = (unsigned)((d1_points(G) + 255) / 256);
        if (G.ax == 1) k_d1<1, ORD><<<b, 256, 0, s>>>(G, yin, d1x, d1y);
        else if (G.ax == 2) k_d1<2, ORD><<<b, 256, 0, s>>>(G, yin, d1x, d1y);
        else k_d1<-1, ORD><<<b, 256, 0, s>>>(G, yin, d1x, d1y);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const bool two = G.ax >= 0;
    if (G.fam == FAM_SPH) {
        return ORD == 8 ? rhs_sph8(two, s, G, yin, d1x, d1y, out, yn, acc, st, load, oa)
                        : rhs_sph4(two, s, G, yin, d1x, d1y, out, yn, acc, st, load, oa);
    }
    return ORD == 8 ? rhs_cyl8(two, s, G, yin, d1x, d1y, out, yn, acc, st, load, oa)
                    : rhs_cyl4(two, s, G, yin, d1x, d1y, out, yn, acc, st, load, oa);
}

cudaError_t launch_rhs(const GridK& G, const double* yin, double* d1x, double* d1y, double* out, const double* yn,
                       double* acc, Stage st, cudaStream_t s, const RhsLoad& load, OuterArgs oa)
{
    return G.ord == 8 ? launch_rhs_ord<8>(G, yin, d1x, d1y, out, yn, acc, st, s, load, oa)
                      : launch_rhs_ord<4>(G, yin, d1x, d1y, out, yn, acc, st, s, load, oa);
}

cudaError_t launch_outer(const GridK& G, const OuterPt* pts, int npts, const double* yin, double* out,
                         const double* yn, double* acc, const double* finf, const double* wspeed, Stage st,
                         cudaStream_t s)
{
    if (npts == 0) return cudaSuccess;
    const int b = 128, n = (npts + b - 1) / b;
    if (G.fam == FAM_SPH) {
        if (G.ord == 8) k_outer<FAM_SPH, 8><<<n, b, 0, s>>>(G, pts, npts, yin, out, yn, acc, finf, wspeed, st);
        else k_outer<FAM_SPH, 4><<<n, b, 0, s>>>(G, pts, npts, yin, out, yn, acc, finf, wspeed, st);
    } else {
        if (G.ord == 8) k_outer<FAM_CYL, 8><<<n, b, 0, s>>>(G, pts, npts, yin, out, yn, acc, finf, wspeed, st);
        else k_outer<FAM_CYL, 4><<<n, b, 0, s>>>(G, pts, npts, yin, out, yn, acc, finf, wspeed, st);
    }
    return cudaGetLastError();
}

cudaError_t launch_inner(const GridK& G, const InnerPt* pts, int npts, double* y, cudaStream_t s)
{
    if (npts == 0) return cudaSuccess;
    dim3 grd((npts + 255) / 256, NGF);
    k_inner<<<grd, 256, 0, s>>>(G.T, pts, npts, y);
    return cudaGetLastError();
}

// compact state: the 24 gridfunctions at the canonical points (interior and pure outer),
// layout [gf][t]; one grid row per gridfunction
__global__ void __launch_bounds__(256) k_gather(long T, const int* __restrict__ canon, long nc,
                                                const double* __restrict__ y, double* __restrict__ out)
{
    const double* src = y + (long)blockIdx.y * T;
    double* dst = out + (long)blockIdx.y * nc;
    for (long t = (long)blockIdx.x * 256 + threadIdx.x; t < nc; t += (long)gridDim.x * 256) dst[t] = src[canon[t]];
}

__global__ void __launch_bounds__(256) k_scatter(long T, const int* __restrict__ canon, long nc,
                                                 const double* __restrict__ in, double* __restrict__ y)
{
    const double* src = in + (long)blockIdx.y * nc;
    double* dst = y + (long)blockIdx.y * T;
    for (long t = (long)blockIdx.x * 256 + threadIdx.x; t < nc; t += (long)gridDim.x * 256) dst[canon[t]] = src[t];
}

cudaError_t launch_compact(const GridK& G, const int* canon, long nc, const double* src, double* dst, bool gather,
                           cudaStream_t s)
{
    if (nc == 0) return cudaSuccess;
    const long bx = std::min<long>((nc + 255) / 256, 4L * 152);
    const dim3 grd((unsigned)bx, NGF);
    if (gather) k_gather<<<grd, 256, 0, s>>>(G.T, canon, nc, src, dst);
    else k_scatter<<<grd, 256, 0, s>>>(G.T, canon, nc, src, dst);
    return cudaGetLastError();
}

cudaError_t launch_bl(const GridK& G, const int* canon_idx, long ncanon, int np, const double* mxyz, double amp,
                      uint64_t seed, double* y, cudaStream_t s, const int* ctr)
{
    const int b = 256;
    const long n = (ncanon + b - 1) / b;
    if (n == 0) return cudaSuccess;
    k_bl<<<(unsigned)n, b, 0, s>>>(G, canon_idx, ctr, ncanon, np, mxyz, amp, seed, y);
    return cudaGetLastError();
}

// Launch shape of the constraints: spread tiles of 32 points while one round of three, four or six blocks per SM holds
// them, else one point per thread.  us per call, spread with three / four / six, one point per thread with six, and with
// all differences in FP64, 64x2xN cylindrical (the others alike); Hamiltonian constraint:
//   256 tiles: 58 / 62 / 64, 88, 64;  8th order 80 / 82 / 88, 148, 117
//   576: 103 / 68 / 72, 90, 64;  142 / 103 / 111, 148, 118
//   896: 107 / 113 / 86, 119, 103;  164 / 157 / 137, 192, 211
//   1216: 149 / 122 / 131, 123 (with three blocks per SM 115), 104;  220 / 181 / 184, 198 (185), 212
//   1792: 198 / 173 / 154, 157 (146), 153;  305 / 257 / 240, 246 (228), 322
// Momentum constraint, four / six: 256: 35 / 35, 43, 37; 896: 58 / 45, 58, 56; 1216: 62 / 68, 58, 56.
enum HamShape { HAM_SPREAD3, HAM_SPREAD4, HAM_SPREAD6, HAM_POINTS3, HAM_POINTS6 };
HamShape ham_shape(const GridK& G, int n_sm)
{
    const long n = (long)G.N0 * G.N1 * G.N2, tiles = (n + 31) / 32, blocks = (n + HAM_THREADS - 1) / HAM_THREADS;
    if (tiles <= 3L * n_sm) return HAM_SPREAD3;
    if (tiles <= 4L * n_sm) return HAM_SPREAD4;
    if (tiles <= 6L * n_sm) return HAM_SPREAD6;
    return blocks <= 3L * n_sm ? HAM_POINTS3 : HAM_POINTS6;
}

int ham_partials_needed(const GridK& G, int n_sm)
{
    const long n = (long)G.N0 * G.N1 * G.N2, points = ham_shape(G, n_sm) <= HAM_SPREAD6 ? 32 : HAM_THREADS;
    return (int)((n + points - 1) / points);
}

template <int FAM, int ORD>
void launch_constraint(bool mom, const GridK& G, const double* y, double* out, double rmin, double rmax, double* partials,
                       int nb, int n_sm, cudaStream_t s)
{
    switch (ham_shape(G, n_sm)) {
    case HAM_SPREAD3:
    case HAM_SPREAD4:
        if (mom) k_constraint_spread<FAM, ORD, true, 4><<<nb, HAM_THREADS, 0, s>>>(G, y, out, rmin, rmax, partials);
        else if (ham_shape(G, n_sm) == HAM_SPREAD3)
            k_constraint_spread<FAM, ORD, false, 3><<<nb, HAM_THREADS, 0, s>>>(G, y, out, rmin, rmax, partials);
        else k_constraint_spread<FAM, ORD, false, 4><<<nb, HAM_THREADS, 0, s>>>(G, y, out, rmin, rmax, partials);
        break;
    case HAM_SPREAD6:
        if (mom) k_constraint_spread<FAM, ORD, true, 6><<<nb, HAM_THREADS, 0, s>>>(G, y, out, rmin, rmax, partials);
        else k_constraint_spread<FAM, ORD, false, 6><<<nb, HAM_THREADS, 0, s>>>(G, y, out, rmin, rmax, partials);
        break;
    case HAM_POINTS3:
        if (mom) k_mom<FAM, ORD><<<nb, HAM_THREADS, 0, s>>>(G, y, out, rmin, rmax, partials);
        else k_ham<FAM, ORD, 3><<<nb, HAM_THREADS, 0, s>>>(G, y, out, rmin, rmax, partials);
        break;
    default:
        if (mom) k_mom<FAM, ORD><<<nb, HAM_THREADS, 0, s>>>(G, y, out, rmin, rmax, partials);
        else k_ham<FAM, ORD, 6><<<nb, HAM_THREADS, 0, s>>>(G, y, out, rmin, rmax, partials);
    }
}

cudaError_t launch_constraints(bool mom, const GridK& G, const double* y, double* out, double rmin, double rmax,
                               double* partials, double* result, int n_sm, cudaStream_t s)
{
    const int nparts = ham_partials_needed(G, n_sm);
    if (G.fam == FAM_SPH) {
        if (G.ord == 8) launch_constraint<FAM_SPH, 8>(mom, G, y, out, rmin, rmax, partials, nparts, n_sm, s);
        else launch_constraint<FAM_SPH, 4>(mom, G, y, out, rmin, rmax, partials, nparts, n_sm, s);
    } else {
        if (G.ord == 8) launch_constraint<FAM_CYL, 8>(mom, G, y, out, rmin, rmax, partials, nparts, n_sm, s);
        else launch_constraint<FAM_CYL, 4>(mom, G, y, out, rmin, rmax, partials, nparts, n_sm, s);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_ham_reduce<<<1, 256, 0, s>>>(partials, nparts, result);
    return cudaGetLastError();
}

cudaError_t launch_ham(const GridK& G, const double* y, double* H, double rmin, double rmax, double* partials,
                       double* result, int n_sm, cudaStream_t s)
{
    return launch_constraints(false, G, y, H, rmin, rmax, partials, result, n_sm, s);
}

cudaError_t launch_mom(const GridK& G, const double* y, double* M, double rmin, double rmax, double* partials,
                       double* result, int n_sm, cudaStream_t s)
{
    return launch_constraints(true, G, y, M, rmin, rmax, partials, result, n_sm, s);
}

cudaError_t launch_ham_reduce(const double* partials, int nparts, double* result, cudaStream_t s)
{
    k_ham_reduce<<<1, 256, 0, s>>>(partials, nparts, result);
    return cudaGetLastError();
}

cudaError_t launch_digest(const GridK& G, const int* canon, long nc, const double* y, unsigned long long* out,
                          cudaStream_t s, const int* ctr)
{
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess || nc == 0) return e;
    const long bx = std::min<long>((nc + 255) / 256, 2L * 152);
    k_digest<<<dim3((unsigned)bx, NGF), 256, 0, s>>>(G.T, canon, ctr, nc, y, out);
    return cudaGetLastError();
}

cudaError_t launch_finite(const GridK& G, const double* y, int* flag, cudaStream_t s)
{
    const int b = 256;
    k_finite<<<(unsigned)((G.T + b - 1) / b), b, 0, s>>>(G.T, y, flag);
    return cudaGetLastError();
}

}  // namespace nrk
