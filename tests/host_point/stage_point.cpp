// Test harness: the per-point bodies of the kernels (nr_stage.cuh), compiled for the host with g++ and run over a
// small grid as the kernels run them: the stored first differences (d1_point), then rhs_point_stage per point
// (k_rhs, k_batch_stage) or rhs_spread_stage per tile of 32 points by four emulated warps (k_rhs_spread); the
// constraints from their tables as k_ham and k_mom, and k_constraint_spread's warps, fill them.
#include <cmath>
#include <cstring>
#include <vector>

#define __device__
#define __host__
#define __forceinline__ inline
#define __global__
static inline long long __double_as_longlong(double x) { long long b; std::memcpy(&b, &x, 8); return b; }
static inline double __longlong_as_double(long long b) { double x; std::memcpy(&x, &b, 8); return x; }
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
template <class T> static inline T __ldg(const T* p) { return *p; }
using std::fabs;
using std::fma;
// the emulated lane; a block's warps run one after the other (the FP64 warp last), so its barrier is passed over
static struct { int x; } threadIdx;
static inline void __syncthreads() {}

#include "../../paper_2505_00097_gb300/csrc/nr_stage.cuh"
using namespace nrk;

namespace {

// x -> A sinh(x/w)/sinh(1/w) and its first two derivatives; linear (A x) without sinh
void radial(double A, double w, bool sinh_kind, double x, double f[3])
{
    if (sinh_kind) {
        const double s = std::sinh(1.0 / w);
        f[0] = A * std::sinh(x / w) / s; f[1] = A * std::cosh(x / w) / (w * s); f[2] = A * std::sinh(x / w) / (w * w * s);
    } else {
        f[0] = A * x; f[1] = A; f[2] = 0.0;
    }
}

struct HostGrid {
    GridK G;
    std::vector<double> a0, a1, a2;
};

template <int ORD>
void make_grid(HostGrid& H, int coords, const int* N, const double* ampl, const double* sinhw, const double* sigma, double eta)
{
    GridK& G = H.G;
    std::memset(&G, 0, sizeof G);
    const bool cyl = coords == 1;
    G.NG = ORD / 2 + 1;
    G.N0 = N[0]; G.N1 = N[1]; G.N2 = N[2];
    G.n0 = N[0] + 2 * G.NG; G.n1 = N[1] + 2 * G.NG; G.n2 = N[2] + 2 * G.NG;
    G.fam = cyl ? FAM_CYL : FAM_SPH;
    G.ax = (cyl && N[1] == 2) ? 1 : (!cyl && N[2] == 2) ? 2 : -1;
    G.ord = ORD;
    G.T = (long)G.n0 * G.n1 * G.n2;
    G.sigma_metric = sigma[0]; G.sigma_gauge = sigma[G_VET]; G.eta = eta;
    const double lo[3] = {0, cyl ? -M_PI : 0, cyl ? -1 : -M_PI}, hi[3] = {1, M_PI, cyl ? 1 : M_PI};
    double dx[3];
    for (int d = 0; d < 3; d++) {
        dx[d] = (hi[d] - lo[d]) / N[d];
        G.inv_d1[d] = 1.0 / (FD<ORD>::den1 * dx[d]);
        G.inv_d2[d] = 1.0 / (FD<ORD>::den2 * dx[d] * dx[d]);
    }
    auto xx = [&](int d, int i) { return lo[d] + ((double)(i - G.NG) + 0.5) * dx[d]; };
    double f[3];
    H.a0.resize(4 * G.n0);
    for (int i = 0; i < G.n0; i++) {
        radial(ampl[0], sinhw[0], coords != 2, xx(0, i), f);
        H.a0[i] = 1.0 / f[1]; H.a0[G.n0 + i] = 1.0 / f[0]; H.a0[2 * G.n0 + i] = f[2] / (f[1] * f[1]); H.a0[3 * G.n0 + i] = f[0];
    }
    H.a1.resize(4 * G.n1);
    H.a2.resize(3 * G.n2);
    if (cyl) {
        for (int i = 0; i < G.n2; i++) {
            radial(ampl[2], sinhw[2], true, xx(2, i), f);
            H.a2[i] = 1.0 / f[1]; H.a2[G.n2 + i] = f[2] / (f[1] * f[1]); H.a2[2 * G.n2 + i] = f[0];
        }
    } else {
        for (int i = 0; i < G.n1; i++) {
            const double th = xx(1, i);
            H.a1[i] = 1.0 / std::sin(th); H.a1[G.n1 + i] = std::cos(th) / std::sin(th);
        }
    }
    G.rfm = Rfm{H.a0.data(), H.a1.data(), H.a2.data()};
}

template <int FAM, int AX, int ORD>
void rhs(const GridK& G, const double* y, double* out, bool spread)
{
    std::vector<double> d1x(N_D1 * G.T, NAN), d1y(N_D1 * G.T, NAN);
    for (long t = 0; t < d1_points(G); t++) d1_point<AX, ORD>(G, y, d1x.data(), d1y.data(), t);
    const Stage st{MODE_RHS, 0, 0.0, 0.0, 0.0};
    const int n = G.N0 * G.N1 * G.N2;
    if (!spread) {
        for (int p = 0; p < n; p++)
            rhs_point_stage<FAM, AX, ORD>(G, y, d1x.data(), d1y.data(), out, nullptr, nullptr, st, p % G.N0, p / G.N0);
        return;
    }
    std::vector<double> mem((RawIx<AX>::N + NGF) * 32);
    double (*tab)[32] = reinterpret_cast<double (*)[32]>(mem.data());
    for (int tile = 0; 32 * tile < n; tile++) {
        for (double& v : mem) v = NAN;
        const int fp = tile % SPREAD_WARPS;
        for (int w = 0; w < SPREAD_WARPS; w++)
            for (int lane = 0; lane < 32; lane++) {
                const int warp = (fp + 1 + w) % SPREAD_WARPS, p = 32 * tile + lane, q = p < n ? p : n - 1;
                threadIdx.x = 32 * warp + lane;
                rhs_spread_stage<FAM, AX, ORD>(G, y, d1x.data(), d1y.data(), out, nullptr, nullptr, st, q % G.N0, q / G.N0,
                                               p < n, warp, fp, tab);
            }
    }
}

// at one point, from a table of stride 1 filled at once, or (spread) of stride 32 filled by four warps in turn
template <int FAM, int ORD, int S>
void constraint_at(const GridK& G, PointIn P, const double* y, double* out, int p0, int p1, int p2, bool momentum)
{
    constexpr int stride = src_stride<S>(), warps = S == SRC_DIAG_SHARED ? SPREAD_WARPS : 1;
    const long idx = P.y - y;
    std::vector<double> raw(DiagIx::N * stride, NAN);
    for (int w = 0; w < warps; w++) {
        if (momentum) mom_table<ORD>(P, raw.data() + stride - 1, stride, w, warps);
        else ham_table<ORD>(P, raw.data() + stride - 1, stride, w, warps);
    }
    P.raw = raw.data() + stride - 1;
    P.g = make_geo<FAM>(G, p0, p1, p2);
    if (momentum) {
        double M[3];
        mom_core<FAM, ORD, S>(P, M);
        for (int q = 0; q < 3; q++) out[q * G.T + idx] = M[q];
    } else {
        out[idx] = ham_core<FAM, ORD, S>(P);
    }
}

template <int FAM, int ORD>
void constraint(const GridK& G, const double* y, double* out, bool momentum, bool spread)
{
    for (int p2 = G.NG; p2 < G.NG + G.N2; p2++)
        for (int p1 = G.NG; p1 < G.NG + G.N1; p1++)
            for (int p0 = G.NG; p0 < G.NG + G.N0; p0++) {
                const PointIn P = point_in<-1>(G, y, nullptr, nullptr, p0, p1, p2);
                if (spread) constraint_at<FAM, ORD, SRC_DIAG_SHARED>(G, P, y, out, p0, p1, p2, momentum);
                else constraint_at<FAM, ORD, SRC_DIAG>(G, P, y, out, p0, p1, p2, momentum);
            }
}

template <int ORD>
void run(int coords, const int* N, const double* ampl, const double* sinhw, const double* sigma, double eta, const double* y,
         double* out, int which)
{
    HostGrid H;
    make_grid<ORD>(H, coords, N, ampl, sinhw, sigma, eta);
    const GridK& G = H.G;
    if (which >= 2) {
        if (G.fam == FAM_CYL) constraint<FAM_CYL, ORD>(G, y, out, which % 2 == 1, which >= 4);
        else constraint<FAM_SPH, ORD>(G, y, out, which % 2 == 1, which >= 4);
    } else if (G.fam == FAM_CYL) {
        if (G.ax == 1) rhs<FAM_CYL, 1, ORD>(G, y, out, which == 1);
        else rhs<FAM_CYL, -1, ORD>(G, y, out, which == 1);
    } else {
        if (G.ax == 2) rhs<FAM_SPH, 2, ORD>(G, y, out, which == 1);
        else rhs<FAM_SPH, -1, ORD>(G, y, out, which == 1);
    }
}

}  // namespace

// which: 0 the right-hand side as k_rhs computes it, 1 as k_rhs_spread, 2 the Hamiltonian constraint, 3 the momentum
// constraint, 4 and 5 the same as k_constraint_spread.  sigma: the dissipation strength per gridfunction (metric at 0, gauge at G_VET).
extern "C" void stage_point(int coords, const int* N, const double* ampl, const double* sinhw, const double* sigma, double eta,
                            const double* y, double* out, int which, int ng)
{
    if (ng == 5) run<8>(coords, N, ampl, sinhw, sigma, eta, y, out, which);
    else run<4>(coords, N, ampl, sinhw, sigma, eta, y, out, which);
}

// the launch shape of the right-hand side (0, 1 spread over three or four blocks per SM; 2, 3 one point per thread, two or
// four blocks per SM)
extern "C" int stage_shape(int fam, int ord, int two_point, int n_sm, long tiles, long outer)
{
    return rhs_shape(fam, ord, two_point != 0, RhsLoad{n_sm, tiles, outer});
}
