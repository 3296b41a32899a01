// Test harness: metric_first and delta_trace of the point code (bssn_point.cuh), compiled for the host with g++.
#include <cmath>
#include <cstring>

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

#include "../../paper_2505_00097_gb300/csrc/bssn_point.cuh"
using namespace nrk;

namespace {
template <int FAM, int AX, int ORD>
void first(const PointIn& P, double* gi, double* dh, double* dtr)
{
    MetricPart M;
    metric_first<FAM, AX, SRC_INLINE, ORD>(P, M);
    for (int s = 0; s < 6; s++) gi[s] = M.gi[s];
    for (int k = 0; k < 3; k++)
        for (int s = 0; s < 6; s++) dh[6 * k + s] = M.dh[k][s];
    delta_trace<AX>(M, dtr);
}
}  // namespace

// gammabar^ij (6), e_k h_ij (3 x 6) and Delta^k_km (3) at the centre of an 11^3 block of 24 gridfunctions;
// geo: the scales D[0..2] and the rotation coefficients a, b, c
extern "C" void metric_point(int cyl, int ax, int ord, const double* y, const double* geo, double* gi, double* dh,
                             double* dtr)
{
    constexpr int n = 11;
    PointIn P;
    std::memset(&P, 0, sizeof P);
    P.y = y + 5 + n * (5 + n * 5);
    P.T = n * n * n;
    P.st[0] = 1; P.st[1] = n; P.st[2] = n * n;
    for (int d = 0; d < 3; d++) P.g.D[d] = geo[d];
    P.g.a = geo[3]; P.g.b = geo[4]; P.g.c = geo[5];
    if (ord == 8) {
        if (cyl) ax == 1 ? first<FAM_CYL, 1, 8>(P, gi, dh, dtr) : first<FAM_CYL, -1, 8>(P, gi, dh, dtr);
        else ax == 2 ? first<FAM_SPH, 2, 8>(P, gi, dh, dtr) : first<FAM_SPH, -1, 8>(P, gi, dh, dtr);
    } else {
        if (cyl) ax == 1 ? first<FAM_CYL, 1, 4>(P, gi, dh, dtr) : first<FAM_CYL, -1, 4>(P, gi, dh, dtr);
        else ax == 2 ? first<FAM_SPH, 2, 4>(P, gi, dh, dtr) : first<FAM_SPH, -1, 4>(P, gi, dh, dtr);
    }
}
