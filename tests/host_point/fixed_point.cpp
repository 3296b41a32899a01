// Test harness: the integer-pipe difference sums of the point code (fixed_sum.cuh and the functions of
// bssn_point.cuh built on it), compiled for the host with g++.
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

// n first differences; f: rows of 9 values, the sum's centre in the middle; out and, fp64, the FP64 sums
extern "C" void fixed_d1(int ord, const double* f, long n, double* out, double* fp64)
{
    for (long i = 0; i < n; i++) {
        const double* c = f + 9 * i + 4;
        if (ord == 8) {
            FxD1<8> e; e.f = c; e.s = 1; e.load(); out[i] = e.sum(); fp64[i] = d1r<8>(c, 1);
        } else {
            FxD1<4> e; e.f = c; e.s = 1; e.load(); out[i] = e.sum(); fp64[i] = d1r<4>(c, 1);
        }
    }
}

// mixed difference at the centre of an n x n block f (n = 9, axis 0 fastest), and the FP64 one
extern "C" void fixed_mix(int ord, const double* f, double* out, double* fp64)
{
    const double* c = f + 4 + 9 * 4;
    *out = ord == 8 ? fx_mix<8>(c, 1, 9) : fx_mix<4>(c, 1, 9);
    *fp64 = ord == 8 ? mixr<8>(c, 1, 9) : mixr<4>(c, 1, 9);
}

extern "C" void fixed_sub(const double* a, const double* b, long n, double* out)
{
    for (long i = 0; i < n; i++) out[i] = fx_sub(a[i], b[i]);
}

namespace {
template <int AX, int ORD>
void advko(const double* f, const double* vet, const double* D, double sigma, double* out, double* fp64)
{
    // a 24-gridfunction state on 11^3 points: vet as given at the centre, f everywhere else's gridfunction 0
    constexpr int n = 11, T = n * n * n, c = 5 + n * (5 + n * 5);
    static double y[24 * T];
    std::memset(y, 0, sizeof y);
    for (int q = 0; q < T; q++) y[q] = f[q];
    for (int d = 0; d < 3; d++) y[(17 + d) * T + c] = vet[d];
    const long st[3] = {1, n, n * n}, ox = AX >= 0 ? st[AX] : 0;
    double sum[24], u[3];
    bool fwd[3];
    adv_ko_sums<AX, ORD>(y + c, T, st, ox, D, sigma, sigma, sum);
    for (int d = 0; d < 3; d++) { u[d] = fabs(vet[d]) * D[d]; fwd[d] = vet[d] > 0; }
    *out = sum[0];
    *fp64 = advko_fp64<AX, ORD>(y + c, st, ox, u, fwd, D, sigma);
}
}  // namespace

// advection + dissipation of gridfunction 0 at the centre of an 11^3 block f (axis 0 fastest)
extern "C" void fixed_advko(int ax, int ord, const double* f, const double* vet, const double* D, double sigma,
                            double* out, double* fp64)
{
    if (ord == 8) {
        if (ax == 1) advko<1, 8>(f, vet, D, sigma, out, fp64);
        else if (ax == 2) advko<2, 8>(f, vet, D, sigma, out, fp64);
        else advko<-1, 8>(f, vet, D, sigma, out, fp64);
    } else {
        if (ax == 1) advko<1, 4>(f, vet, D, sigma, out, fp64);
        else if (ax == 2) advko<2, 4>(f, vet, D, sigma, out, fp64);
        else advko<-1, 4>(f, vet, D, sigma, out, fp64);
    }
}
