// Test harness: the integer-pipe difference sums of the point code on the device (fixed_sum.cuh takes other
// instructions there: shr.u64, __mulhi, __clzll), with the interface of the host harness fixed_point.cpp.
#include <cuda_runtime.h>

#include "../../paper_2505_00097_gb300/csrc/bssn_point.cuh"
using namespace nrk;

namespace {

template <int ORD>
__global__ void d1(const double* f, long n, double* out)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fx_d1_inline<ORD>(f + 9 * i + 4, 1);
}
template <int ORD>
__global__ void mix(const double* f, long n, double* out)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fx_mix<ORD>(f + 81 * i + 40, 1, 9);
}
__global__ void sub(const double* a, const double* b, long n, double* out)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fx_sub(a[i], b[i]);
}
// gridfunction 0 of item i of n, each 24 gridfunctions on 11^3 points, with par = {D[3], sigma}
template <int AX, int ORD>
__global__ void adv(const double* y, const double* par, long n, double* out)
{
    constexpr int m = 11, T = m * m * m;
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const long st[3] = {1, m, m * m}, ox = AX >= 0 ? st[AX >= 0 ? AX : 0] : 0;
    double sum[NGF];
    adv_ko_sums<AX, ORD>(y + i * 24 * T + 5 + m * (5 + m * 5), T, st, ox, par + 4 * i, par[4 * i + 3], par[4 * i + 3], sum);
    out[i] = sum[0];
}

// runs `launch` on device copies of the inputs; 0 or the CUDA error
template <class F>
int with(const double* a, size_t na, const double* b, size_t nb, double* out, size_t no, F launch)
{
    double *da = nullptr, *db = nullptr, *dout = nullptr;
    cudaError_t e = cudaMalloc(&da, 8 * na);
    if (e == cudaSuccess) e = cudaMalloc(&db, 8 * (nb ? nb : 1));
    if (e == cudaSuccess) e = cudaMalloc(&dout, 8 * no);
    if (e == cudaSuccess) e = cudaMemcpy(da, a, 8 * na, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && nb) e = cudaMemcpy(db, b, 8 * nb, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        launch(da, db, dout);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, dout, 8 * no, cudaMemcpyDeviceToHost);
    cudaFree(da);
    cudaFree(db);
    cudaFree(dout);
    return (int)e;
}

}  // namespace

extern "C" int device_d1(int ord, const double* f, long n, double* out)
{
    return with(f, 9 * n, nullptr, 0, out, n, [=](double* a, double*, double* o) {
        ord == 8 ? d1<8><<<(n + 127) / 128, 128>>>(a, n, o) : d1<4><<<(n + 127) / 128, 128>>>(a, n, o);
    });
}
extern "C" int device_mix(int ord, const double* f, long n, double* out)
{
    return with(f, 81 * n, nullptr, 0, out, n, [=](double* a, double*, double* o) {
        ord == 8 ? mix<8><<<(n + 127) / 128, 128>>>(a, n, o) : mix<4><<<(n + 127) / 128, 128>>>(a, n, o);
    });
}
extern "C" int device_sub(const double* x, const double* y, long n, double* out)
{
    return with(x, n, y, n, out, n, [=](double* a, double* b, double* o) { sub<<<(n + 127) / 128, 128>>>(a, b, n, o); });
}
extern "C" int device_adv(int ax, int ord, const double* y, const double* par, long n, double* out)
{
    return with(y, (size_t)n * 24 * 1331, par, 4 * n, out, n, [=](double* a, double* b, double* o) {
        const int g = (int)((n + 31) / 32);
        if (ord == 8) {
            if (ax == 1) adv<1, 8><<<g, 32>>>(a, b, n, o);
            else if (ax == 2) adv<2, 8><<<g, 32>>>(a, b, n, o);
            else adv<-1, 8><<<g, 32>>>(a, b, n, o);
        } else {
            if (ax == 1) adv<1, 4><<<g, 32>>>(a, b, n, o);
            else if (ax == 2) adv<2, 4><<<g, 32>>>(a, b, n, o);
            else adv<-1, 4><<<g, 32>>>(a, b, n, o);
        }
    });
}
