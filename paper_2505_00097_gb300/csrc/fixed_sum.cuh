// fixed_sum.cuh -- weighted sums of FP64 values in block fixed point, on the integer pipe.
//
// An FP64 instruction holds an SM's FP64 pipe of this chip for 16 to 20 cycles per warp (2 lanes a
// cycle); a 32-bit integer add or logic instruction takes 0.27, a shift 0.54 and a 32 x 32 -> 64
// multiply-add 1.34 (measured, 2 or 4 blocks of 128 threads per SM).  A finite-difference sum
// has integer weights, so once its values are aligned to their largest exponent it is exact integer
// arithmetic: about 11 cycles a value against 19 for one FMA, on pipes that the FP64 work leaves idle.
//
// Values enter as m = mantissa * 2^SH >> (E - e): integers in units of 2^(E - 1075 - SH), where E is the
// largest biased exponent of the sum's values and SH the guard bits below the mantissa.  Values within
// SH binades of the largest enter exactly; the rest are off by less than one unit, at most 2^-(52 + SH)
// of the largest (an FP64 sum rounds at 2^-53 of each partial sum).  Zeros and values more than
// 64 binades down enter as 0.  Results are rounded to nearest, ties away from zero, the same for either sign.  The
// callers keep E away from both ends of the exponent range and
// leave sums outside to FP64 arithmetic, which also handles infinities and NaNs.
#pragma once

namespace nrk {

typedef unsigned long long fx_u64;
typedef long long fx_i64;

// logical right shift; 0 for n >= 64
__device__ __forceinline__ fx_u64 fx_shr(fx_u64 x, int n)
{
#ifdef __CUDA_ARCH__
    fx_u64 r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
#else
    return n >= 64 ? 0 : x >> n;
#endif
}

// exponent key of a value: the top word without the sign (its biased exponent is key >> 20)
__device__ __forceinline__ int fx_key(fx_u64 b) { return (int)(b >> 32) & 0x7FFFFFFF; }
__device__ __forceinline__ int fx_max(int a, int b) { return a > b ? a : b; }

// the value with bits b as an integer in units of 2^(E - 1075 - SH)
template <int SH>
__device__ __forceinline__ fx_i64 fx_in(fx_u64 b, int E)
{
    const unsigned hi = (unsigned)(b >> 32);
    const fx_u64 m = ((b & 0x000FFFFFFFFFFFFFULL) | 0x0010000000000000ULL) << SH;
    const fx_u64 a = fx_shr(m, E - (int)((hi >> 20) & 0x7FF));
    const fx_i64 s = (fx_i64)((int)hi >> 31);
    return (fx_i64)((a ^ (fx_u64)s) - (fx_u64)s);
}

// m = h 2^32 + l with l signed: products of the parts are signed 32 x 32 -> 64 multiplies.  m < 2^63 - 2^31, above which
// the carry of a negative l takes h out of 32 bits.
struct FxSplit {
    int h, l;
};
__device__ __forceinline__ FxSplit fx_split(fx_i64 m)
{
    FxSplit r;
    r.l = (int)m;
    r.h = (int)(m >> 32) + (int)((unsigned)m >> 31);
    return r;
}

// a sum of products of 64-bit integers, in units of 2^64 (hh), 2^32 (cross and the upper half of the
// low products): |sum of h h|, |sum of cross products| must stay below 2^63
struct FxDot {
    fx_i64 hh, cross;
};
__device__ __forceinline__ int fx_mulhi(int a, int b)
{
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int)(((fx_i64)a * b) >> 32);
#endif
}
__device__ __forceinline__ void fx_mac(FxDot& d, FxSplit a, FxSplit b)
{
    d.hh += (fx_i64)a.h * b.h;
    d.cross += (fx_i64)a.h * b.l;
    d.cross += (fx_i64)a.l * b.h;
    d.cross += fx_mulhi(a.l, b.l);
}

// x / 2^Q and (h 2^32 + l) / 2^Q rounded to nearest, ties away from zero: the same for either sign, so that a sum of
// negated values is the negated sum (a field and its mirror image stay mirror images)
template <int Q>
__device__ __forceinline__ fx_i64 fx_shift(fx_i64 x) { return (x + (1LL << (Q - 1)) + (x >> 63)) >> Q; }
template <int Q>
__device__ __forceinline__ fx_i64 fx_shift(fx_i64 h, fx_i64 l)
{
    const fx_i64 t = h + (l >> 32);
    return (t << (32 - Q)) + ((fx_i64)((fx_u64)(unsigned)l + (1ULL << (Q - 1)) + (fx_u64)(t >> 63)) >> Q);
}

__device__ __forceinline__ int fx_clz(fx_u64 a) { return __clzll((fx_i64)a); }   // 64 for 0

// a 2^e (a = 1.x 2^63, or 0) with sign s (0 or -1) as an FP64 number, rounded to nearest
__device__ __forceinline__ double fx_pack(fx_u64 a, int e, fx_i64 s)
{
    // the hidden bit adds one to the exponent field
    const fx_u64 f = ((fx_u64)(unsigned)(e + 63 + 1022) << 52) + (a >> 11) + ((a >> 10) & 1);
    return __longlong_as_double((fx_i64)((a ? f : 0) | ((fx_u64)s << 63)));
}

// R 2^ex as an FP64 number, rounded to nearest; the result's exponent must be in the normal range
__device__ __forceinline__ double fx_out(fx_i64 R, int ex)
{
    const fx_i64 s = R >> 63;
    const fx_u64 a = (fx_u64)((R ^ s) - s);
    const int n = fx_clz(a);
    return fx_pack(a << (n & 63), ex - n, s);
}

// (H 2^32 + L) 2^ex
__device__ __forceinline__ double fx_out2(fx_i64 H, fx_i64 L, int ex)
{
    fx_i64 t = H + (L >> 32);
    unsigned lo = (unsigned)L;
    const fx_i64 s = t >> 63;
    // magnitude of t 2^32 + lo
    lo = (lo ^ (unsigned)s) - (unsigned)s;
    t = (t ^ s) + (s & (fx_i64)(lo == 0));
    const bool small = (fx_u64)t < 0x80000000ULL;   // the sum fits one 64-bit word
    const fx_u64 w = small ? ((fx_u64)t << 32) | lo : (fx_u64)t;
    const int n = fx_clz(w);   // below 33 unless small
    const fx_u64 a = (w << (n & 63)) | (small ? 0 : ((fx_u64)lo << (n & 63)) >> 32);
    return fx_pack(a, ex + (small ? 0 : 32) - n, s);
}

}  // namespace nrk
