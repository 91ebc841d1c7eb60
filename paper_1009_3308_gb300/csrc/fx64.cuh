// 64-bit fixed-point complex arithmetic for the FP64 longitude transforms.
//
// GB300 retires about two FP64 operations per clock per SM, while its integer
// ALUs run at the full FP32 rate: a 64-bit add takes two instructions and a
// fixed-point twiddle product 12 wide multiply-adds, so a radix-8 butterfly
// with its twiddles costs about a sixth of its FP64 time.  The values of one
// spectrum are scaled by one power of two so that the sum of their magnitudes
// (a bound on every intermediate of the transform) stays below 2^61; rounding
// is then about 2^-60 of that sum per butterfly, below the 2^-53 relative
// rounding of FP64 arithmetic at the spectrum's norm.
//
// Coefficients (twiddles, the constants of the small DFTs) are Q62 integers
// split as hi 2^32 + lo with lo in [-2^31, 2^31).
#pragma once
#include <cuda_runtime.h>

#include "fft_small.cuh"

namespace sph {

struct fx {
    long long v;
};
__device__ __forceinline__ fx operator+(fx a, fx b) { return {a.v + b.v}; }
__device__ __forceinline__ fx operator-(fx a, fx b) { return {a.v - b.v}; }
__device__ __forceinline__ fx operator-(fx a) { return {-a.v}; }

// a Q62 coefficient and a value split into signed 32-bit halves
struct fx2 {
    int h, l;
};
__host__ __device__ constexpr fx2 fx_split(long long v) {
    return {int((v + 0x80000000LL) >> 32), int(static_cast<unsigned>(static_cast<unsigned long long>(v)))};
}
// cos and sin of the small DFTs, rounded to Q62
constexpr long long Q62_SQRT3_2 = 3993837246235628775LL;   // sqrt(3) / 2
constexpr long long Q62_SQRT1_2 = 3260954456333195553LL;   // sqrt(2) / 2
constexpr long long Q62_C1_9 = 3532756447825785444LL, Q62_S1_9 = 2964334632409774423LL;    // 2 pi / 9
constexpr long long Q62_C2_9 = 800810873071977681LL, Q62_S2_9 = 4541624145405292212LL;    // 4 pi / 9
constexpr long long Q62_C4_9 = -4333567320897763126LL, Q62_S4_9 = 1577289512995517789LL;   // 8 pi / 9

// a w for a real coefficient w: the product of the two low halves (at most one
// unit of the result) is dropped
__device__ __forceinline__ fx fx_mulc(fx a, fx2 w) {
    const fx2 s = fx_split(a.v);
    const long long mid = (long long)s.h * w.l + ((long long)s.l * w.h + (1LL << 29));
    return {(((long long)s.h * w.h) << 2) + (mid >> 30)};
}

// z (wr + i wi), |z| <= 2^61: every partial sum fits 64 bits
__device__ __forceinline__ cx<fx> fx_cmul(cx<fx> z, fx2 wr, fx2 wi) {
    const fx2 a = fx_split(z.x.v), b = fx_split(z.y.v);
    const long long hr = (long long)a.h * wr.h - (long long)b.h * wi.h;
    const long long hi = (long long)a.h * wi.h + (long long)b.h * wr.h;
    const long long mr = (long long)a.h * wr.l + (long long)a.l * wr.h - (long long)b.h * wi.l -
                         (long long)b.l * wi.h + (1LL << 29);
    const long long mi = (long long)a.h * wi.l + (long long)a.l * wi.h + (long long)b.h * wr.l +
                         (long long)b.l * wr.h + (1LL << 29);
    return {{(hr << 2) + (mr >> 30)}, {(hi << 2) + (mi >> 30)}};
}

// a b 2^-62 of two values (the pointwise products)
__device__ __forceinline__ long long fx_mul62(long long a, long long b) {
    const long long h = __mul64hi(a, b);
    const unsigned long long l = (unsigned long long)a * (unsigned long long)b;
    return (h << 2) | (long long)(l >> 62);
}
// v 2^s, rounded (s < 0: s > -64 or the result is 0)
__device__ __forceinline__ long long fx_shift(long long v, int s) {
    if (s >= 0) return v << s;
    if (s <= -63) return 0;
    return (v + (1LL << (-s - 1))) >> -s;
}

// ---- small DFTs (the radix-2 and radix-4 forms of fft_small.cuh use only
// sums and differences of T) --------------------------------------------------
__device__ __forceinline__ void fx_dft2(cx<fx>* v) {
    const cx<fx> a = v[0], b = v[1];
    v[0] = {a.x + b.x, a.y + b.y};
    v[1] = {a.x - b.x, a.y - b.y};
}
template <int S>
__device__ __forceinline__ void fx_dft3(cx<fx>& v0, cx<fx>& v1, cx<fx>& v2) {
    constexpr fx2 h = fx_split(S * Q62_SQRT3_2);
    const cx<fx> t1{v1.x + v2.x, v1.y + v2.y};
    const cx<fx> t2{{v0.x.v - (t1.x.v >> 1)}, {v0.y.v - (t1.y.v >> 1)}};
    const cx<fx> t3{fx_mulc(v1.x - v2.x, h), fx_mulc(v1.y - v2.y, h)};
    v0 = {v0.x + t1.x, v0.y + t1.y};
    v1 = {t2.x - t3.y, t2.y + t3.x};
    v2 = {t2.x + t3.y, t2.y - t3.x};
}
template <int S>
__device__ __forceinline__ void fx_dft4(cx<fx>* v) {
    const cx<fx> a0{v[0].x + v[2].x, v[0].y + v[2].y}, a1{v[0].x - v[2].x, v[0].y - v[2].y};
    const cx<fx> b0{v[1].x + v[3].x, v[1].y + v[3].y}, b1{v[1].x - v[3].x, v[1].y - v[3].y};
    const cx<fx> ib1 = S > 0 ? cx<fx>{-b1.y, b1.x} : cx<fx>{b1.y, -b1.x};
    v[0] = {a0.x + b0.x, a0.y + b0.y};
    v[2] = {a0.x - b0.x, a0.y - b0.y};
    v[1] = {a1.x + ib1.x, a1.y + ib1.y};
    v[3] = {a1.x - ib1.x, a1.y - ib1.y};
}
template <int S>
__device__ __forceinline__ void fx_dft8(cx<fx>* v) {
    cx<fx> e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    fx_dft4<S>(e);
    fx_dft4<S>(o);
    constexpr fx2 h = fx_split(Q62_SQRT1_2);
    // w^1 = h (1, S), w^2 = (0, S), w^3 = h (-1, S)
    const cx<fx> s1 = S > 0 ? cx<fx>{o[1].x - o[1].y, o[1].y + o[1].x} : cx<fx>{o[1].x + o[1].y, o[1].y - o[1].x};
    const cx<fx> s3 = S > 0 ? cx<fx>{-o[3].x - o[3].y, o[3].x - o[3].y} : cx<fx>{o[3].y - o[3].x, -o[3].y - o[3].x};
    const cx<fx> t1{fx_mulc(s1.x, h), fx_mulc(s1.y, h)};
    const cx<fx> t2 = S > 0 ? cx<fx>{-o[2].y, o[2].x} : cx<fx>{o[2].y, -o[2].x};
    const cx<fx> t3{fx_mulc(s3.x, h), fx_mulc(s3.y, h)};
    v[0] = {e[0].x + o[0].x, e[0].y + o[0].y};
    v[4] = {e[0].x - o[0].x, e[0].y - o[0].y};
    v[1] = {e[1].x + t1.x, e[1].y + t1.y};
    v[5] = {e[1].x - t1.x, e[1].y - t1.y};
    v[2] = {e[2].x + t2.x, e[2].y + t2.y};
    v[6] = {e[2].x - t2.x, e[2].y - t2.y};
    v[3] = {e[3].x + t3.x, e[3].y + t3.y};
    v[7] = {e[3].x - t3.x, e[3].y - t3.y};
}
// n = 3 a + b, k = c + 3 d: three 3-point DFTs over a, twiddles e^{S 2 pi i b c / 9},
// three 3-point DFTs over b
template <int S>
__device__ __forceinline__ void fx_dft9(cx<fx>* v) {
#pragma unroll
    for (int b = 0; b < 3; ++b) fx_dft3<S>(v[b], v[3 + b], v[6 + b]);
    // element 3 c + b now holds (b, c)
    v[4] = fx_cmul(v[4], fx_split(Q62_C1_9), fx_split(S * Q62_S1_9));
    v[5] = fx_cmul(v[5], fx_split(Q62_C2_9), fx_split(S * Q62_S2_9));
    v[7] = fx_cmul(v[7], fx_split(Q62_C2_9), fx_split(S * Q62_S2_9));
    v[8] = fx_cmul(v[8], fx_split(Q62_C4_9), fx_split(S * Q62_S4_9));
#pragma unroll
    for (int c = 0; c < 3; ++c) fx_dft3<S>(v[3 * c], v[3 * c + 1], v[3 * c + 2]);
    // k = c + 3 d from element 3 c + d: transpose
    cx<fx> t;
    t = v[1]; v[1] = v[3]; v[3] = t;
    t = v[2]; v[2] = v[6]; v[6] = t;
    t = v[5]; v[5] = v[7]; v[7] = t;
}
template <int R, int S>
__device__ __forceinline__ void fx_dft(cx<fx>* v) {
    if constexpr (R == 9) fx_dft9<S>(v);
    else if constexpr (R == 8) fx_dft8<S>(v);
    else if constexpr (R == 4) fx_dft4<S>(v);
    else if constexpr (R == 3) fx_dft3<S>(v[0], v[1], v[2]);
    else fx_dft2(v);
}

// ---- binary64 <-> fixed point ---------------------------------------------
__device__ __forceinline__ int f64_bexp(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }
__device__ __forceinline__ unsigned long long f64_mant(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return (b & 0xFFFFFFFFFFFFFULL) | (f64_bexp(x) ? 1ULL << 52 : 0ULL);
}
// |x| 2^34 / 2^(E - 1022 + 50), truncated, plus one: the leading 16 bits of x
// in units of 2^-16 of the largest value of biased exponent E
__device__ __forceinline__ unsigned f64_top16(double x, int E) {
    const int e = f64_bexp(x), sh = 37 + E - (e ? e : 1);
    return (sh < 64 ? unsigned(f64_mant(x) >> sh) : 0u) + 1u;
}
// round(x 2^k), |x 2^k| < 2^62
__device__ __forceinline__ long long f64_to_fx(double x, int k) {
    const int e = f64_bexp(x), sh = (e ? e : 1) - 1075 + k;
    const long long m = fx_shift((long long)f64_mant(x), sh);
    return __double2hiint(x) < 0 ? -m : m;
}
// d 2^e on the integer ALU where neither side is subnormal
__device__ __forceinline__ double f64_scale(double d, int e) {
    const int b = f64_bexp(d);
    if (b != 0 && b + e > 0 && b + e < 2047 && b != 2047)
        return __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
    return scalbn(d, e);
}

}  // namespace sph
