// The binomial series of the equation of state, in a file that needs nothing but
// bit-cast and warp intrinsics, so that it also compiles on the host.
#pragma once

namespace grist {

// r^g for a ratio r close to 1 by the binomial series
// (1 + x)^g = sum_n C(g, n) x^n, Horner in FP64, with the binomial
// coefficients C(g, n) = C(g, n-1) (g - n + 1)/n formed on the host.  For
// |g| < 2 they are at most n + 1 in magnitude (about 2 for the g of air), so
// after N terms the omitted tail is below (N + 1) |x|^N: the warp takes the
// shortest series with |x|^N <= 2^-60 for the largest |x| among its lanes
// (N = 4, 5, 6, 8, 10 for |x| < 2^-15, 2^-12, 2^-10, 2^-8, 2^-6) - a
// warp-uniform branch, so no FP64 issue slot is spent on terms no lane
// needs.  A lane with |x| > 2^-6 uses the library pow().  mask: the lanes
// executing the call.
//
// Every term is in FP64: with the terms whose |x|^n is below 2^-30 in binary32
// (2 to 6 FP64 instructions instead of 3 to 9) the largest error, in units of
// 2^-53 against 64-bit significands, was 1.82 instead of 1.01 (g = -1.4,
// |x| < 2^-15).
struct Binom {
    double c[10];
    float f[6];   // the same coefficients in binary32 (GRIST_MIX_DF increments)
};

template <int N> __device__ __forceinline__ double horner(double x, const Binom &B) {
    double s = B.c[N - 1];
#pragma unroll
    for (int n = N - 2; n >= 0; n--) s = fma(s, x, B.c[n]);
    return s;
}

// (1 + x)^g for a small x given directly.
__device__ __forceinline__ double pow1p_near0(double x, double g, const Binom &B, unsigned mask) {
    // high word of |x|: exponent and leading fraction bits, monotone in |x|
    const unsigned hx = (unsigned)__double2hiint(x) & 0x7fffffffu;
    const unsigned hm = __reduce_max_sync(mask, hx);
    if (hm < 0x3f000000u) return horner<4>(x, B);    // |x| < 2^-15
    if (hm < 0x3f300000u) return horner<5>(x, B);    // 2^-12
    if (hm < 0x3f500000u) return horner<6>(x, B);    // 2^-10
    if (hm < 0x3f700000u) return horner<8>(x, B);    // 2^-8
    if (hx > 0x3f900000u || (hx == 0x3f900000u && __double2loint(x) != 0)) return pow(1.0 + x, g);
    return horner<10>(x, B);
}

inline Binom binomial(double g) {
    Binom b;
    b.c[0] = 1.0;
    for (int n = 1; n < 10; n++) b.c[n] = b.c[n - 1] * (g - (n - 1)) / n;
    for (int n = 0; n < 6; n++) b.f[n] = (float)b.c[n];
    return b;
}

}  // namespace grist
