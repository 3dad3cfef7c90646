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

// Reference columns of the hydrostatic equation of state.  pow() costs about
// 100 FP64 instructions, which bounded the hydrostatic diagnostics (pipe 90 %
// active); but Rd (p/p0)^kappa / p at level k depends on the column's mass
// dps = ps - pi_top alone, p = pi_top + B_k dps with the mid-layer coordinate
// B_k, so a table of reference columns turns it into a short series: with the
// reference at the middle dps_c of the bin that dps falls in,
//   Rd (p/p0)^kappa / p = [Rd (p_c/p0)^kappa / p_c] (1 + x)^(kappa - 1),
//   x = B_k (dps - dps_c) / p_c,   |x| <= 2^-8 since B_k dps_c <= p_c,
// summed by the 8-term series of pow1p_near0 (tail below 2^-60).  A bin is one
// value of the exponent and the first 7 fraction bits of dps; the table
// covers the two octaves that end at twice the one of p0 - pi_top (32.8 to
// 131 kPa for p0 = 1e5), other columns call pow().
__device__ __forceinline__ double exner_centre(int base, int bin) {
    return __hiloint2double(((base + bin) << 13) | (1 << 12), 0);
}

// Entry {the bracket, B_k / p_c} for B_k = bm + bl.  The bracket carries the
// error of pow() and half an ulp: the roundings of p_c, of p_c/p0 and of the
// product are collected and added at the end.  With a plain bracket and the
// series rounded before the product, the largest error of alpha was 6.7 to 7.4
// units of 2^-53 and its rms 1.45, where pow() of the pressure itself gives 6.2
// and 1.30; as it is, 5.6 and 1.23.
__device__ __forceinline__ double2 exner_entry(double pi_top, double bm, double bl, double c, double p0, double rd,
                                               double kappa) {
    const double h = __dmul_rn(bm, c), s = __dadd_rn(pi_top, h), b = __dadd_rn(s, -pi_top);
    const double e = __dadd_rn(__dadd_rn(pi_top, -__dadd_rn(s, -b)), __dadd_rn(h, -b)) + fma(bl, c, fma(bm, c, -h));
    const double pc = __dadd_rn(s, e), dpc = __dadd_rn(e, -__dadd_rn(pc, -s));   // p_c = pc + dpc
    const double q = pc / p0, dq = fma(-q, p0, pc) + dpc;                       // p_c/p0 = q (1 + dq/pc)
    const double y = pow(q, kappa), t = __dmul_rn(rd, y), z = t / pc;
    const double dt = fma(rd, y, -t) + t * ((kappa * dq - dpc) / pc);
    return make_double2(z + (fma(-z, pc, t) + dt) / pc, bm / pc);
}

// The bracket times (1 + x)^(kappa - 1), x = r.y off: the series less its one is
// added in the product, which rounds once.
__device__ __forceinline__ double exner_at(double2 r, double off, const Binom &B) {
    const double x = r.y * off;
    double s = B.c[7];
#pragma unroll
    for (int n = 6; n >= 1; n--) s = fma(s, x, B.c[n]);
    return fma(r.x, x * s, r.x);
}

}  // namespace grist
