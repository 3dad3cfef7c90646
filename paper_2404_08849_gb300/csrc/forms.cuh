// Comparisons, signs, differences and ratios of binary64 (and their binary32
// counterparts) kept off the FP64 pipe, shared by the kernels.  The file needs
// f2d, sub_near and rcp_approx (common.cuh) and the bit-cast and rounding intrinsics only, so
// that it also compiles on the host.
#pragma once

namespace grist {

// Comparisons, maxima and minima of binary64 in integer arithmetic.  A DSETP
// occupies the FP64 pipe, which bounds the FP64 policy, like an addition: 64
// cycles of a scheduler for a warp; the integer form is 8 to 12 instructions of
// the otherwise idle ALU.  The order key of a double's bits: negative
// numbers with their magnitude bits inverted, so that keys compare like the
// numbers (+-NaN beyond the infinities); the map is its own inverse.
__device__ __forceinline__ long long okey(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double of_okey(long long k) {
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}
constexpr long long kKeyInf = 0x7ff0000000000000ll;       // of +infinity
constexpr long long kKeyNegInf = ~kKeyInf;                 // of -infinity

// x >= 0, with -0 (NaN by its sign)
__device__ __forceinline__ bool nonneg(double x) {
    const long long b = __double_as_longlong(x);
    return b >= 0 || b == (long long)0x8000000000000000ull;
}
__device__ __forceinline__ bool nonneg(float x) { return x >= 0.f; }
// x > 0 and x != 0 for the finite mesh weights
__device__ __forceinline__ bool pos(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool pos(float x) { return x > 0.f; }
__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }
__device__ __forceinline__ bool nonzero(float x) { return x != 0.f; }
__device__ __forceinline__ bool is_nan(double x) { return (__double_as_longlong(x) & 0x7fffffffffffffffll) > kKeyInf; }

// Running maximum and minimum that ignore NaN as fmax and fmin do.
template <typename TC> struct Bounds;
template <> struct Bounds<float> {
    float hi, lo;
    __device__ __forceinline__ Bounds() {}
    __device__ __forceinline__ Bounds(float a, float b) : hi(a), lo(b) {}
    __device__ __forceinline__ void take(float a, float b) {
        hi = fmaxf(hi, a);
        lo = fminf(lo, b);
    }
    __device__ __forceinline__ float max() const { return hi; }
    __device__ __forceinline__ float min() const { return lo; }
};
template <> struct Bounds<double> {
    long long hi, lo;   // keys; NaN starts as the key that every number beats
    __device__ __forceinline__ Bounds() {}
    __device__ __forceinline__ Bounds(double a, double b) : hi(okey(a)), lo(okey(b)) {
        if (hi > kKeyInf) hi = (long long)0x8000000000000000ull;
        if (lo < kKeyNegInf) lo = 0x7fffffffffffffffll;
    }
    __device__ __forceinline__ void take(double a, double b) {
        const long long ka = okey(a), kb = okey(b);
        if (ka > hi && ka <= kKeyInf) hi = ka;
        if (kb < lo && kb >= kKeyNegInf) lo = kb;
    }
    __device__ __forceinline__ double max() const { return of_okey(hi); }
    __device__ __forceinline__ double min() const { return of_okey(lo); }
};
// min(a, b) of two numbers (no NaN)
__device__ __forceinline__ float min_num(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double min_num(double a, double b) { return okey(b) < okey(a) ? b : a; }

// a <= b (false for NaN), |a|
__device__ __forceinline__ bool le_num(float a, float b) { return a <= b; }
__device__ __forceinline__ bool le_num(double a, double b) {
    const long long ka = okey(a), k = okey(b), kb = k == -1 ? 0 : k;   // -0 as 0
    return ka <= kb && kb <= kKeyInf && ka >= kKeyNegInf;
}
__device__ __forceinline__ float abs_num(float x) { return fabsf(x); }
__device__ __forceinline__ double abs_num(double x) { return fabs(x); }
// a == b for a value and a copy of it
__device__ __forceinline__ bool same_num(float a, float b) { return a == b; }
__device__ __forceinline__ bool same_num(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }

// pm += max(0, x), pp += max(0, -x): the other sum would gain a zero, so one
// addition serves both.  NaN adds nothing.
__device__ __forceinline__ void add_signed(float x, float &pp, float &pm) {
    pp += fmaxf(0.f, -x);
    pm += fmaxf(0.f, x);
}
__device__ __forceinline__ void add_signed(double x, double &pp, double &pm) {
    const bool neg = __double2hiint(x) < 0;
    const double acc = neg ? pp : pm;
    double sum = acc + fabs(x);
    if (is_nan(x)) sum = acc;
    pp = neg ? sum : pp;
    pm = neg ? pm : sum;
}

// min(1, Q / P) for P >= TINY > 0, the division's value (1 where that is NaN).
// binary32: Markstein's division (IBM J. Res. Dev. 34, 1990).  From a reciprocal
// within one ulp one Newton step gives the correctly rounded one, except where
// all bits of P's significand are set (one in 2^23); the product with it,
// corrected by its remainder, is the rounded quotient.  The scaling by a power of
// two keeps every intermediate normal (left over: operands of 2^62 and more with a
// quotient below 2^-100, to 2 ulp, or beyond -2^120, perhaps -infinity).  Where
// that is NaN, by P = infinity (0) or a quotient beyond the range (infinite), the
// plain product stands.  No branches, so that a
// thread's eight ratios overlap: k_tr_ratios, level 7, 4 tracers, 60 levels, us a
// launch 345; the division itself, which takes its slow path (a call) where P is
// near TINY, that is wherever a tracer is constant, 545; the division behind
// Q < P and Q != 0, 359.
__device__ __forceinline__ float fct_ratio(float Q, float P) {
    const float s = fmaxf(fabsf(Q), P) < 0x1p62f ? 0x1p64f : 0x1p-64f, p = P * s, q = Q * s;
    float y = rcp_approx(p);
    const float plain = q * y;
    y = fmaf(fmaf(-p, y, 1.f), y, y);
    float a = q * y;
    a = fmaf(fmaf(-a, p, q), y, a);
    a = a == a ? a : plain;
    return fminf(1.f, a);
}
// binary64: the division, reached only where Q < P (decided on the keys) and not
// for Q = 0; 2107 us there, 2813 with a refined reciprocal and one correction.
__device__ __forceinline__ double fct_ratio(double Q, double P) {
    if (okey(Q) >= okey(P) || is_nan(Q) || is_nan(P)) return 1.0;
    if (!nonzero(Q)) return Q;
    const double a = Q / P;
    return is_nan(a) ? 1.0 : a;
}

// (double)a - (double)b of two binary32 numbers, bit for bit: where the binary32
// difference is exact (its TwoSum error is zero) it is that number.
__device__ __forceinline__ double wind_diff(double a, double b) { return sub_near(a, b); }
__device__ __forceinline__ double wind_diff(float a, float b) {
    const float s = __fsub_rn(a, b), bb = __fsub_rn(s, a);
    const float err = __fsub_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fadd_rn(b, bb));
    if (err == 0.f) return f2d(s);
    return f2d(a) - f2d(b);
}

}  // namespace grist
