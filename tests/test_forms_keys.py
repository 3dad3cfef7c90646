"""The integer forms of comparisons, bounds, signs and differences (csrc/forms.cuh,
sub_near of csrc/common.cuh) against the operations themselves on the host: 4
million operand sets each, with NaN, signed zeros, infinities and subnormals, and
how many of the differences took the integer or binary32 path."""
import os

from forms_host import CSRC, run

SHIM = r"""
static int __clzll(long long x) { return x ? __builtin_clzll(x) : 64; }
static int min(int a, int b) { return a < b ? a : b; }
static long fell = 0, converted = 0;     // FP64 subtractions in sub_near, conversions in wind_diff
static double f2d(float f) { converted++; return (double)f; }
static float rcp_approx(float x) { return 1 / x; }
"""

MAIN = r"""
static std::mt19937_64 r(13);
template <class T> T any() {
    using L = std::numeric_limits<T>;
    const T ends[] = {0, -(T)0, L::min(), -L::min(), L::denorm_min(), -L::denorm_min(), L::max(), -L::max(),
                      L::infinity(), -L::infinity(), L::quiet_NaN(), -L::quiet_NaN(), 1, -1, 1 + L::epsilon()};
    const int how = (int)(r() % 4);
    if (how == 0) return ends[r() % 15];
    if (how == 1) return (T)((double)((int64_t)(r() % 2001) - 1000) / 8.0);   // close ones, equal ones
    // NaN quiet: the host's fmax treats signalling ones apart
    const T x = sizeof(T) == 8 ? (T)real(r()) : (T)real32((uint32_t)r());
    return std::isnan(x) ? std::copysign(L::quiet_NaN(), x) : x;
}
template <class T> T number() {
    T x;
    do x = any<T>(); while (std::isnan(x));
    return x;
}
template <class T> bool eq(T a, T b) { return a == b || (std::isnan(a) && std::isnan(b)); }   // either zero
template <class T> long compare() {
    long bad = 0;
    for (long i = 0; i < 4000000; i++) {
        const T a = any<T>(), b = any<T>(), m = number<T>(), n = number<T>();
        bad += le_num(a, b) != (a <= b);
        bad += !eq(min_num(m, n), std::fmin(m, n));
        bad += nonneg(m) != (m >= 0);
        bad += pos(m) != (m > 0) || nonzero(m) != (m != 0);
        bad += !same(abs_num(a), std::fabs(a));
        bad += same_num(m, m) != true || (m != n && same_num(m, n));
        T hi = any<T>(), lo = any<T>();
        Bounds<T> B(hi, lo);
        for (int k = (int)(r() % 7); k > 0; k--) {
            const T x = any<T>(), y = any<T>();
            B.take(x, y);
            hi = std::fmax(hi, x);
            lo = std::fmin(lo, y);
        }
        bad += !eq(B.max(), hi) || !eq(B.min(), lo);
        T pp = std::fabs(number<T>()), pm = std::fabs(number<T>()), p = pp, q = pm;
        add_signed(a, pp, pm);
        p += std::fmax((T)0, -a);
        q += std::fmax((T)0, a);
        bad += !same(pp, p) || !same(pm, q);
    }
    return bad;
}
int main() {
    const long b64 = compare<double>(), b32 = compare<float>();
    long keys = 0, wind = 0, exact = 0, near_ = 0, pairs = 0;
    for (long i = 0; i < 4000000; i++) {
        const double a = any<double>(), b = any<double>();
        keys += bits(of_okey(okey(a))) != bits(a);
        keys += is_nan(a) != std::isnan(a);
        if (!std::isnan(a) && !std::isnan(b) && a != b) keys += (okey(a) < okey(b)) != (a < b);
        const float u = any<float>(), v = i % 2 ? any<float>() : u * (1 + (float)(r() % 1000) * 1e-4f);
        converted = 0;
        wind += !same(wind_diff(u, v), (double)u - (double)v);
        exact += converted == 1;
        // neighbours of one field: a few per cent apart
        const double p = std::ldexp(1.0 + (double)(r() % 1000000007) / 1e9, (int)(r() % 40) - 20) * (r() & 1 ? 1 : -1);
        const double s = p * (1.0 + ((double)(r() % 2001) - 1000.0) * 1e-4);
        near_ += !same(sub_near(p, s), p - s) || !same(sub_near(a, b), a - b);
        fell = 0;
        sub_near(p, s);
        pairs += fell == 0;
    }
    printf("%ld %ld %ld %ld %ld %ld %ld\n", b64, b32, keys, wind, near_, exact, pairs);
}
"""


def test_integer_forms_have_the_results_of_the_operations(tmp_path):
    src = open(os.path.join(CSRC, "common.cuh")).read()
    sub = src[src.index("__device__ __forceinline__ double sub_near"):]
    sub = sub[:sub.index("\n}\n") + 3]
    assert sub.count("return a - b;") == 1
    sub = sub.replace("return a - b;", "fell++; return a - b;")
    b64, b32, keys, wind, near, exact, pairs = run(tmp_path, "forms.cuh", MAIN, SHIM + sub)
    assert (b64, b32, keys, wind, near) == (0, 0, 0, 0, 0)
    # the paths that the forms are for: close pairs nearly always, half of the
    # winds drawn here
    assert pairs >= 3.99e6 and exact >= 1.5e6
