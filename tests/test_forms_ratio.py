"""The limiter's ratio min(1, Q / P) (csrc/forms.cuh: fct_ratio) is the division's
value for every operand, overflowing and subnormal ones included, from any
binary32 reciprocal within one ulp."""
from forms_host import PLAIN, run

MAIN = r"""
template <class T> T pick(std::mt19937_64 &r, int how) {
    using L = std::numeric_limits<T>;
    const T ends[] = {0, -(T)0, L::min(), L::denorm_min(), -L::denorm_min(), L::max(), -L::max(), L::infinity(),
                      -L::infinity(), L::quiet_NaN(), 1, -1, L::min() * 3, L::epsilon()};
    if (how == 0) return ends[r() % 14];
    T x;
    do {
        if (sizeof(T) == 8) x = (T)real(r());
        else x = (T)real32((uint32_t)r());
    } while (std::isnan(x) && how == 1);
    return x;
}
template <class T> void check(long &bad, long &divided) {
    std::mt19937_64 r(11);
    for (long i = 0; i < 4000000; i++) {
        T Q = pick<T>(r, (int)(r() % 5)), P = std::fabs(pick<T>(r, (int)(r() % 5)));
        if (i % 3 == 0) {   // operands of one size, as in a limited cell
            P = std::ldexp((T)(1.0 + (double)(r() % 1000000007) / 1e9), (int)(r() % 80) - 40);
            Q = P * (T)((double)(r() % 1000000007) / 0.8e9);
        }
        if (i % 11 == 0) P = std::numeric_limits<T>::infinity();
        if (P < std::numeric_limits<T>::min()) P = std::numeric_limits<T>::min();
        const T ref = std::fmin((T)1, Q / P), x = fct_ratio(Q, P);
        // large operands: the scaled remainder of a quotient below 2^-100, or the
        // scaled P of one beyond -2^120, leaves the normal range
        const bool large = sizeof(T) == 4 && std::fmax(std::fabs(Q), P) >= (T)0x1p62;
        if (large && std::fabs(ref) < (T)0x1p-100) {
            if (!(std::fabs(x - ref) <= std::fabs(ref) * (T)0x1p-22 + (T)0x1p-148)) bad++;
        } else if (large && ref < -(T)0x1p120) {
            if (!(x < -(T)0x1p119)) bad++;
        } else if (!(x == ref)) {
            bad++;
        }
        if (Q < P && Q != 0) divided++;
    }
}
int main() {
    long b32 = 0, b64 = 0, n32 = 0, n64 = 0;
    check<float>(b32, n32);
    check<double>(b64, n64);
    printf("%ld %ld %ld %ld\n", b32, b64, n32, n64);
}
"""


def test_ratio_is_the_quotient(tmp_path):
    bad32, bad64, n32, n64 = run(tmp_path, "forms.cuh", MAIN, PLAIN)
    assert bad32 == 0 and bad64 == 0
    assert n32 > 1e6 and n64 > 1e6
