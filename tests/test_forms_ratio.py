"""The limiter's ratio min(1, Q / P) (csrc/forms.cuh: fct_ratio) has the bits of
the division for every operand, overflowing and subnormal ones included."""
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
        if (!same(x, ref)) bad++;
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


def test_ratio_has_the_bits_of_the_division(tmp_path):
    bad32, bad64, n32, n64 = run(tmp_path, "forms.cuh", MAIN, PLAIN)
    assert bad32 == 0 and bad64 == 0
    assert n32 > 1e6 and n64 > 1e6
