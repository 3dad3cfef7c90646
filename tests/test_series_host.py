"""The series of the equation of state (csrc/series.cuh) on the host, against
64-bit significands (long double, where that is wider than binary64)."""
import pytest

from forms_host import run

WARP = """
static unsigned __reduce_max_sync(unsigned, unsigned x) { return x; }
static double __dmul_rn(double a, double b) { return a * b; }
static double __dadd_rn(double a, double b) { return a + b; }
struct double2 { double x, y; };
static double2 make_double2(double x, double y) { return double2{x, y}; }
"""

POW = r"""
int main() {
    std::mt19937_64 r(5);
    double worst = 0;
    const double cp = 1004.64, rd = 287.04, gs[] = {cp / (cp - rd), -cp / (cp - rd), rd / cp - 1, 1.999, -1.999, 0.5};
    for (double g : gs) {
        const Binom B = binomial(g);
        for (long i = 0; i < 400000; i++) {
            const double m = std::exp2(-6.0 - 24.0 * (double)(r() >> 11) * 0x1p-53), x = r() & 1 ? m : -m;
            const long double e = std::pow((long double)1 + x, (long double)g);
            const double err = std::fabs((double)((pow1p_near0(x, g, B, 1u) - e) / e)) * 0x1p53;
            const double bound = 1 + 3 * std::fabs(g * x) + 11 * 0x1p-7;
            worst = std::fmax(worst, err / bound);
        }
    }
    printf("%g %d\n", worst, std::numeric_limits<long double>::digits);
}
"""


def test_power_of_a_ratio_near_one(tmp_path):
    """The last addition rounds once, 2^-53 of the result; what it adds, g x,
    carries three roundings of its own; |C(g, n)| <= n + 1 for |g| < 2, so the
    terms omitted after N are below (N + 1) |x|^N, 11 2^-60 at most."""
    worst, digits = run(tmp_path, "series.cuh", POW, WARP)
    assert worst <= 1.0 and digits >= 53
    if digits < 64:
        pytest.skip("no wider type on this machine: the reference rounds too")
