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


TABLE = r"""
int main(int, char **) {
    std::mt19937_64 r(9);
    auto uni = [&](double a, double b) { return a + (b - a) * ((double)(r() >> 11) * 0x1p-53); };
    const double p0 = 1e5, rd = 287.04, kappa = rd / 1004.64;
    const Binom B = binomial(kappa - 1.0);
    for (double pi_top : {0.0, 225.0, 20000.0}) {
        int e2 = 0;
        std::frexp(p0 - pi_top, &e2);
        const int base = (1023 + e2 - 2) << 7;
        double table[2] = {0, 0}, power[2] = {0, 0}, p_new = 0, p_old = 0;   // largest, sum of squares
        const long n = 600000;
        for (long i = 0; i < n; i++) {
            // a layer of a stretched grid, a column of the table's two octaves
            const int L = i & 1 ? 60 : 30, k = (int)(r() % L);
            const double b0 = std::pow((double)k / L, 1.3), b1 = k + 1 == L ? 1.0 : std::pow((double)(k + 1) / L, 1.3);
            const double lo = __hiloint2double(base << 13, 0);
            double dps = lo * std::exp2(uni(0.0, 2.0));
            if (i % 5 == 0) {                        // a bin's edge, or the number before it
                dps = __hiloint2double((base + (int)(r() % 256)) << 13, 0);
                if (i % 2) dps = std::nextafter(dps, 0.0);
                if (dps < lo) dps = lo;
            }
            const int bin = (__double2hiint(dps) >> 13) - base;
            if (bin < 0 || bin > 255) { printf("bin\n"); return 1; }
            const double dB = b1 - b0, rdB = 1 / dB, rdps = 1 / dps, sum = b0 + b1, bm = 0.5 * sum,
                         bl = 0.5 * (b0 - (sum - b1)), th = dB * dps * uni(250, 500);
            const long double P = (long double)pi_top + ((long double)b0 + b1) / 2 * dps;
            const long double A = (long double)rd * ((long double)th / (((long double)b1 - b0) * dps)) *
                                  std::pow(P / p0, (long double)rd / (long double)1004.64) / P;
            const double2 e = exner_entry(pi_top, bm, bl, exner_centre(base, bin), p0, rd, kappa);
            const double a = th * exner_at(e, dps - exner_centre(base, bin), B) * (rdB * rdps);
            const double pk = std::fma(bm, dps, std::fma(bl, dps, pi_top));
            const double pw = 0.5 * (std::fma(b0, dps, pi_top) + std::fma(b1, dps, pi_top));
            const double w = rd * (th * rdB * rdps) * std::pow(pw / p0, kappa) / pw;
            const double ea = std::fabs((double)((a - A) / A)) * 0x1p53, ew = std::fabs((double)((w - A) / A)) * 0x1p53;
            table[0] = std::fmax(table[0], ea);
            table[1] += ea * ea;
            power[0] = std::fmax(power[0], ew);
            power[1] += ew * ew;
            p_new += std::pow((double)((pk - P) / P) * 0x1p53, 2);
            p_old += std::pow((double)((pw - P) / P) * 0x1p53, 2);
        }
        printf("%g %g %g %g %g %g ", table[0], std::sqrt(table[1] / n), power[0], std::sqrt(power[1] / n),
               std::sqrt(p_new / n), std::sqrt(p_old / n));
    }
    printf("%d\n", std::numeric_limits<long double>::digits);
}
"""


def test_alpha_from_the_table_is_as_accurate_as_from_the_power(tmp_path):
    """alpha and p over both octaves of the table, the bins' edges among them.
    alpha rounds in rdB, rdps, their product, the bracket, its product with the
    series, theta's and the last one, each 1 unit of 2^-53 (relative) at most,
    and pow() and the series once each: below 10 units; and no larger than with
    pow() of the pressure itself, both in the rms (to a hundredth)."""
    out = run(tmp_path, "series.cuh", TABLE, WARP)
    if out[-1] < 64:
        pytest.skip("no wider type on this machine")
    for j in range(3):
        top, rms, top_pow, rms_pow, p, p_pow = out[6 * j:6 * j + 6]
        assert top <= 10.0
        assert rms <= rms_pow * 1.01
        assert p <= p_pow * 1.01
