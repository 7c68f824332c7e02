// root_check.cpp -- 1/sqrt(r^2 + eps^2) as the potentials take it
// (csrc/nb_fixed.cuh), over all separations: as a pair of floats (pair terms) it is
// exact to 2^-46 or no number, as a double (energies) to 2^-52 over the doubles'
// range, never of the wrong sign or scale.  Prints "ok <cases>" or the first
// violation.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../../paper_1812_00367_gb300/csrc/nb_fixed.cuh"

using namespace nb;
typedef long double L;

#define CHECK(cond, ...)                       \
    do {                                       \
        if (!(cond)) {                         \
            std::printf("FAIL %s: ", #cond);   \
            std::printf(__VA_ARGS__);          \
            std::printf("\n");                 \
            std::exit(1);                      \
        }                                      \
    } while (0)

int main() {
    const FxK K{1, 2};
    std::mt19937_64 rng(5);
    long n = 0, inside = 0, nans = 0;
    for (int it = 0; it < 400000; ++it) {
        const double eps = it % 4 == 0 ? std::ldexp(1.0 + (double)(rng() >> 12) * 0x1p-52, (int)(rng() % 300) - 200) : 0.0;
        double r[3];
        const int e = (int)(rng() % 2000) - 980;
        for (int k = 0; k < 3; ++k) r[k] = std::ldexp((double)(int64_t)rng(), e - 63);
        uint64_t eps_x;
        uint32_t emin;
        fx_eps2(eps * eps, eps_x, emin);
        const Fx3 R = fx_decode(r, emin);
        const FxS Rs[3] = {fx_split(R.w[0]), fx_split(R.w[1]), fx_split(R.w[2])};
        const FxRoot t = fx_root(Rs, R.e, eps_x, emin, K);
        // 1/sqrt of the scaled sum: long double has the range of the squares
        const L x = r[0], y = r[1], z = r[2], e2 = (L)(eps * eps);
        const L want = 1 / std::sqrt(x * x + y * y + z * z + e2);
        const double d = fx_root_to_double(t, R.e);
        CHECK(std::fabs((L)d - want) <= want * 0x1p-51L, "double: r %g %g %g eps %g: %g", r[0], r[1], r[2], eps, d);
        float yh, yl;
        fx_root_to_floats(t, yh, yl);
        if (want > 0x1p-100L && want < 0x1p125L) {
            CHECK(std::fabs((L)yh + (L)yl - want) <= want * 0x1p-46L, "floats: r %g: %g", r[0], yh);
            ++inside;
        } else if (want < 0x1p-104L || want > 0x1p127L) {
            CHECK(std::isnan(yh), "floats outside their range: r %g: %g", r[0], yh);
            ++nans;
        } else {
            CHECK(std::isnan(yh) || std::fabs((L)yh + (L)yl - want) <= want * 0x1p-46L, "floats at an end: r %g: %g", r[0], yh);
        }
        ++n;
    }
    // beyond the doubles' squares and at their very end: positive and tiny
    for (double big : {0x1p1020, 0x1p1021, 0x1p1022, 1.7e308}) {
        const double r[3] = {big, -big, big};
        const Fx3 R = fx_decode(r, 0);
        const FxS Rs[3] = {fx_split(R.w[0]), fx_split(R.w[1]), fx_split(R.w[2])};
        const double d = fx_root_to_double(fx_root(Rs, R.e, 0, 0, K), R.e);
        CHECK(d > 0 && d < 1e-300, "r = %g: %g", big, d);
    }
    CHECK(inside > 10000 && nans > 10000, "%ld inside, %ld outside", inside, nans);
    std::printf("ok %ld\n", n);
    return 0;
}
