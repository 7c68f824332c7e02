// fixed_check.cpp -- the block fixed-point pair terms of the FP64 evaluation
// (csrc/nb_fixed.cuh) on the CPU, against long double, beside the same terms
// in plain doubles.  Prints "ok <pairs>" or the first violated property.
//
// Classes of pairs: separations, velocities and accelerations from normal
// distributions over wide ranges of scale, eps = 0 and eps above and below the
// separation, cold systems (velocities, accelerations or both equal to a few
// parts in a thousand), one particle's vectors far larger than the other's.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <limits>
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

static const FxK K{1, 2};

struct Pair {
    double xi[3], xj[3], vi[3], vj[3], ai[3], aj[3], m, eps;
};
struct Term {
    L a[3], j[3], s[3], y;
};

template <class T>
static Term plain(const Pair &p) {
    T r[3], v[3], a[3];
    for (int k = 0; k < 3; ++k) {
        r[k] = (T)p.xj[k] - (T)p.xi[k];
        v[k] = (T)p.vj[k] - (T)p.vi[k];
        a[k] = (T)p.aj[k] - (T)p.ai[k];
    }
    const double e2 = p.eps * p.eps;
    const T r2 = std::fma(r[0], r[0], std::fma(r[1], r[1], std::fma(r[2], r[2], (T)e2)));
    const T y = (T)(1 / std::sqrt((L)r2)), y2 = y * y, q = (T)p.m * y2 * y;
    const T rv = std::fma(r[0], v[0], std::fma(r[1], v[1], r[2] * v[2]));
    const T w = std::fma(v[0], v[0], std::fma(v[1], v[1], std::fma(v[2], v[2],
                std::fma(r[0], a[0], std::fma(r[1], a[1], r[2] * a[2])))));
    const T al = rv * y2, be = std::fma(al, al, w * y2);
    Term o;
    for (int k = 0; k < 3; ++k) {
        const T w1 = std::fma(-3 * al, r[k], v[k]);
        const T w2 = std::fma(-3 * be, r[k], std::fma(-6 * al, w1, a[k]));
        o.a[k] = (L)q * (L)r[k];
        o.j[k] = (L)q * (L)w1;
        o.s[k] = (L)q * (L)w2;
    }
    o.y = y;
    return o;
}

// the device's pair (csrc/nb_eval.cuh), its FP64 differences and branch included
static Term fixed(const Pair &p) {
    double r[3];
    for (int k = 0; k < 3; ++k) r[k] = p.xj[k] - p.xi[k];
    uint64_t eps_x, mm;
    uint32_t emin, sign;
    int em;
    fx_eps2(p.eps * p.eps, eps_x, emin);
    fx_pack_mass(p.m, mm, em, sign);
    const Fx3 Vi = fx_pack(p.vi[0], p.vi[1], p.vi[2]), Vj = fx_pack(p.vj[0], p.vj[1], p.vj[2]);
    const Fx3 Ai = fx_pack(p.ai[0], p.ai[1], p.ai[2]), Aj = fx_pack(p.aj[0], p.aj[1], p.aj[2]);
    const Fx3 R = fx_decode(r, emin);
    const Fx3 V = fx_diff_norm(Vj.w, Vj.e, Vi.w, Vi.e), A = fx_diff_norm(Aj.w, Aj.e, Ai.w, Ai.e);
    FxS Rs[3], Vs[3];
    for (int k = 0; k < 3; ++k) {
        Rs[k] = fx_split(R.w[k]);
        Vs[k] = fx_split(V.w[k]);
    }
    const FxRoot t = fx_root(Rs, R.e, eps_x, emin, K);
    const double q = fx_q(fx_y3(t, K), t.g, mm, em, sign, false, K);
    double w1[3], w2[3];
    if (fx_inside(r, emin)) {
        double v[3], a[3];
        for (int k = 0; k < 3; ++k) {
            v[k] = fx_to_double(V.w[k], V.e - 61 + 1023);
            a[k] = fx_to_double(A.w[k], A.e - 61 + 1023);
        }
        const double y2 = fx_to_double((int64_t)t.y2, -60 - 2 * t.g + 1023);
        const double al = std::fma(r[0], v[0], std::fma(r[1], v[1], r[2] * v[2])) * y2;
        const double w = std::fma(v[0], v[0], std::fma(v[1], v[1], std::fma(v[2], v[2],
                         std::fma(r[0], a[0], std::fma(r[1], a[1], r[2] * a[2])))));
        const double be3 = 3.0 * std::fma(al, al, w * y2);
        for (int k = 0; k < 3; ++k) {
            w1[k] = std::fma(-3.0 * al, r[k], v[k]);
            w2[k] = std::fma(-be3, r[k], std::fma(-6.0 * al, w1[k], a[k]));
        }
    } else {
        const FxS Y2 = fx_split((int64_t)t.y2);
        const FxW1 u = fx_w1(Rs, Vs, V.w, t, Y2, K);
        int64_t x2[3];
        int ez;
        fx_w2(Rs, R.e, Vs, V.e, A, t, Y2, u, x2, ez, K);
        for (int k = 0; k < 3; ++k) {
            w1[k] = fx_to_double(u.w[k], V.e - 59 + 1023);
            w2[k] = fx_to_double(x2[k], ez - R.e - 52 + 1023);
        }
    }
    Term o;
    for (int k = 0; k < 3; ++k) {
        o.a[k] = (L)q * (L)r[k];
        o.j[k] = (L)q * (L)w1[k];
        o.s[k] = (L)q * (L)w2[k];
    }
    o.y = std::ldexp((L)t.y, -62 - t.g);
    return o;
}

static L norm(const L *a) { return std::sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]); }

static std::mt19937_64 rng(11);
static double gauss() { return std::normal_distribution<double>()(rng); }
static double uni(double lo, double hi) { return std::uniform_real_distribution<double>(lo, hi)(rng); }

struct Class {
    const char *name;
    double eps_lo, eps_hi;  // log10, eps_lo > eps_hi: eps = 0
    double d_lo, d_hi;      // separation, log10
    double v, v_common, a, a_common;  // random and common parts
    double skew;                      // factor on particle i's vectors
    double span;                      // further random scale, decades
};

static long check_class(const Class &c) {
    const int n = 60000;
    const L u = std::ldexp((L)1, -53);
    L sum[2][3] = {}, max_y = 0;
    long cnt[3] = {};
    for (int it = 0; it < n; ++it) {
        Pair p;
        p.eps = c.eps_lo > c.eps_hi ? 0.0 : std::pow(10.0, uni(c.eps_lo, c.eps_hi));
        const double d = std::pow(10.0, uni(c.d_lo, c.d_hi));
        const double sv = std::pow(10.0, uni(-c.span, c.span)), sa = std::pow(10.0, uni(-c.span, c.span));
        p.m = (uni(0, 1) < 0.1 ? -1.0 : 1.0) * std::pow(10.0, uni(-8, 2));
        for (int k = 0; k < 3; ++k) {
            p.xi[k] = c.span > 0 ? 0.0 : gauss();
            p.xj[k] = p.xi[k] + d * gauss();
            p.vi[k] = (c.v_common * (k + 1.3) + c.v * gauss()) * sv;
            p.vj[k] = (c.v_common * (k + 1.3) + c.v * gauss()) * sv;
            p.ai[k] = (c.a_common * (1.7 - k) + c.a * gauss()) * sa;
            p.aj[k] = (c.a_common * (1.7 - k) + c.a * gauss()) * sa;
            p.vi[k] *= c.skew;
            p.ai[k] *= c.skew;
        }
        const Term e = plain<L>(p), f = plain<double>(p), x = fixed(p);
        const L *te[3] = {e.a, e.j, e.s}, *tf[3] = {f.a, f.j, f.s}, *tx[3] = {x.a, x.j, x.s};
        max_y = std::max(max_y, std::fabs(x.y / e.y - 1));
        for (int t = 0; t < 3; ++t) {
            const L ne = norm(te[t]);
            if (!(ne > 0)) {  // a term that vanishes exactly vanishes here too
                CHECK(norm(tx[t]) == 0, "%s: term %d is not zero", c.name, t);
                continue;
            }
            L df[3], dx[3];
            for (int k = 0; k < 3; ++k) {
                df[k] = (tf[t][k] - te[t][k]) / ne;
                dx[k] = (tx[t][k] - te[t][k]) / ne;
            }
            sum[0][t] += df[0] * df[0] + df[1] * df[1] + df[2] * df[2];
            sum[1][t] += dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2];
            ++cnt[t];
        }
    }
    // the root: its argument carries the rounding of r's components (relative
    // u each, so 2 u in r^2 and u in y); its own error: r^2 within two units of
    // at least 2^58, the residual within two units of 2^-58, each halved in y
    CHECK(max_y <= 1.125 * u, "%s: 1/sqrt off by %Lg u", c.name, max_y / u);
    for (int t = 0; t < 3; ++t) {
        if (!cnt[t]) continue;
        const L rf = std::sqrt(sum[0][t] / cnt[t]), rx = std::sqrt(sum[1][t] / cnt[t]);
        std::printf("%-14s term %d: rms error %.3Lf u in doubles, %.3Lf u in fixed point\n", c.name, t,
                    rf / u, rx / u);
        CHECK(rx <= rf, "%s: term %d is less exact than in doubles", c.name, t);
    }
    return n;
}

static void check_conversions() {
    for (int it = 0; it < 200000; ++it) {
        int64_t w = (int64_t)(rng() >> (1 + rng() % 63));
        if (rng() & 1) w = -w;
        const int b = (int)(rng() % 1200) - 600;
        // exact up to the one's complement of a negative and half an ulp
        const double got = fx_to_double(w, b + 1023);
        const L ref = std::ldexp((L)w, b);
        CHECK(std::fabs((L)got - ref) <= std::ldexp((L)1, b) + std::fabs(ref) * std::ldexp((L)1, -53),
              "fx_to_double(%lld)", (long long)w);
        CHECK(fx_high(w) == 0 || fx_to_double_high(w, b + 1023) == got, "fx_to_double_high(%lld)", (long long)w);
        CHECK(w < 0 || w >> 53 || (L)got == ref, "fx_to_double(%lld) is not exact", (long long)w);
    }
    CHECK(fx_to_double(0, 1023) == 0.0, "zero");
    for (int it = 0; it < 100000; ++it) {
        const double e2 = std::ldexp(uni(1, 2), (int)(rng() % 1900) - 1000);
        uint64_t x;
        uint32_t em;
        fx_eps2(e2, x, em);
        const int E = (int)(em >> 20) - 1023;
        CHECK((x >> 58) != 0 && (x >> 60) == 0, "eps_x %llx", (unsigned long long)x);
        CHECK(std::ldexp((L)x, 2 * E - 58) == (L)e2, "eps2 %g", e2);
    }
    uint64_t x;
    uint32_t em;
    fx_eps2(0.0, x, em);
    CHECK(x == 0 && em == 0, "eps = 0");
    const double inf = std::numeric_limits<double>::infinity(), nan = std::nan("");
    for (double bad : {inf, -inf, nan, 1e200}) {
        CHECK(fx_pack(0.0, bad, 1.0).e == kFxBad, "a component %g must be flagged", bad);
    }
    const Fx3 z = fx_pack(0.0, -0.0, 0.0);
    CHECK(z.w[0] == 0 && z.w[1] == 0 && z.w[2] == 0 && z.e == kFxMinExp, "zero vector");
    // a vanishing or excluded mass gives exactly zero, a mass that is not finite no number
    const double r[3] = {0.3, -0.1, 0.2};
    const Fx3 R = fx_decode(r, 0);
    const FxS Rs[3] = {fx_split(R.w[0]), fx_split(R.w[1]), fx_split(R.w[2])};
    const FxRoot t = fx_root(Rs, R.e, 0, 0, K);
    uint64_t mm;
    uint32_t sg;
    int e;
    fx_pack_mass(0.0, mm, e, sg);
    CHECK(fx_q(fx_y3(t, K), t.g, mm, e, sg, false, K) == 0.0, "massless");
    fx_pack_mass(1.0, mm, e, sg);
    CHECK(fx_q(fx_y3(t, K), t.g, mm, e, sg, true, K) == 0.0, "excluded");
    CHECK(fx_q(fx_y3(t, K), t.g, mm, e, sg, false, K) > 0.0, "mass 1");
    fx_pack_mass(-1.0, mm, e, sg);
    CHECK(fx_q(fx_y3(t, K), t.g, mm, e, sg, false, K) < 0.0, "mass -1");
    for (double bad : {inf, nan}) {
        fx_pack_mass(bad, mm, e, sg);
        CHECK(!std::isfinite(fx_q(fx_y3(t, K), t.g, mm, e, sg, false, K)), "mass %g", bad);
    }
    // coincident particles without softening: no finite q
    const double zero[3] = {0, 0, 0};
    const Fx3 Z = fx_decode(zero, 0);
    const FxS Zs[3] = {fx_split(Z.w[0]), fx_split(Z.w[1]), fx_split(Z.w[2])};
    fx_pack_mass(1.0, mm, e, sg);
    const FxRoot z0 = fx_root(Zs, Z.e, 0, 0, K);
    CHECK(!std::isfinite(fx_q(fx_y3(z0, K), z0.g, mm, e, sg, false, K)), "r = 0, eps = 0");
}

int main() {
    const Class classes[] = {
        {"typical", -4, -4, -5, 1, 1, 0, 1, 0, 1, 0},
        {"near", -4, -4, -3, -1.5, 1, 0, 1, 0, 1, 0},
        {"unsoftened", 1, 0, -5, 1, 1, 0, 1, 0, 1, 0},
        {"bulk motion", -4, -4, -5, 1, 1e-3, 1, 1, 0, 1, 0},
        {"cold", -4, -4, -5, 1, 0, 0, 1e-3, 1, 1, 0},
        {"cold, moving", -4, -4, -5, 1, 1e-3, 1, 1e-3, 1, 1, 0},
        {"strong a", -4, -4, -5, 1, 1, 0, 1e6, 0, 1, 0},
        {"fast", -4, -4, -5, 1, 1e3, 0, 1, 0, 1, 0},
        {"uneven", -4, -4, -5, 1, 1, 0, 1, 0, 1e4, 0},
        {"softened", -2, -1, -5, -1, 1, 0, 1, 0, 1, 0},
        {"any scale", 1, 0, -30, 30, 1, 0, 1, 0, 1, 8},
        {"any eps", -30, 2, -30, 2, 1, 0, 1, 0, 1, 8},
    };
    check_conversions();
    long n = 0;
    for (const Class &c : classes) n += check_class(c);
    std::printf("ok %ld\n", n);
    return 0;
}
