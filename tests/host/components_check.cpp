// components_check.cpp -- the FP64 evaluation's pair vectors (fx_vectors,
// csrc/nb_fixed.cuh) on the CPU, component by component: against long double,
// beside the same terms in plain doubles.  The error of a component is measured
// against its own summands (jerk: |v_k| + 3 |alpha r_k|, snap: |a_k| + 6 |alpha
// w1_k| + 3 |beta r_k|, alpha and beta from the absolute products), which is
// what doubles keep it small against, whatever the other components are.
// Prints "ok <pairs>" or the first violated property.
//
// Classes of pairs: systems thin along one axis or two, down to 1e-12; chains
// along x that move along y; bulk motion in the thin plane; every component of
// its own scale; isotropic ones; velocities and accelerations of 1e100 and more.
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
    L j[3], s[3];    // jerk and snap terms
    L cj[3], cs[3];  // the sums of their summands' absolute values
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
    L arv = 0, aw = 0;
    for (int k = 0; k < 3; ++k) {
        arv += std::fabs((L)r[k] * (L)v[k]);
        aw += (L)v[k] * (L)v[k] + std::fabs((L)r[k] * (L)a[k]);
    }
    const L aal = arv * (L)y2, abe = aw * (L)y2 + aal * aal, aq = std::fabs((L)q);
    for (int k = 0; k < 3; ++k) {
        const T w1 = std::fma(-3 * al, r[k], v[k]);
        const T w2 = std::fma(-3 * be, r[k], std::fma(-6 * al, w1, a[k]));
        o.j[k] = (L)q * (L)w1;
        o.s[k] = (L)q * (L)w2;
        const L c1 = std::fabs((L)v[k]) + 3 * aal * std::fabs((L)r[k]);
        o.cj[k] = aq * c1;
        o.cs[k] = aq * (std::fabs((L)a[k]) + 6 * aal * c1 + 3 * abe * std::fabs((L)r[k]));
    }
    return o;
}

// the device's pair (csrc/nb_eval.cuh)
static Term fixed(const Pair &p) {
    double r[3];
    for (int k = 0; k < 3; ++k) r[k] = (p.xj[k] + 0.0) - (p.xi[k] + 0.0);
    const FxP3 pj[2] = {fx_pack_components(p.vj), fx_pack_components(p.aj)};
    const FxP3 pi[2] = {fx_pack_components(p.vi), fx_pack_components(p.ai)};
    FxC3 D[2];
    int32_t top[2];
    fx_differences<2>(pj, pi, D, top);
    uint64_t eps_x, mm;
    uint32_t emin, sign;
    int em;
    fx_eps2(p.eps * p.eps, eps_x, emin);
    fx_pack_mass(p.m, mm, em, sign);
    FxRoot t;
    double w1[3], w2[3], x1[3], x2[3];
    fx_vectors<true>(r, D[0], D[1], std::max(top[0], top[1]), eps_x, emin, K, t, w1, w2);
    fx_vectors<false>(r, D[0], D[1], top[0], eps_x, emin, K, t, x1, x2);  // the 4th order's jerk
    const double q = fx_q(fx_y3(t, K), t.g, mm, em, sign, false, K);
    Term o;
    for (int k = 0; k < 3; ++k) {
        o.j[k] = (L)q * (L)w1[k];
        o.s[k] = (L)q * (L)w2[k];
        CHECK(w1[k] == x1[k], "w1 differs between the orders");
    }
    return o;
}

static std::mt19937_64 rng(17);
static double gauss() { return std::normal_distribution<double>()(rng); }
static double uni(double lo, double hi) { return std::uniform_real_distribution<double>(lo, hi)(rng); }

struct Class {
    const char *name;
    double sx[3], sv[3], sa[3];  // scales along the axes
    double common;               // bulk velocity and acceleration, in units of the scales
    double span;                 // decades of every component's own further scale
    double eps;
};

static long check_class(const Class &c) {
    const int n = 40000;
    const L u = std::ldexp((L)1, -53);
    L sum[2][2][3] = {};
    for (int it = 0; it < n; ++it) {
        Pair p;
        p.eps = c.eps;
        p.m = (uni(0, 1) < 0.1 ? -1.0 : 1.0) * std::pow(10.0, uni(-8, 2));
        const double d = std::pow(10.0, uni(-4, 0));
        for (int k = 0; k < 3; ++k) {
            const double tx = std::pow(10.0, uni(-c.span, c.span)), tv = std::pow(10.0, uni(-c.span, c.span)),
                         ta = std::pow(10.0, uni(-c.span, c.span));
            p.xi[k] = c.span > 0 ? 0.0 : c.sx[k] * gauss();
            p.xj[k] = p.xi[k] + c.sx[k] * d * gauss() * tx;
            p.vi[k] = c.sv[k] * (c.common * (k + 1.3) + gauss()) * tv;
            p.vj[k] = c.sv[k] * (c.common * (k + 1.3) + gauss()) * tv;
            p.ai[k] = c.sa[k] * (c.common * (1.7 - k) + gauss()) * ta;
            p.aj[k] = c.sa[k] * (c.common * (1.7 - k) + gauss()) * ta;
        }
        const Term e = plain<L>(p), f = plain<double>(p), x = fixed(p);
        for (int k = 0; k < 3; ++k) {
            const L te[2] = {e.j[k], e.s[k]}, tf[2] = {f.j[k], f.s[k]}, tx[2] = {x.j[k], x.s[k]};
            const L ce[2] = {e.cj[k], e.cs[k]};
            for (int t = 0; t < 2; ++t) {
                if (!(ce[t] > 0)) {  // a component without summands vanishes
                    CHECK(tx[t] == 0, "%s: component %d of term %d is not zero", c.name, k, t + 1);
                    continue;
                }
                const L df = (tf[t] - te[t]) / ce[t], dx = (tx[t] - te[t]) / ce[t];
                sum[0][t][k] += df * df;
                sum[1][t][k] += dx * dx;
            }
        }
    }
    for (int t = 0; t < 2; ++t)
        for (int k = 0; k < 3; ++k) {
            const L rf = std::sqrt(sum[0][t][k] / n) / u, rx = std::sqrt(sum[1][t][k] / n) / u;
            std::printf("%-16s term %d %c: rms error %.3Lf u in doubles, %.3Lf u here\n", c.name, t + 1, "xyz"[k], rf, rx);
            CHECK(rx <= rf, "%s: term %d, component %d is less exact than in doubles", c.name, t + 1, k);
        }
    return n;
}

// Ends of the range: what is finite in doubles is finite here, to 2^-44 of its
// summands, and what overflows there is not finite here.
static long check_ends() {
    long cnt = 0;
    for (int it = 0; it < 200000; ++it) {
        Pair p;
        p.eps = it % 2 ? 1e-4 : 0.0;
        p.m = 1.0;
        const double sx = std::pow(10.0, uni(-12, 12));
        const double sv = std::pow(2.0, uni(-300, 1017)), sa = std::pow(2.0, uni(-300, 1017));
        for (int k = 0; k < 3; ++k) {
            p.xi[k] = 0.0;
            p.xj[k] = sx * gauss();
            p.vi[k] = sv * uni(-1, 1);
            p.vj[k] = sv * uni(-1, 1);
            p.ai[k] = sa * uni(-1, 1);
            p.aj[k] = sa * uni(-1, 1);
        }
        const Term f = plain<double>(p), e = plain<L>(p), x = fixed(p);
        for (int k = 0; k < 3; ++k)
            for (int t = 0; t < 2; ++t) {
                const L tf = t ? f.s[k] : f.j[k], te = t ? e.s[k] : e.j[k], tx = t ? x.s[k] : x.j[k];
                const L ce = t ? e.cs[k] : e.cj[k], q = std::fabs(e.cj[k]);
                if (std::isfinite((double)tf)) {
                    CHECK(std::fabs(tx - te) <= std::ldexp(ce, -44), "finite in doubles: %Lg, %Lg here, exactly %Lg", tf, tx, te);
                    ++cnt;
                } else if (std::fabs(te) > std::numeric_limits<double>::max() && q < std::numeric_limits<double>::max()) {
                    CHECK(!std::isfinite((double)tx), "overflow: %Lg, %Lg here", te, tx);
                }
            }
    }
    CHECK(cnt > 400000, "cases %ld", cnt);
    // what is not finite is seen in the exponent fields
    const double inf = std::numeric_limits<double>::infinity(), nan = std::nan("");
    for (double bad : {inf, -inf, nan})
        for (int k = 0; k < 3; ++k) {
            double b[3] = {1.0, 0.0, -2.0}, o[3] = {0.1, -0.5, 0.4};
            b[k] = bad;
            const FxP3 B = fx_pack_components(b), O = fx_pack_components(o);
            FxC3 D;
            int32_t f;
            fx_differences<1>(&B, &O, &D, &f);
            CHECK(f == 0x7ff, "component %d %g of j", k, bad);
            fx_differences<1>(&O, &B, &D, &f);
            CHECK(f == 0x7ff, "component %d %g of i", k, bad);
            fx_differences<1>(&O, &O, &D, &f);
            CHECK(f < 0x7ff && D.w[k] == 0, "finite");
        }
    return cnt;
}

int main() {
    const Class classes[] = {
        {"isotropic", {1, 1, 1}, {1, 1, 1}, {1, 1, 1}, 0, 0, 1e-4},
        {"unsoftened", {1, 1, 1}, {1, 1, 1}, {1, 1, 1}, 0, 0, 0},
        {"softened", {1, 1, 1}, {1, 1, 1}, {1, 1, 1}, 0, 0, 10},
        {"thin 1e-2", {1, 1, 1e-2}, {1, 1, 1e-2}, {1, 1, 1e-2}, 0, 0, 1e-4},
        {"thin 1e-4", {1, 1, 1e-4}, {1, 1, 1e-4}, {1, 1, 1e-4}, 0, 0, 1e-4},
        {"thin 1e-6", {1, 1, 1e-6}, {1, 1, 1e-6}, {1, 1, 1e-6}, 0, 0, 0},
        {"thin 1e-12", {1, 1, 1e-12}, {1, 1, 1e-12}, {1, 1, 1e-12}, 0, 0, 1e-2},
        {"thin, softened", {1, 1, 1e-6}, {1, 1, 1e-6}, {1, 1, 1e-6}, 0, 0, 10},
        {"thin, moving", {1, 1, 1e-5}, {1, 1, 1e-5}, {1, 1, 1e-5}, 1e4, 0, 1e-4},
        {"needle", {1, 1e-5, 1e-9}, {1, 1e-5, 1e-9}, {1, 1e-5, 1e-9}, 0, 0, 0},
        {"chain", {1, 1e-8, 1e-8}, {1e-8, 1, 1e-8}, {1e-8, 1e-8, 1}, 0, 0, 0},
        {"planar", {1, 1, 0}, {1, 1, 0}, {1, 1, 0}, 0, 0, 1e-4},
        {"cold", {1, 1, 1e-4}, {0, 0, 0}, {1, 1, 1e-4}, 0, 0, 1e-4},
        {"strong a", {1, 1, 1e-4}, {1, 1, 1e-4}, {1e6, 1e6, 1e2}, 0, 0, 1e-4},
        {"fast", {1, 1, 1e-4}, {1e4, 1e4, 1}, {1, 1, 1e-4}, 0, 0, 1e-4},
        {"own scales", {1, 1, 1}, {1, 1, 1}, {1, 1, 1}, 0, 6, 0},
        {"huge", {1, 1, 1e-3}, {1e120, 1e120, 1e117}, {1e180, 1e180, 1e177}, 0, 0, 1e-4},
        {"tiny", {1, 1, 1e-3}, {1e-120, 1e-120, 1e-123}, {1e-200, 1e-200, 1e-203}, 0, 0, 1e-4},
    };
    long n = check_ends();
    for (const Class &c : classes) n += check_class(c);
    std::printf("ok %ld\n", n);
    return 0;
}
