// nb_eval.cuh -- the hot O(N_active x N) evaluation of acceleration, jerk,
// snap and potential (the paper's Sec. 4 kernel; 6th-order Hermite pair terms
// of Nitadori & Makino 2008) in three arithmetics, plus its j-split reduction.
//
// Per pair, with r = x_j - x_i, v = v_j - v_i, a = a_j - a_i (predicted),
// y = (r.r + eps^2)^{-1/2}, q = m_j y^3, alpha = (r.v) y^2, zeta = (v.v + r.a) y^2,
// beta = zeta + alpha^2:
//   w1 = v - 3 alpha r,            A1 = q w1         (jerk term)
//   w2 = a - 6 alpha w1 - 3 beta r, A2 = q w2         (snap term)
//   A0 = q r,  pot -= m_j y
// i.e. NM08's A1 = m v/s^3 - 3 alpha A0 and A2 = m a/s^3 - 6 alpha A1 - 3 beta A0
// with the large alpha terms cancelling inside each pair before it is summed
// (that keeps the FP32 path within its bound on strongly cancelling sums).
// FP64: the pair terms run in fixed point on the integer pipes
// (nb_fixed.cuh); 12 FP64 instructions per pair remain, the coordinate
// differences and the nine running sums (9 in the 4th-order form); the
// potential m y is summed in float-float on the FP32 pipe.  The 4th-order
// scheme (Makino & Aarseth 1992) keeps A0, A1 and the potential only
// (interact4).
//
// Work decomposition: a piece of work is (cluster, i-tile, j-range).  An
// i-tile holds kTPB / gl active particles; gl lanes of a warp share one i and
// take every gl-th j of each tile (gl = 1: i-parallel, j broadcast from
// shared memory; gl = 32: j-parallel for tiny active sets, warp-shuffle
// reduction).  A batch of clusters is cut into split items (each cluster's j
// range split S ways, items fetched dynamically); a single cluster into
// stream-K ranges (CTA k takes units [U k / G, U (k+1) / G) of the U =
// i-tiles x j-tiles units).  j-tiles of kTJ particles are copied global ->
// shared by the TMA engine (cp.async.bulk) into a ring of stages guarded by
// mbarriers.  When an i-tile's j range is covered by several pieces, each
// writes FP64 partial sums; the CTA that finishes the i-tile last (atomic
// counter) adds them in piece order (deterministic) and finalises.  Thread 0
// describes each piece in a shared-memory record so that the pair loop keeps
// only its own state in registers.
#pragma once

#include <type_traits>

#include "nb_fixed.cuh"
#include "nb_internal.cuh"
#include "nb_step.cuh"

namespace nb {

template <int P>
struct Prec;

// ===================================================================== FP64
// Fixed-point pair terms (nb_fixed.cuh): the coordinate differences and the nine
// running sums stay on the FP64 pipe (12 instructions per pair, 9 in the 4th-order
// form), everything between them runs on the integer pipes.
// Bound: the issue of half-rate integer instructions (shifts, logic,
// IMAD.WIDE; 760 instructions a pair and warp, 461 in the 4th-order form; ALU 59 %
// and FP64 pipe 54 % busy).
// Measured, N = 65536, A = 1000: 2.46 ms (2.67e10 pairs/s) against 5.70 ms for the
// same terms in doubles (50 DFMA a pair, the FP64 pipe 95 % busy); A = 48: 154
// against 324 us; all: 151 against 361 ms.  Residency: 3 and 4 CTAs per SM measured within 1 % of one
// another over the FP64 cases (A = 48 3 % faster, a batch 3 % slower with 3).
// Converting w1, w2 with the count of leading zeros of the high word (a general
// conversion where a component is that small) instead of a float's exponent: 138.6
// -> 133.2 ms for all pairs of N = 65536, with one exponent a vector.
template <>
struct Prec<NB_FP64> {
    using J = JFX;
    static constexpr int kPerRec = 1;  // particles per record
    struct I {
        double x[3];
        FxP3 v, a;
        double m1;       // -1.0 from the kernel parameters (see Dev)
        uint64_t eps_x;  // eps^2 as a fixed-point number and its block exponent
        uint32_t emin;
        FxK K;
    };
    struct Acc {
        double a[3], j[3], s[3], p;
        ff pf;         // the current j-tile's potential as a float pair
        int32_t fv, fa;  // largest exponent field of a velocity, an acceleration
    };
    static __device__ __forceinline__ void prepare(I &i, const Dev &d) {
        i.m1 = d.neg_one;
        i.eps_x = d.eps_x;
        i.emin = d.eps_emin;
        i.K = d.fxk;
    }
    static __device__ __forceinline__ I load_i(const J *jarr, int64_t k) {
        const J e = jarr[k];
        I r;
#pragma unroll
        for (int q = 0; q < 3; ++q) r.x[q] = e.x[q];
        r.v = jfx_v(e);
        r.a = jfx_a(e);
        return r;
    }
    static __device__ __forceinline__ void zero(Acc &c) {
#pragma unroll
        for (int k = 0; k < 3; ++k) c.a[k] = c.j[k] = c.s[k] = 0.0;
        c.p = 0.0;
        c.pf = ff{0.f, 0.f};
        c.fv = c.fa = 0;
    }
    // potential term m y in float-float, renormalised every term (|lo| stays
    // below half an ulp of hi): a 64-term tile sum is good to ~2^-45, and
    // tiles add up in FP64
    static __device__ __forceinline__ void pot_term(float2 m, float yh, float yl, ff &sum) {
        const bool none = m.x == 0.f;  // massless or excluded: zero at any separation
        sum = ff_add(sum, ff_mul_lazy(ff{m.x, m.y}, ff{none ? 0.f : yh, none ? 0.f : yl}));
    }
    // After 64 pairs: their float-pair potential joins the FP64 total.
    static __device__ __forceinline__ void tile_done(Acc &c) {
        c.p += (double)c.pf.hi + (double)c.pf.lo;
        c.pf = ff{0.f, 0.f};
    }
    // What a pair's sums are formed from: y, r, w1, w2 (w2 in the 6th-order form).
    struct Terms {
        FxRoot t;
        double r[3], w1[3], w2[3];
    };
    template <bool kOrder6>
    static __device__ __forceinline__ void terms(const I &i, const J &jj, Acc &c, Terms &o) {
#pragma unroll
        for (int k = 0; k < 3; ++k) o.r[k] = fma_rn_f64(i.x[k], i.m1, jj.x[k]);
        FxC3 D[2] = {};  // v, a
        int top[2] = {0, 0};
        const FxP3 pj[2] = {jfx_v(jj), jfx_a(jj)}, pi[2] = {i.v, i.a};
        fx_differences<kOrder6 ? 2 : 1>(pj, pi, D, top);
        c.fv = max(c.fv, top[0]);
        if constexpr (kOrder6) c.fa = max(c.fa, top[1]);
        fx_vectors<kOrder6>(o.r, D[0], D[1], max(top[0], top[1]), i.eps_x, i.emin, i.K, o.t, o.w1, o.w2);
    }
    template <bool kOrder6>
    static __device__ __forceinline__ void pair(const I &i, const J &jj, bool self, Acc &c) {
        Terms o;
        terms<kOrder6>(i, jj, c, o);
        float yh, yl;
        fx_root_to_floats(o.t, yh, yl);
        pot_term(self ? make_float2(0.f, 0.f) : jj.mf, yh, yl, c.pf);
        const double q = fx_q(fx_y3(o.t, i.K), o.t.g, jj.mm, jfx_em(jj), jfx_sign(jj), self, i.K);
        add<kOrder6>(q, o, c);
    }
    template <bool kOrder6>
    static __device__ __forceinline__ void add(double q, const Terms &o, Acc &c) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            c.a[k] = fma(q, o.r[k], c.a[k]);
            c.j[k] = fma(q, o.w1[k], c.j[k]);
            if constexpr (kOrder6) c.s[k] = fma(q, o.w2[k], c.s[k]);
        }
    }
    static __device__ __forceinline__ void interact(const I &i, const J &jj, bool self, Acc &c) {
        pair<true>(i, jj, self, c);
    }
    // 4th-order pair term (Makino & Aarseth 1992): A0 = q r, A1 = q (v - 3 alpha r)
    static __device__ __forceinline__ void interact4(const I &i, const J &jj, bool self, Acc &c) {
        pair<false>(i, jj, self, c);
    }
    template <bool kOrder6>
    static __device__ __forceinline__ void finish(const Acc &c, double o[10]) {
        // what is not finite spreads as in doubles: a position (seen in the
        // acceleration, its differences are doubles) takes every sum, a
        // velocity jerk and snap, an acceleration the snap; the 4th-order form
        // has no snap: zero whatever the state
        const double nan = __hiloint2double(0x7ff80000, 0);
        const bool bad_x = !(isfinite(c.a[0]) && isfinite(c.a[1]) && isfinite(c.a[2]));
        const bool bad_v = bad_x || c.fv >= 0x7ff, bad_a = bad_v || c.fa >= 0x7ff;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            o[k] = bad_x ? nan : c.a[k];
            o[3 + k] = bad_v ? nan : c.j[k];
            o[6 + k] = !kOrder6 ? 0.0 : (bad_a ? nan : c.s[k]);
        }
        o[9] = bad_x ? nan : -(c.p + ((double)c.pf.hi + (double)c.pf.lo));
    }
};

// ========================================================= FP64 potential
// The potential alone (energy diagnostics), from the FP64 records: the root on
// the integer pipes as in the FP64 pair terms, four FP64 instructions a pair
// (differences and m y; 12 before).  Bound: the FP64 pipe (64 of 77 SM clocks
// per warp of pairs).  Energy of N = 65536: 32.9 ms (1.31e11 pairs/s) against
// 92.9 ms with the root and the products in doubles.
template <>
struct Prec<kPrecPot> {
    using J = J64;
    static constexpr int kPerRec = 1;
    struct I {
        double x[3], m1;
        uint64_t eps_x;
        uint32_t emin;
        FxK K;
    };
    struct Acc {
        double p;
    };
    static __device__ __forceinline__ void prepare(I &i, const Dev &d) {
        i.m1 = d.neg_one;
        i.eps_x = d.eps_x;
        i.emin = d.eps_emin;
        i.K = d.fxk;
    }
    static __device__ __forceinline__ I load_i(const J *jarr, int64_t k) {
        const J e = jarr[k];
        I r;
        r.x[0] = e.q[0].x;
        r.x[1] = e.q[0].y;
        r.x[2] = e.q[1].x;
        return r;
    }
    static __device__ __forceinline__ void zero(Acc &c) { c.p = 0.0; }
    static __device__ __forceinline__ double root(const I &i, const J &jj) {
        const double2 q0 = jj.q[0], q1 = jj.q[1];
        const double r[3] = {fma_rn_f64(i.x[0], i.m1, q0.x), fma_rn_f64(i.x[1], i.m1, q0.y),
                             fma_rn_f64(i.x[2], i.m1, q1.x)};
        const Fx3 R = fx_decode(r, i.emin);
        const FxS Rs[3] = {fx_split(R.w[0]), fx_split(R.w[1]), fx_split(R.w[2])};
        const FxRoot t = fx_root(Rs, R.e, i.eps_x, i.emin, i.K);
        return fx_root_to_double(t, R.e);
    }
    static __device__ __forceinline__ void interact_pot(const I &i, const J &jj, bool self, Acc &c) {
        c.p = fma(self ? 0.0 : jj.q[1].y, root(i, jj), c.p);
    }
    static __device__ __forceinline__ void finish(const Acc &c, double o[10]) {
#pragma unroll
        for (int k = 0; k < 9; ++k) o[k] = 0.0;
        o[9] = -c.p;
    }
};

// ======================================================================= EX
// Float-float pair terms, two j per thread and step like the FP32 path: the
// record (JEXP) gives both particles' hi and lo parts as two-lane operands
// and every float-float primitive runs on float2 lanes (ff2).  Sums and
// products are kept unnormalised wherever the next operation only folds lo
// into first-order terms (the lazy forms); the accumulators are renormalised
// once per j-tile.
template <>
struct Prec<NB_EX> {
    using J = JEXP;
    static constexpr int kPerRec = 2;
    struct I {  // the i-particle, both lanes equal
        ff2 x[3], v[3], a[3];
    };
    struct Acc {  // lane l sums the j of parity l
        ff2 a[3], j[3], s[3], p;
    };
    static __device__ __forceinline__ ff2 dup(float hi, float lo) { return ff2{f2s(hi), f2s(lo)}; }
    static __device__ __forceinline__ I load_i(const J *jarr, int64_t k) {
        const float *f = reinterpret_cast<const float *>(jarr + (k >> 1)) + (k & 1);
        I r;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            r.x[q] = dup(f[2 * q], f[2 * (4 + q)]);
            r.v[q] = dup(f[2 * (8 + q)], f[2 * (12 + q)]);
        }
        r.a[0] = dup(f[2 * 11], f[2 * 15]);
        r.a[1] = dup(f[2 * 16], f[2 * 18]);
        r.a[2] = dup(f[2 * 17], f[2 * 19]);
        return r;
    }
    static __device__ __forceinline__ void zero(Acc &c) {
        const float2 z = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 3; ++k) c.a[k] = c.j[k] = c.s[k] = ff2{z, z};
        c.p = ff2{z, z};
    }
    // relative positions and velocities, normalised (after cancellation lo
    // can exceed hi)
    static __device__ __forceinline__ void rel(const I &i, const J &jj, ff2 r[3], ff2 v[3]) {
        const float4 q0 = jj.q[0], q1 = jj.q[1], q2 = jj.q[2], q3 = jj.q[3];
        const float4 q4 = jj.q[4], q5 = jj.q[5], q6 = jj.q[6], q7 = jj.q[7];
        r[0] = ff_sub(ff2{lo2(q0), lo2(q2)}, i.x[0]);
        r[1] = ff_sub(ff2{hi2(q0), hi2(q2)}, i.x[1]);
        r[2] = ff_sub(ff2{lo2(q1), lo2(q3)}, i.x[2]);
        v[0] = ff_sub(ff2{lo2(q4), lo2(q6)}, i.v[0]);
        v[1] = ff_sub(ff2{hi2(q4), hi2(q6)}, i.v[1]);
        v[2] = ff_sub(ff2{lo2(q5), lo2(q7)}, i.v[2]);
    }
    static __device__ __forceinline__ void exclude_self(bool self0, bool self1, ff2 &r2, ff2 &m) {
        r2.hi.x = self0 ? 1.f : r2.hi.x;  // selects, not arithmetic
        r2.lo.x = self0 ? 0.f : r2.lo.x;
        m.hi.x = self0 ? 0.f : m.hi.x;
        m.lo.x = self0 ? 0.f : m.lo.x;
        r2.hi.y = self1 ? 1.f : r2.hi.y;
        r2.lo.y = self1 ? 0.f : r2.lo.y;
        m.hi.y = self1 ? 0.f : m.hi.y;
        m.lo.y = self1 ? 0.f : m.lo.y;
    }
    static __device__ __forceinline__ void interact(const I &i, const J &jj, bool self0, bool self1,
                                                    ff2 eps2, Acc &c) {
        ff2 r[3], v[3], a[3];
        rel(i, jj, r, v);
        a[0] = ff_sub(ff2{hi2(jj.q[5]), hi2(jj.q[7])}, i.a[0]);
        a[1] = ff_sub(ff2{lo2(jj.q[8]), lo2(jj.q[9])}, i.a[1]);
        a[2] = ff_sub(ff2{hi2(jj.q[8]), hi2(jj.q[9])}, i.a[2]);
        ff2 r2 = ff_dot3_add_lazy(r, r, eps2);
        ff2 m{hi2(jj.q[1]), hi2(jj.q[3])};
        exclude_self(self0, self1, r2, m);
        const ff2 y = rsqrt_ff(r2);
        const ff2 rv = ff_dot3_lazy(r, v);
        const ff2 y2 = ff_sqr_lazy(y);
        const ff2 my = ff_mul_lazy(m, y);
        const ff2 q = ff_mul_lazy(my, y2);
        const ff2 w = ff_dot3x2_lazy(v, v, r, a);
        const ff2 al = ff_mul_lazy(rv, y2);
        const ff2 ze = ff_mul_lazy(w, y2);
        const ff2 al3 = ff_mul_f_lazy(al, f2s(3.0f));
        const ff2 be3 = ff_mul_f_lazy(ff_sum_lazy(ff_sqr_lazy(al), ze), f2s(3.0f));
        const ff2 al6 = ff2{add2(al3.hi, al3.hi), add2(al3.lo, al3.lo)};  // exact
        ff_add_lazy(c.p, my);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const ff2 w1 = ff_fnma_lazy(al3, r[k], v[k]);
            const ff2 w2 = ff_fnma_lazy(be3, r[k], ff_fnma_lazy(al6, w1, a[k]));
            ff_fma_acc_lazy(c.a[k], q, r[k]);
            ff_fma_acc_lazy(c.j[k], q, w1);
            ff_fma_acc_lazy(c.s[k], q, w2);
        }
    }
    static __device__ __forceinline__ void interact4(const I &i, const J &jj, bool self0, bool self1,
                                                     ff2 eps2, Acc &c) {
        ff2 r[3], v[3];
        rel(i, jj, r, v);
        ff2 r2 = ff_dot3_add(r, r, eps2);
        ff2 m{hi2(jj.q[1]), hi2(jj.q[3])};
        exclude_self(self0, self1, r2, m);
        const ff2 y = rsqrt_ff(r2);
        const ff2 y2 = ff_sqr_lazy(y);
        const ff2 my = ff_mul_lazy(m, y);
        const ff2 q = ff_mul_lazy(my, y2);
        const ff2 al3 = ff_mul_f_lazy(ff_mul_lazy(ff_dot3(r, v), y2), f2s(3.0f));
        ff_add_lazy(c.p, my);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const ff2 w1 = ff_fnma_lazy(al3, r[k], v[k]);
            ff_fma_acc_lazy(c.a[k], q, r[k]);
            ff_fma_acc_lazy(c.j[k], q, w1);
        }
    }
    // End of a j-tile: renormalise the lazily kept sums.
    static __device__ __forceinline__ void tile_done(Acc &c) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            c.a[k] = ff_renorm(c.a[k].hi, c.a[k].lo);
            c.j[k] = ff_renorm(c.j[k].hi, c.j[k].lo);
            c.s[k] = ff_renorm(c.s[k].hi, c.s[k].lo);
        }
        c.p = ff_renorm(c.p.hi, c.p.lo);
    }
    // both lanes' float-float sums as one double (each hi + lo is exact in
    // FP64; one rounding joins the lanes)
    static __device__ __forceinline__ double to_d(ff2 a) {
        return ((double)a.hi.x + (double)a.lo.x) + ((double)a.hi.y + (double)a.lo.y);
    }
    static __device__ __forceinline__ void finish(const Acc &c, const double *, int, double o[10]) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            o[k] = to_d(c.a[k]);
            o[3 + k] = to_d(c.j[k]);
            o[6 + k] = to_d(c.s[k]);
        }
        o[9] = -to_d(c.p);
    }
};

// ===================================================================== FP32
// Two j per thread and step: the pair record (J32P) gives both particles'
// values as two-lane operands, and every add, multiply and FMA of the pair
// terms is one packed f32x2 instruction (per lane the same IEEE operations
// as the scalar form).  Lane l of every packed value belongs to particle
// 2 k + l of the tile.
template <>
struct Prec<NB_FP32> {
    using J = J32P;
    static constexpr int kPerRec = 2;  // particles per record
    struct I {  // the i-particle's values, both lanes equal
        float2 xh[3], xl[3], vh[3], vl[3], a[3];
    };
    // Two FP32 levels: per-tile sums (64 pairs, two lanes) are added into
    // chunk sums, which are promoted to FP64 every kFp32FlushTiles tiles.
    struct Acc {
        float2 a[3], j[3], s[3], p;
        float ca[3], cj[3], cs[3], cp;
    };
    static __device__ __forceinline__ I load_i(const J *jarr, int64_t k) {
        const float *f = reinterpret_cast<const float *>(jarr + (k >> 1)) + (k & 1);
        I r;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            r.xh[q] = f2s(f[2 * q]);
            r.xl[q] = f2s(f[2 * (4 + q)]);
            r.vh[q] = f2s(f[2 * (8 + q)]);
            r.vl[q] = f2s(f[2 * (12 + q)]);
            r.a[q] = f2s(f[2 * (7 + 4 * q)]);
        }
        return r;
    }
    static __device__ __forceinline__ void zero(Acc &c) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            c.a[k] = c.j[k] = c.s[k] = make_float2(0.f, 0.f);
            c.ca[k] = c.cj[k] = c.cs[k] = 0.f;
        }
        c.p = make_float2(0.f, 0.f);
        c.cp = 0.f;
    }
    // relative coordinates from the hi/lo split: (hi_j - hi_i) + (lo_j - lo_i)
    static __device__ __forceinline__ void rel(const I &i, const J &jj, float2 r[3], float2 v[3]) {
        const float4 q0 = jj.q[0], q1 = jj.q[1], q2 = jj.q[2], q3 = jj.q[3];
        const float4 q4 = jj.q[4], q5 = jj.q[5], q6 = jj.q[6], q7 = jj.q[7];
        r[0] = add2(sub2(lo2(q0), i.xh[0]), sub2(lo2(q2), i.xl[0]));
        r[1] = add2(sub2(hi2(q0), i.xh[1]), sub2(hi2(q2), i.xl[1]));
        r[2] = add2(sub2(lo2(q1), i.xh[2]), sub2(lo2(q3), i.xl[2]));
        v[0] = add2(sub2(lo2(q4), i.vh[0]), sub2(lo2(q6), i.vl[0]));
        v[1] = add2(sub2(hi2(q4), i.vh[1]), sub2(hi2(q6), i.vl[1]));
        v[2] = add2(sub2(lo2(q5), i.vh[2]), sub2(lo2(q7), i.vl[2]));
    }
    // 1/sqrt(r2) per lane: SFU value and one Newton step y (3/2 - r2 y^2 / 2)
    static __device__ __forceinline__ float2 rsqrt2(float2 r2) {
        float2 y;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(r2.x));
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(r2.y));
        const float2 t = mul2(mul2(f2s(-0.5f), r2), y);
        return mul2(y, fma2(t, y, f2s(1.5f)));
    }
    static __device__ __forceinline__ void interact(const I &i, const J &jj, bool self0, bool self1,
                                                    float2 eps2, Acc &c) {
        float2 r[3], v[3];
        rel(i, jj, r, v);
        const float2 ax = sub2(hi2(jj.q[3]), i.a[0]);
        const float2 ay = sub2(hi2(jj.q[5]), i.a[1]);
        const float2 az = sub2(hi2(jj.q[7]), i.a[2]);
        float2 r2 = fma2(r[0], r[0], fma2(r[1], r[1], fma2(r[2], r[2], eps2)));
        float2 m = hi2(jj.q[1]);
        r2.x = self0 ? 1.f : r2.x;  // selects, not arithmetic
        r2.y = self1 ? 1.f : r2.y;
        m.x = self0 ? 0.f : m.x;
        m.y = self1 ? 0.f : m.y;
        const float2 y = rsqrt2(r2);
        const float2 y2 = mul2(y, y);
        const float2 my = mul2(m, y);
        const float2 q = mul2(my, y2);
        c.p = add2(c.p, my);
        const float2 rv = fma2(r[0], v[0], fma2(r[1], v[1], mul2(r[2], v[2])));
        const float2 w = fma2(v[0], v[0], fma2(v[1], v[1], fma2(v[2], v[2],
                         fma2(r[0], ax, fma2(r[1], ay, mul2(r[2], az))))));
        const float2 al = mul2(rv, y2);
        const float2 ze = mul2(w, y2);
        const float2 nal3 = mul2(f2s(-3.f), al);              // -3 alpha
        const float2 nbe3 = mul2(f2s(-3.f), fma2(al, al, ze)); // -3 beta
        const float2 nal6 = add2(nal3, nal3);
        const float2 aa[3] = {ax, ay, az};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float2 w1 = fma2(nal3, r[k], v[k]);
            const float2 w2 = fma2(nbe3, r[k], fma2(nal6, w1, aa[k]));
            c.a[k] = fma2(q, r[k], c.a[k]);
            c.j[k] = fma2(q, w1, c.j[k]);
            c.s[k] = fma2(q, w2, c.s[k]);
        }
    }
    static __device__ __forceinline__ void interact4(const I &i, const J &jj, bool self0, bool self1,
                                                     float2 eps2, Acc &c) {
        float2 r[3], v[3];
        rel(i, jj, r, v);
        float2 r2 = fma2(r[0], r[0], fma2(r[1], r[1], fma2(r[2], r[2], eps2)));
        float2 m = hi2(jj.q[1]);
        r2.x = self0 ? 1.f : r2.x;
        r2.y = self1 ? 1.f : r2.y;
        m.x = self0 ? 0.f : m.x;
        m.y = self1 ? 0.f : m.y;
        const float2 y = rsqrt2(r2);
        const float2 y2 = mul2(y, y);
        const float2 my = mul2(m, y);
        const float2 q = mul2(my, y2);
        c.p = add2(c.p, my);
        const float2 nal3 =
            mul2(f2s(-3.f), mul2(fma2(r[0], v[0], fma2(r[1], v[1], mul2(r[2], v[2]))), y2));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float2 w1 = fma2(nal3, r[k], v[k]);
            c.a[k] = fma2(q, r[k], c.a[k]);
            c.j[k] = fma2(q, w1, c.j[k]);
        }
    }
    // End of a tile: add both lanes of the tile sums into the chunk sums.
    static __device__ __forceinline__ void tile_done(Acc &c) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            c.ca[k] += c.a[k].x + c.a[k].y;
            c.cj[k] += c.j[k].x + c.j[k].y;
            c.cs[k] += c.s[k].x + c.s[k].y;
            c.a[k] = c.j[k] = c.s[k] = make_float2(0.f, 0.f);
        }
        c.cp += c.p.x + c.p.y;
        c.p = make_float2(0.f, 0.f);
    }
    // Promote the FP32 chunk sums into the FP64 totals and restart them.
    // t64: the ten FP64 totals, element q at t64[q * st]
    static __device__ __forceinline__ void flush(Acc &c, double *t64, int st) {
        tile_done(c);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            t64[k * st] += (double)c.ca[k];
            t64[(3 + k) * st] += (double)c.cj[k];
            t64[(6 + k) * st] += (double)c.cs[k];
        }
        t64[9 * st] += (double)c.cp;
        zero(c);
    }
    static __device__ __forceinline__ void finish(Acc &c, double *t64, int st, double o[10]) {
        flush(c, t64, st);
#pragma unroll
        for (int k = 0; k < 9; ++k) o[k] = t64[k * st];
        o[9] = -t64[9 * st];
    }
};

// ==================================================================== FP32X
// The acceleration and the potential in float-float (the EX pair terms'
// arithmetic), jerk and snap in FP32 (the FP32 pair terms' arithmetic, on
// the float-float relative position and coefficients rounded to FP32): the
// 6th-order step criterion interpolates a^(3..5) from differences of the
// accelerations at both step ends over h^3..h^5 and needs the acceleration
// to about 1e-8, the jerk and snap only to about 1e-5.  Two j per thread and
// step on packed f32x2 lanes, from the EX records.
template <>
struct Prec<NB_FP32X> {
    using J = JEXP;
    static constexpr int kPerRec = 2;
    struct I {  // both lanes equal
        ff2 x[3];
        float2 vh[3], vl[3], a[3];
    };
    struct Acc {
        ff2 a[3], p;         // float-float sums, renormalised per j-tile
        float2 j[3], s[3];   // FP32 tile sums, lane l for the j of parity l
        float cj[3], cs[3];  // FP32 chunk sums, promoted to FP64 every kFp32FlushTiles tiles
    };
    static __device__ __forceinline__ I load_i(const J *jarr, int64_t k) {
        const float *f = reinterpret_cast<const float *>(jarr + (k >> 1)) + (k & 1);
        I r;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            r.x[q] = ff2{f2s(f[2 * q]), f2s(f[2 * (4 + q)])};
            r.vh[q] = f2s(f[2 * (8 + q)]);
            r.vl[q] = f2s(f[2 * (12 + q)]);
        }
        r.a[0] = f2s(f[2 * 11]);
        r.a[1] = f2s(f[2 * 16]);
        r.a[2] = f2s(f[2 * 17]);
        return r;
    }
    static __device__ __forceinline__ void zero(Acc &c) {
        const float2 z = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            c.a[k] = ff2{z, z};
            c.j[k] = c.s[k] = z;
            c.cj[k] = c.cs[k] = 0.f;
        }
        c.p = ff2{z, z};
    }
    // float-float relative positions (normalised), FP32 relative velocities
    // from the hi/lo split
    static __device__ __forceinline__ void rel(const I &i, const J &jj, ff2 r[3], float2 v[3]) {
        const float4 q0 = jj.q[0], q1 = jj.q[1], q2 = jj.q[2], q3 = jj.q[3];
        const float4 q4 = jj.q[4], q5 = jj.q[5], q6 = jj.q[6], q7 = jj.q[7];
        r[0] = ff_sub(ff2{lo2(q0), lo2(q2)}, i.x[0]);
        r[1] = ff_sub(ff2{hi2(q0), hi2(q2)}, i.x[1]);
        r[2] = ff_sub(ff2{lo2(q1), lo2(q3)}, i.x[2]);
        v[0] = add2(sub2(lo2(q4), i.vh[0]), sub2(lo2(q6), i.vl[0]));
        v[1] = add2(sub2(hi2(q4), i.vh[1]), sub2(hi2(q6), i.vl[1]));
        v[2] = add2(sub2(lo2(q5), i.vh[2]), sub2(lo2(q7), i.vl[2]));
    }
    // the float-float part: y, y^2 and q = m y^3; the sums of a and pot
    static __device__ __forceinline__ void acc_part(const ff2 r[3], ff2 r2, ff2 m, Acc &c, float2 &y2f,
                                                    float2 &qf) {
        const ff2 y = rsqrt_ff(r2);
        const ff2 y2 = ff_sqr_lazy(y);
        const ff2 my = ff_mul_lazy(m, y);
        const ff2 q = ff_mul_lazy(my, y2);
        ff_add_lazy(c.p, my);
#pragma unroll
        for (int k = 0; k < 3; ++k) ff_fma_acc_lazy(c.a[k], q, r[k]);
        y2f = y2.hi;  // the lazy pair's high part: the product rounded to FP32
        qf = q.hi;
    }
    static __device__ __forceinline__ void interact(const I &i, const J &jj, bool self0, bool self1,
                                                    ff2 eps2, Acc &c) {
        ff2 r[3];
        float2 v[3];
        rel(i, jj, r, v);
        const float2 aa[3] = {sub2(hi2(jj.q[5]), i.a[0]), sub2(lo2(jj.q[8]), i.a[1]),
                              sub2(hi2(jj.q[8]), i.a[2])};
        ff2 r2 = ff_dot3_add_lazy(r, r, eps2);
        ff2 m{hi2(jj.q[1]), hi2(jj.q[3])};
        Prec<NB_EX>::exclude_self(self0, self1, r2, m);
        float2 y2f, qf;
        acc_part(r, r2, m, c, y2f, qf);
        const float2 rf[3] = {r[0].hi, r[1].hi, r[2].hi};
        const float2 rv = fma2(rf[0], v[0], fma2(rf[1], v[1], mul2(rf[2], v[2])));
        const float2 w = fma2(v[0], v[0], fma2(v[1], v[1], fma2(v[2], v[2],
                         fma2(rf[0], aa[0], fma2(rf[1], aa[1], mul2(rf[2], aa[2]))))));
        const float2 al = mul2(rv, y2f);
        const float2 ze = mul2(w, y2f);
        const float2 nal3 = mul2(f2s(-3.f), al);
        const float2 nbe3 = mul2(f2s(-3.f), fma2(al, al, ze));
        const float2 nal6 = add2(nal3, nal3);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float2 w1 = fma2(nal3, rf[k], v[k]);
            const float2 w2 = fma2(nbe3, rf[k], fma2(nal6, w1, aa[k]));
            c.j[k] = fma2(qf, w1, c.j[k]);
            c.s[k] = fma2(qf, w2, c.s[k]);
        }
    }
    static __device__ __forceinline__ void interact4(const I &i, const J &jj, bool self0, bool self1,
                                                     ff2 eps2, Acc &c) {
        ff2 r[3];
        float2 v[3];
        rel(i, jj, r, v);
        ff2 r2 = ff_dot3_add_lazy(r, r, eps2);
        ff2 m{hi2(jj.q[1]), hi2(jj.q[3])};
        Prec<NB_EX>::exclude_self(self0, self1, r2, m);
        float2 y2f, qf;
        acc_part(r, r2, m, c, y2f, qf);
        const float2 rf[3] = {r[0].hi, r[1].hi, r[2].hi};
        const float2 nal3 =
            mul2(f2s(-3.f), mul2(fma2(rf[0], v[0], fma2(rf[1], v[1], mul2(rf[2], v[2]))), y2f));
#pragma unroll
        for (int k = 0; k < 3; ++k) c.j[k] = fma2(qf, fma2(nal3, rf[k], v[k]), c.j[k]);
    }
    // End of a j-tile: renormalise the float-float sums, add both lanes of
    // the FP32 tile sums into the chunk sums.
    static __device__ __forceinline__ void tile_done(Acc &c) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            c.a[k] = ff_renorm(c.a[k].hi, c.a[k].lo);
            c.cj[k] += c.j[k].x + c.j[k].y;
            c.cs[k] += c.s[k].x + c.s[k].y;
            c.j[k] = c.s[k] = make_float2(0.f, 0.f);
        }
        c.p = ff_renorm(c.p.hi, c.p.lo);
    }
    // Promote the FP32 chunk sums of jerk and snap into the FP64 totals
    // (t64[q * st], q = 3..8) and restart them.
    static __device__ __forceinline__ void flush(Acc &c, double *t64, int st) {
        tile_done(c);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            t64[(3 + k) * st] += (double)c.cj[k];
            t64[(6 + k) * st] += (double)c.cs[k];
            c.cj[k] = c.cs[k] = 0.f;
        }
    }
    static __device__ __forceinline__ void finish(Acc &c, double *t64, int st, double o[10]) {
        flush(c, t64, st);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            o[k] = Prec<NB_EX>::to_d(c.a[k]);
            o[3 + k] = t64[(3 + k) * st];
            o[6 + k] = t64[(6 + k) * st];
        }
        o[9] = -Prec<NB_EX>::to_d(c.p);
    }
};

// ================================================================ kernel
// Per-arithmetic launch configuration of the evaluation kernel.
template <int P>
struct EvalCfg {
    static constexpr int stages = kStages;
    static constexpr int min_blocks = NB_EVAL_MIN_BLOCKS;
    static constexpr bool t64_smem = false;
};
template <>
struct EvalCfg<NB_EX> {
    static constexpr int stages = kStages;
    static constexpr int min_blocks = NB_EX_MIN_BLOCKS;
    static constexpr bool t64_smem = false;
};
// Resident CTAs per SM the compiler must allow for one kernel.  The packed EX
// pair terms of the 4th-order modes measured faster at 3 CTAs per SM (140
// registers: 1.16e11 against 1.10e11 pairs/s at 4 CTAs, N = 65536); the
// 6th-order ones are as fast at 4 (128 registers) as at 3 (166).
template <int P, int MODE>
constexpr int eval_min_blocks() {
    if constexpr (P == NB_EX && is_order4_mode(MODE)) return NB_EX4_MIN_BLOCKS;
    if constexpr (P == kPrecPot) return 8;
    if constexpr (P == NB_FP64 && uses_order4_terms(MODE)) return 5;
    return EvalCfg<P>::min_blocks;
}
template <>
struct EvalCfg<NB_FP32> {
    static constexpr int stages = NB_FP32_STAGES;
    static constexpr int min_blocks = NB_FP32_MIN_BLOCKS;
    static constexpr bool t64_smem = NB_FP32_T64_SMEM != 0;
};
template <>
struct EvalCfg<NB_FP32X> {
    static constexpr int stages = kStages;
    static constexpr int min_blocks = NB_FP32X_MIN_BLOCKS;
    static constexpr bool t64_smem = true;
};

// Pieces from which an i-tile's sum is formed by groups, and the partial sums
// (doubles) per group counter: a group has at least six pieces of at least 40
// doubles, so groups' first slots lie in different counters' ranges.
constexpr int kTreePieces = 32;
static_assert(6 * 10 * (kTPB / 32) >= kGrpStride, "groups' first slots must not share a counter");
// ... and the pieces times i's, below which the second level of counters costs
// more than it spares (us, FP64: N = 10007, A = 16, 128 pieces of 4 i's: 26.9 ->
// 25.3; N = 16384, A = 1, 128 pieces of one: 17.6 -> 18.7).
constexpr int kTreeSums = 512;

// One piece of work, described by the first warp for the whole CTA.
struct PieceRec {
    long long tb, te;          // j-tiles of the piece
    long long local, tile0, pslot0, off, nc, ntj;
    int c, gl, split, A, tile;  // c < 0: no more work
};

// What the pieces are described from (the launch's fields, kept out of registers).
struct WorkRec {
    long long item, item_end;  // item / unit to describe next and the end of this CTA's work
    const ClusterPlan *plan;   // planned launches; NULL: direct
    const int64_t *offsets, *jofs, *order_item0;
    const int32_t *order_cluster;
    const void *jarr;
    long long n;
    int n_clusters, sk;        // sk: stream-K ranges
    int cluster, gl, split, A, jt0, jt1;  // direct launches
};

template <int P>
struct SmemLayout {
    typename Prec<P>::J tile[EvalCfg<P>::stages][kTJ / Prec<P>::kPerRec];
    double red[10 * kTPB];  // cross-split reduction: group sums, then totals
    double t64[EvalCfg<P>::t64_smem ? 10 * kTPB : 1];  // FP32 totals, [q][thread]
    uint64_t bar[EvalCfg<P>::stages];
    PieceRec pc;
    WorkRec work;
    int flag;
    int fail;
};

// Sums over the gl lanes that share an i, by recursive halving: at each step a
// lane keeps half of its values and hands the other half to its partner, so
// ten values over 32 lanes take 12 additions and 12 exchanges a lane where a
// butterfly on every value takes 50 of each (an FP64 addition is 16 SM clocks
// a warp: 12,800 against 3,000 clocks for the 16 resident warps).  Every sum is
// the butterfly's: own + partner at distances gl / 2, ..., 1.
struct LaneSums {
    int off, lim, n;  // the lane holds the sums off .. min(off + n, lim) - 1
    // element q of the lane's i goes to dst[q * st]
    __device__ __forceinline__ void store(const double o[10], double *dst, int st) const {
#pragma unroll
        for (int k = 0; k < 10; ++k)
            if (k < n && off + k < lim) dst[(off + k) * st] = o[k];
    }
};
template <int N>
__device__ __forceinline__ void halve_lanes(double *o, LaneSums &s, int w, int jsub) {
    constexpr int H = (N + 1) / 2;  // the lower lane keeps H values, the upper N - H
    const bool up = (jsub & w) != 0;
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const double hi = H + k < N ? o[H + k] : 0.0;
        const double keep = N == 1 ? o[0] : (up ? hi : o[k]), give = N == 1 ? o[0] : (up ? o[k] : hi);
        o[k] = keep + __shfl_xor_sync(0xffffffffu, give, w);
    }
    s.n = H;
    if (N == 1) s.lim = up ? s.off : s.lim;  // both hold it: one writes
    else if (up) s.off += H;
    else s.lim = min(s.lim, s.off + H);
}
// Not inlined: inlined, it changed the register allocation of the pair loops
// (FP32 2 % slower).
static __device__ __noinline__ LaneSums reduce_lanes(double *o, int gl, int jsub) {
    LaneSums s{0, 10, 10};
    if (gl >= 2) halve_lanes<10>(o, s, gl >> 1, jsub);
    if (gl >= 4) halve_lanes<5>(o, s, gl >> 2, jsub);
    if (gl >= 8) halve_lanes<3>(o, s, gl >> 3, jsub);
    if (gl >= 16) halve_lanes<2>(o, s, gl >> 4, jsub);
    if (gl >= 32) halve_lanes<1>(o, s, gl >> 5, jsub);
    return s;
}

// Largest k with item0[k] <= item, by a full warp: 32 probes a round, so
// that up to 1024 clusters take two loads in a row where a bisection takes ten.
__device__ __forceinline__ int find_cluster(const int64_t *item0, int nc, int64_t item) {
    const int lane = threadIdx.x & 31;
    int lo = 0;
    while (nc > 1) {  // the answer lies in [lo, lo + nc)
        const int step = (nc + 31) / 32;
        const int k = lane * step;
        const unsigned le = __ballot_sync(0xffffffffu, k < nc && item0[lo + min(k, nc - 1)] <= item);
        const int hit = (__popc(le) - 1) * step;
        lo += hit;
        nc = min(step, nc - hit);
    }
    return lo;
}

template <int P, int MODE>
__device__ __forceinline__ void finalize_one(const Dev &d, const EvalLaunch &L, int c, int64_t gi,
                                             int iloc, const double o[10]) {
    if constexpr (MODE == kModeOut || MODE == kModeOut4) {
        for (int q = 0; q < 10; ++q) L.out[(int64_t)q * L.n_active + iloc] = o[q];
    } else if constexpr (MODE == kModeInit1 || MODE == kModeInit2 || MODE == kModeInit4) {
        const int64_t n = d.n;
        for (int k = 0; k < 3; ++k) {
            d.a[k * n + gi] = o[k];
            d.j[k * n + gi] = o[3 + k];
            d.s[k * n + gi] = (MODE == kModeInit2) ? o[6 + k] : 0.0;
        }
        d.pot[gi] = o[9];
        // the 4th-order start-up has no snap: dt0 = eta_init |a| / |j|
        if constexpr (MODE != kModeInit1) d.dt[gi] = dt_start(d, o);
    } else {  // kModePot
        d.pot_tmp[gi] = o[9];
    }
}

// One j-tile's pairs of this thread: every gl-th record from jsub on.  js: the
// i's own place in the tile (outside [0, kTJ): not in it), read only with
// kSelf.
template <int P, int MODE, bool kSelf>
__device__ __forceinline__ void tile_pairs(const Dev &d, const typename Prec<P>::I &me,
                                           const typename Prec<P>::J *tl, int js, int jsub, int gl,
                                           typename Prec<P>::Acc &acc) {
    using T = Prec<P>;
    constexpr int kRecs = kTJ / T::kPerRec;  // records per j-tile
    constexpr int kUnroll = P == NB_FP32 ? kEvalUnroll : 1;
#pragma unroll kUnroll
    for (int k = jsub; k < kRecs; k += gl) {
        if constexpr (T::kPerRec == 1) {
            const bool self = kSelf && k == js;
            if constexpr (MODE == kModePot) T::interact_pot(me, tl[k], self, acc);
            else if constexpr (uses_order4_terms(MODE)) T::interact4(me, tl[k], self, acc);
            else T::interact(me, tl[k], self, acc);
        } else {
            // record k holds particles 2k and 2k + 1 of the tile
            const bool s0 = kSelf && 2 * k == js, s1 = kSelf && 2 * k + 1 == js;
            if constexpr (P == NB_FP32) {
                if constexpr (uses_order4_terms(MODE)) T::interact4(me, tl[k], s0, s1, d.eps2_hi2, acc);
                else T::interact(me, tl[k], s0, s1, d.eps2_hi2, acc);
            } else {
                const ff2 eps2{d.eps2_hi2, d.eps2_lo2};
                if constexpr (uses_order4_terms(MODE)) T::interact4(me, tl[k], s0, s1, eps2, acc);
                else T::interact(me, tl[k], s0, s1, eps2, acc);
            }
        }
    }
}

// Units of a stream-K launch (one cluster): i-tiles x j-tiles (of the
// launch's j-range).
__device__ __forceinline__ int64_t sk_units(const Dev &d, const EvalLaunch &L) {
    const int c = L.direct ? L.cluster : 0;
    const int64_t tiles = L.direct ? L.tiles : d.plan[0].tiles;
    const int64_t ntj = cdiv(d.n_clusters == 1 ? d.n : d.offsets[c + 1] - d.offsets[c], kTJ);
    return tiles * (L.direct ? (L.jt1 > 0 ? (int64_t)L.jt1 : ntj) - L.jt0 : ntj);
}

// The first warp: describes the piece at work.item (or the end of the work), and thread 0 starts the copies of its first j-tiles; the CTA reads the
// record after its next barrier.  Out of line: inlined, it cost the pair loop 4-8 registers.
template <int P>
__device__ __noinline__ void describe(SmemLayout<P> &S) {
    constexpr int kSt = EvalCfg<P>::stages;
    using J = typename Prec<P>::J;
    constexpr int kRecs = kTJ / Prec<P>::kPerRec;
    WorkRec &W = S.work;
    PieceRec &N = S.pc;
    __syncwarp();
    const int64_t item = W.item, item_end = W.item_end;
    const bool one = W.n_clusters == 1;
    int c = 0;
    if (item < item_end && W.plan && !one) c = W.order_cluster[find_cluster(W.order_item0, W.n_clusters, item)];
    if (threadIdx.x != 0) return;
    if (item >= item_end) {
        N.c = -1;
        return;
    }
    int gl, split, A;
    int64_t item0 = 0, tile0 = 0, pslot0 = 0;
    if (W.plan) {
        const ClusterPlan pl = W.plan[c];
        gl = pl.gl; split = pl.split; A = pl.active; item0 = pl.item0; tile0 = pl.tile0;
        pslot0 = pl.pslot0;
    } else {
        c = W.cluster; gl = W.gl; split = W.split; A = W.A;
    }
    const int64_t off = one ? 0 : W.offsets[c];
    const int64_t nc = one ? W.n : W.offsets[c + 1] - off;
    const int64_t jofs = one ? 0 : W.jofs[c];
    // the j-tiles this launch covers: all of the cluster's, or a host-given
    // range [jt0, jt0 + ntj) of them (direct launches)
    const int64_t jt0 = W.plan ? 0 : W.jt0;
    const int64_t ntj = (!W.plan && W.jt1 > 0 ? (int64_t)W.jt1 : cdiv(nc, kTJ)) - jt0;
    int tile;
    int64_t tb, te, local = 0;
    if (W.sk) {
        tile = (int)(item / ntj);
        tb = item - (int64_t)tile * ntj;
        te = min(ntj, tb + (item_end - item));
        W.item = item + (te - tb);
    } else {
        local = item - item0;
        tile = (int)(local / split);
        const int sidx = (int)(local % split);
        tb = ntj * sidx / split;
        te = ntj * (sidx + 1) / split;
    }
    tb += jt0;
    te += jt0;
    const J *jc = reinterpret_cast<const J *>(W.jarr) + jofs / Prec<P>::kPerRec;
    for (int s = 0; s < kSt && tb + s < te; ++s) {
        mbar_expect_tx(&S.bar[s], kRecs * sizeof(J));
        tma_load_1d(&S.tile[s][0], jc + (tb + s) * kRecs, kRecs * sizeof(J), &S.bar[s]);
    }
    N.c = c; N.gl = gl; N.split = split; N.A = A; N.tile = tile;
    N.tile0 = tile0; N.pslot0 = pslot0; N.local = local;
    N.off = off; N.nc = nc; N.ntj = ntj; N.tb = tb; N.te = te;
}

template <int P, int MODE>
__global__ void __launch_bounds__(kTPB, (eval_min_blocks<P, MODE>())) k_eval(const Dev d, const EvalLaunch L) {
    using T = Prec<P>;
    constexpr int kSt = EvalCfg<P>::stages;
    using J = typename T::J;
    constexpr int kRecs = kTJ / T::kPerRec;  // records per j-tile
    extern __shared__ __align__(128) unsigned char smem_raw[];
    SmemLayout<P> &S = *reinterpret_cast<SmemLayout<P> *>(smem_raw);
    const int tid = threadIdx.x;
    if (L.gate && *L.gate == 0) return;  // done by the form that takes each pair once

    // Work: a stream-K launch (one cluster) gives CTA k the unit range
    // [U k / G, U (k+1) / G) and walks it piece by piece (one piece per i-tile
    // it touches).  Otherwise work items (cluster, i-tile, split index):
    // direct launches (equal-cost items of one cluster) take a static round
    // robin; planned launches take item blockIdx.x first and the others
    // dynamically, since clusters of a batch give items of unequal cost.
    // Either way a piece's arithmetic and the reduction order do not depend on
    // the CTA that runs it.  The pieces' bookkeeping stays in shared memory, so
    // that the pair loop holds only what it uses in registers.
    if (tid == 0) {
        for (int s = 0; s < kSt; ++s) mbar_init(&S.bar[s], 1);
        S.fail = 0;
        fence_mbar_init();
        WorkRec &W = S.work;
        W.plan = L.direct ? nullptr : d.plan;
        W.offsets = d.offsets; W.jofs = d.jofs; W.jarr = d.jarr;
        W.order_item0 = d.order_item0; W.order_cluster = d.order_cluster;
        W.n = d.n; W.n_clusters = d.n_clusters;
        W.cluster = L.cluster; W.gl = L.gl; W.split = L.split; W.A = L.n_active;
        W.jt0 = L.jt0; W.jt1 = L.jt1;
        W.sk = L.direct ? L.streamk != 0 : (d.n_clusters == 1 && d.plan[0].streamk != 0);
        if (W.sk) {
            const int64_t U = sk_units(d, L);
            W.item = sk_begin(U, gridDim.x, blockIdx.x);
            W.item_end = sk_begin(U, gridDim.x, blockIdx.x + 1);
        } else {
            W.item = blockIdx.x;
            W.item_end = L.direct ? (int64_t)L.tiles * L.split : *d.n_items;
        }
    }
    uint32_t phase = 0;  // bit s: parity of stage s
    if (tid < 32) describe<P>(S);

    const PieceRec &R = S.pc;
    for (;;) {
        // every thread is done with the last piece; this one's record is there
        __syncthreads();
        if (R.c < 0) break;

        const int gl = R.gl;
        const int64_t tb = R.tb, te = R.te;
        const int ilane = tid / gl;
        const int jsub = tid % gl;
        const J *jc = reinterpret_cast<const J *>(d.jarr) + (d.n_clusters == 1 ? 0 : d.jofs[R.c] / T::kPerRec);
        // this thread's i: global index, bounds-checked against its cluster
        auto i_of = [&](int64_t off, int64_t nc, int il, bool &bad) -> int64_t {
            int64_t g;
            if (L.identity) g = off + il;
            else if (L.direct) g = L.active[il];
            else g = d.active[off + il];
            bad = g < off || g >= off + nc;
            return bad ? off : g;
        };
        const int il0 = R.tile * (kTPB / gl) + ilane;
        int64_t ji = 0;
        if (il0 < R.A) {
            bool bad;
            ji = i_of(R.off, R.nc, il0, bad) - R.off;
            if (bad) atomicOr(d.err, kErrIndex);  // caller-given index outside the cluster
        }
        typename T::I me = T::load_i(jc, ji);
        if constexpr (P == NB_FP64 || P == kPrecPot) T::prepare(me, d);
        typename T::Acc acc;
        T::zero(acc);
        double t64r[EvalCfg<P>::t64_smem ? 1 : 10];
        double *t64 = EvalCfg<P>::t64_smem ? S.t64 + tid : t64r;
        constexpr int t64st = EvalCfg<P>::t64_smem ? kTPB : 1;
#pragma unroll
        for (int q = 0; q < 10; ++q) t64[q * t64st] = 0.0;
        const bool warp_active = __any_sync(0xffffffffu, il0 < R.A);

        bool ok = true;
        // FP64 and FP32 count the piece's tiles in 32 bits from its first, EX
        // and FP32X by their index in the cluster: the same work, but the loop's
        // registers differ (all active, N = 65536: FP64 4th order 21.0 -> 20.0
        // ms, FP32 4th order 5.75 -> 5.71 ms, the other way round EX 1 % and
        // FP32X 1 % slower)
        constexpr bool kRel = P == NB_FP64 || P == NB_FP32 || P == kPrecPot;
        using Tix = std::conditional_t<kRel, int, int64_t>;
        const Tix t0 = kRel ? 0 : (Tix)tb, t1 = kRel ? (Tix)(te - tb) : (Tix)te;
        int jrel = (int)(ji - tb * kTJ);  // the thread's i as a j of the current tile
        for (Tix t = t0; t < t1; ++t) {
            const int s = (int)((t - t0) % kSt);
            if (ok) ok = mbar_wait_bounded(&S.bar[s], (phase >> s) & 1u);
            phase ^= 1u << s;
            if (ok && warp_active) {
                const J *tl = &S.tile[s][0];
                // the pairs i = j of a warp lie in a few tiles: the others run a
                // loop without the exclusion's compares and selects (FP32X 5 %,
                // FP32 3-5 %, EX 1.5-2.5 % faster, the same results)
                int js;
                if constexpr (kRel) js = min(max(jrel, -1), kTJ);
                else js = (int)min(max(ji - t * kTJ, (int64_t)-1), (int64_t)kTJ);
                if (__any_sync(0xffffffffu, (unsigned)js < (unsigned)kTJ))
                    tile_pairs<P, MODE, true>(d, me, tl, js, jsub, gl, acc);
                else
                    tile_pairs<P, MODE, false>(d, me, tl, js, jsub, gl, acc);
                if constexpr (P == NB_FP32 || P == NB_FP32X) {
                    if ((t - t0 + 1) % kFp32FlushTiles == 0) T::flush(acc, t64, t64st);
                    else T::tile_done(acc);
                } else if constexpr (P == NB_EX) {
                    T::tile_done(acc);
                } else if constexpr (P == NB_FP64) {
                    // every 64 pairs of the lane (four FP64 operations)
                    if (((int)(t - t0 + 1) & (gl - 1)) == 0) T::tile_done(acc);
                }
            }
            jrel -= kTJ;
            if (!ok) S.fail = 1 + (int)(t - t0);
            __syncthreads();
            if (S.fail) break;
            if (tid == 0 && t + kSt < t1) {
                mbar_expect_tx(&S.bar[s], kRecs * sizeof(J));
                tma_load_1d(&S.tile[s][0], jc + ((kRel ? tb : 0) + t + kSt) * kRecs, kRecs * sizeof(J), &S.bar[s]);
            }
        }
        if (S.fail) {
            // a copy did not land in time: record it, drain (bounded) what this
            // CTA still has in flight (from the failing tile on; the parity of
            // its stage is one ahead already), and leave the kernel
            if (tid == 0) {
                atomicOr(d.err, kErrTimeout);
                const int k0 = S.fail - 1, nt = (int)(te - tb);
                phase ^= 1u << (k0 % kSt);
                for (int k = k0; k < nt && k < k0 + kSt; ++k)
                    (void)mbar_wait_bounded(&S.bar[k % kSt], (phase >> (k % kSt)) & 1u);
            }
            return;
        }

        // ---- epilogue: the piece's bookkeeping comes back from shared memory;
        // past the barrier below the record describes the next piece.  The
        // next item is fetched ahead of the sums and its first j-tiles are
        // under way while this piece's sums are joined.
        long long next = 0;
        if (tid == 0 && !S.work.sk)
            next = gridDim.x + (L.direct ? S.work.item : (long long)atomicAdd(d.item_ctr, 1ull));
        const int c = R.c, tile = R.tile, A = R.A, split = R.split;
        const int Ti = kTPB / R.gl;
        const int64_t off = R.off, nc = R.nc, ntj = R.ntj, tile0 = R.tile0;
        const bool sk = S.work.sk;
        // pieces of this i-tile: split items, or the CTAs whose ranges meet it
        int npieces = split;
        int64_t sk_first = 0, sk_maxp = 0, sk_loc0 = 0;
        if (sk) {
            const int64_t U = sk_units(d, L);
            sk_first = sk_owner(U, gridDim.x, (int64_t)tile * ntj);
            npieces = (int)(sk_owner(U, gridDim.x, (int64_t)(tile + 1) * ntj - 1) - sk_first + 1);
            sk_maxp = sk_max_pieces(U, gridDim.x, ntj);
            // the first piece's CTA may have started in an earlier i-tile; the
            // others start inside this one (their local tile index is 0)
            sk_loc0 = tile - sk_begin(U, gridDim.x, sk_first) / ntj;
        }
        const int64_t pslot0 = R.pslot0;
        // partial-sum slot (doubles) of piece s of this tile: CTA k keeps one
        // slot per i-tile its range touches
        auto piece_slot = [&](int64_t s) -> int64_t {
            if (sk) return ((sk_first + s) * sk_maxp + (s == 0 ? sk_loc0 : 0)) * (10 * Ti);
            return pslot0 + ((int64_t)tile * split + s) * (10 * Ti);
        };
        double o[10];
        if constexpr (P == NB_FP64) T::template finish<!uses_order4_terms(MODE)>(acc, o);
        else if constexpr (P == kPrecPot) T::finish(acc, o);
        else T::finish(acc, t64, t64st, o);
        // the sums of the lanes sharing an i; after this, the lane holds those
        // of q in [held.off, held.lim) in o[0 ..]
        const LaneSums held = reduce_lanes(o, R.gl, tid & (R.gl - 1));
        const int slot = tid / R.gl;
        // this CTA's piece of the tile, and its group when the groups' sums are
        // formed by their own last CTAs
        const int piece = sk ? (int)((int64_t)blockIdx.x - sk_first) : (int)(R.local - (int64_t)tile * split);
        const int Rg = min((npieces + 7) / 8, kTPB / Ti);
        const int nv = min(Ti, A - tile * Ti);  // valid i in this tile
        constexpr bool kStep = MODE == kModeStep || MODE == kModeStep4;
        auto particle = [&](int il) -> int64_t {
            bool bad;
            const int64_t gi = i_of(off, nc, tile * Ti + il, bad);
            return bad ? -1 : gi;
        };
        const bool tree = npieces >= kTreePieces && npieces * nv >= kTreeSums;
        const int grp = tree ? ((piece + 1) * Rg - 1) / npieces : 0;
        const int g0 = npieces * grp / Rg, g1 = npieces * (grp + 1) / Rg;
        if (npieces > 1) {
            held.store(o, d.partial + piece_slot(piece) + slot, Ti);
            __threadfence();
        } else if (Ti < kTPB || kStep) {
            held.store(o, S.red + slot, Ti);
        }
        __syncthreads();
        if (tid < 32) {
            int prev = 0;
            if (tid == 0) {
                if (tree) prev = atomicAdd(&d.grp_cnt[piece_slot(g0) / kGrpStride], 1);
                else if (npieces > 1) prev = atomicAdd(&d.tile_cnt[tile0 + tile], 1);
                if (!sk) S.work.item = next;
            }
            describe<P>(S);
            if (tid == 0) S.flag = (prev == (tree ? g1 - g0 : npieces) - 1);
        }
        if (npieces == 1 && kStep) {
            correct_tile<MODE == kModeStep4>(d, nv, d.tnext[c], S.red, Ti, particle);
        } else if (npieces == 1) {
            // one thread per i (gathering its ten sums if lanes shared it)
            const int il = tile * Ti + tid;
            if (tid < Ti && il < A) {
                if (Ti < kTPB) {
#pragma unroll
                    for (int q = 0; q < 10; ++q) o[q] = S.red[q * Ti + tid];
                }
                bool bad;
                const int64_t gi = i_of(off, nc, il, bad);
                if (!bad) finalize_one<P, MODE>(d, L, c, gi, il, o);
            }
        } else {
            // The last CTA of this i-tile adds the pieces for every (i, q) pair
            // in two fixed-order levels: contiguous groups of pieces, each in
            // piece order, then the group sums in group order.  The order
            // depends only on the pieces and the tile's width, so results are
            // reproducible and the same for every i.  Groups of eight pieces
            // (more when S.red would overflow): a chain of hundreds of loads and
            // additions in a handful of threads took longer than the pairs
            // themselves.  From kTreePieces pieces on, the last CTA of each group
            // forms its sum (in the place of the group's first piece): one CTA
            // adding 76 pieces of 16 i's took 38 us at the end of a launch of
            // 316 (N = 65536, A = 128), its SM alone at work.
            const int npair = nv * 10;
            // pieces at a fixed stride (the first of a stream-K tile sits elsewhere)
            const int64_t stride = (sk ? sk_maxp : (int64_t)1) * (10 * Ti);
            double *first = d.partial + piece_slot(0);
            double *rest = first - (sk ? sk_loc0 : (int64_t)0) * (10 * Ti);
            auto at = [&](int s) { return s == 0 ? first : rest + s * stride; };
            // the sum of pieces s0 .. s1 - 1 at an offset, eight loads in flight
            auto sum_pieces = [&](int s0, int s1, int col) {
                double sum = 0.0;
                for (int sp = s0; sp < s1; sp += 8) {
                    double t[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) t[u] = sp + u < s1 ? __ldcg(at(sp + u) + col) : 0.0;
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (sp + u < s1) sum += t[u];
                }
                return sum;
            };
            __syncthreads();
            if (tree && S.flag) {
                __threadfence();
                for (int p = tid; p < npair; p += kTPB) {
                    const int col = p / nv * Ti + p % nv;
                    at(g0)[col] = sum_pieces(g0, g1, col);
                }
                __threadfence();
                __syncthreads();
                if (tid == 0) {
                    d.grp_cnt[piece_slot(g0) / kGrpStride] = 0;
                    S.flag = atomicAdd(&d.tile_cnt[tile0 + tile], 1) == Rg - 1;
                }
                __syncthreads();
            }
            if (S.flag) {
                __threadfence();
                for (int w = tid; w < npair * Rg; w += kTPB) {
                    const int p = w % npair, r = w / npair;
                    const int col = p / nv * Ti + p % nv;
                    const int s0 = npieces * r / Rg, s1 = npieces * (r + 1) / Rg;
                    S.red[r * npair + p] = tree ? __ldcg(at(s0) + col) : sum_pieces(s0, s1, col);
                }
                __syncthreads();
                for (int p = tid; p < npair; p += kTPB) {
                    double a2 = S.red[p];
                    for (int r = 1; r < Rg; ++r) a2 += S.red[r * npair + p];
                    S.red[p] = a2;
                }
                __syncthreads();
                if constexpr (kStep) {
                    correct_tile<MODE == kModeStep4>(d, nv, d.tnext[c], S.red, nv, particle);
                } else if (tid < nv) {
                    double sum[10];
#pragma unroll
                    for (int q = 0; q < 10; ++q) sum[q] = S.red[q * nv + tid];
                    const int il = tile * Ti + tid;
                    bool bad;
                    const int64_t g2 = i_of(off, nc, il, bad);
                    if (!bad) finalize_one<P, MODE>(d, L, c, g2, il, sum);
                }
                if (tid == 0) d.tile_cnt[tile0 + tile] = 0;
            }
        }
    }
}

template <int P, int MODE>
cudaError_t launch_eval_t(const Dev &d, const EvalLaunch &L, int grid, cudaStream_t st) {
    const size_t smem = sizeof(SmemLayout<P>);  // < 48 KB: no opt-in attribute needed
    static_assert(sizeof(SmemLayout<P>) <= 48 * 1024, "evaluation tile ring exceeds 48 KB");
    k_eval<P, MODE><<<grid, kTPB, smem, st>>>(d, L);
    return cudaGetLastError();
}

template <int P, int MODE>
int occupancy_t() {
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_eval<P, MODE>, kTPB, sizeof(SmemLayout<P>));
    return b;
}

}  // namespace nb
