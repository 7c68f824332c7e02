// nb_step.cuh -- per-particle FP64 device functions of the integrator:
// predictor, corrector + quintic derivatives + time step, start-up step,
// and the 4th-order Hermite corrector + cubic derivatives + Aarseth step.
//
// Method: the paper's Sec. 2 integrator (Hermite 6th order, block time
// steps, inherited from HiGPUs); formulas after Nitadori & Makino 2008,
// power-of-two steps after Makino 1991 / Aarseth 2003.
#pragma once

#include "nb_internal.cuh"

namespace nb {

// Largest power of two <= x for normal positive x (exponent bits only).
__device__ __forceinline__ double pow2_floor_dev(double x) {
    return __hiloint2double(__double2hiint(x) & 0x7ff00000, 0);
}

__device__ __forceinline__ double norm3_dev(double a, double b, double c) {
    return sqrt(fma(a, a, fma(b, b, c * c)));
}

// Start-up step: eta_init * min(|a|/|j|, sqrt(|a|/|s|)), quantised down to a
// power of two and clamped; a vanishing denominator imposes no limit.
__device__ __forceinline__ double dt_start(const Dev &d, const double o[10]) {
    const double an = norm3_dev(o[0], o[1], o[2]);
    const double jn = norm3_dev(o[3], o[4], o[5]);
    const double sn = norm3_dev(o[6], o[7], o[8]);
    double r = INFINITY;
    if (jn > 0.0) r = an / jn;
    if (sn > 0.0) r = fmin(r, sqrt(an / sn));
    const double dt0 = d.eta_init * r;
    double dt;
    if (!(dt0 > 0.0)) dt = d.dt_min;          // zero or NaN
    else if (isinf(dt0)) dt = d.dt_max;
    else dt = fmin(fmax(pow2_floor_dev(dt0), d.dt_min), d.dt_max);
    return dt;
}

// Power-of-two block step from the criterion's dt: shrink to the largest
// power of two below it, double once when it allows twice the old step and
// t1 is a multiple of that, clamp to [dt_min, dt_max]; a criterion below
// dt_min (or NaN) is counted as an underflow.
__device__ __forceinline__ double block_step_quantize(const Dev &d, double dtc, double dt_old,
                                                      double tn) {
    double dtn = dt_old;
    if (!(dtc >= d.dt_min)) {               // below the floor, or NaN
        dtn = d.dt_min;
        atomicAdd(d.ctr_underflow, 1ull);
    } else if (dtc < dt_old) {
        dtn = pow2_floor_dev(dtc);
    } else if (dtc >= 2.0 * dt_old) {
        const double q = tn * (0.5 / dt_old);  // exact: power-of-two scaling
        if (q == trunc(q)) dtn = 2.0 * dt_old;
    }
    return fmin(fmax(dtn, d.dt_min), d.dt_max);
}

// Predict particle i (global index) to time tn, in Horner form with the
// divided steps h, h/2, h/3, ...:  x_p = x + h (v + h/2 (a + h/3 (j + ...))),
// one FMA a term (42 FP64 operations a particle, which bound the predictor;
// the power form took 57).  The 4th-order scheme predicts through jerk only
// (its s and c hold the interpolated derivatives used by the time-step
// criterion).
__device__ __forceinline__ void predict_particle(const Dev &d, int64_t i, double tn,
                                                 double xp[3], double vp[3], double ap[3]) {
    const int64_t n = d.n;
    const bool through_crackle = d.order != 4;
    const double h = tn - d.t[i];
    const double h2 = h * 0.5, h3 = h * (1.0 / 3.0), h4 = h * 0.25, h5 = h * 0.2;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double x = d.x[k * n + i], v = d.v[k * n + i], a = d.a[k * n + i];
        const double jj = d.j[k * n + i];
        if (through_crackle) {
            const double s = d.s[k * n + i], c = d.c[k * n + i];
            xp[k] = fma(h, fma(h2, fma(h3, fma(h4, fma(h5, c, s), jj), a), v), x);
            vp[k] = fma(h, fma(h2, fma(h3, fma(h4, c, s), jj), a), v);
            ap[k] = fma(h, fma(h2, fma(h3, c, s), jj), a);
        } else {
            xp[k] = fma(h, fma(h2, fma(h3, jj, a), v), x);
            vp[k] = fma(h, fma(h2, jj, a), v);
            ap[k] = fma(h, jj, a);
        }
    }
}

// Powers of a step h > 0.  A power of two, as every block step is, has its
// inverse and h^3 / 120 without divisions (both exact scalings, so the same
// doubles); a division is about ten FP64 operations.
struct StepH {
    double h, hh, hhh120, inv;
};
__device__ __forceinline__ StepH step_powers(double h) {
    const double hh = h * h, hhh = hh * h;
    const int hi = __double2hiint(h);
    const int e = hi >> 20;
    if (((hi & 0xfffff) | __double2loint(h)) == 0 && e > 723 && e < 1323)
        return StepH{h, hh, hhh * (1.0 / 120.0), __hiloint2double((2046 - e) << 20, 0)};
    return StepH{h, hh, hhh / 120.0, 1.0 / h};
}

// Corrector and interpolated derivatives of one coordinate (formulas below).
struct Axis6 {
    double x1, v1, d3, d4, d5;
};
__device__ __forceinline__ Axis6 correct_axis6(const StepH &H, double x0, double v0, double a0, double j0,
                                               double s0, double a1, double j1, double s1) {
    const double h = H.h, hh = H.hh, hinv = H.inv;
    const double hinv2 = hinv * hinv;
    const double hinv3 = hinv2 * hinv;
    const double hinv5 = hinv3 * hinv2;
    Axis6 r;
    r.v1 = v0 + (0.5 * h * (a1 + a0) - 0.1 * hh * (j1 - j0) + H.hhh120 * (s1 + s0));
    r.x1 = x0 + (0.5 * h * (r.v1 + v0) - 0.1 * hh * (a1 - a0) + H.hhh120 * (j1 + j0));
    const double D = a1 - a0, Jp = j1 + j0, Jm = j1 - j0, Sp = s1 + s0, Sm = s1 - s0;
    const double c5 = (6.0 * D - 3.0 * h * Jp + 0.5 * hh * Sm) * hinv5;
    const double c4 = (0.25 * h * Sp - 0.5 * Jm) * hinv3;
    r.d5 = 120.0 * c5;
    r.d4 = 24.0 * c4 + 60.0 * h * c5;
    r.d3 = Sm * hinv + 12.0 * h * c4 + 10.0 * hh * c5;
    return r;
}
struct Axis4 {
    double x1, v1, a2, a3;
};
__device__ __forceinline__ Axis4 correct_axis4(double h, double hinv, double x0, double v0, double a0, double j0,
                                               double a1, double j1) {
    const double hinv2 = hinv * hinv;
    const double hh12 = h * h * (1.0 / 12.0);
    Axis4 r;
    r.v1 = v0 + (0.5 * h * (a0 + a1) + hh12 * (j0 - j1));
    r.x1 = x0 + (0.5 * h * (v0 + r.v1) + hh12 * (a0 - a1));
    const double D = a0 - a1;
    r.a2 = (6.0 * D + 2.0 * h * (j0 + 2.0 * j1)) * hinv2;
    r.a3 = (12.0 * D + 6.0 * h * (j0 + j1)) * (hinv2 * hinv);
    return r;
}

// The criteria's dt from the vectors (formulas below).
__device__ __forceinline__ double criterion6(const Dev &d, const double a[3], const double j[3], const double s[3],
                                             const double d3[3], const double d4[3], const double d5[3]) {
    const double an = norm3_dev(a[0], a[1], a[2]);
    const double jn = norm3_dev(j[0], j[1], j[2]);
    const double sn = norm3_dev(s[0], s[1], s[2]);
    const double A1 = sqrt(an * sn) + jn;
    const double A4 = sqrt(norm3_dev(d3[0], d3[1], d3[2]) * norm3_dev(d5[0], d5[1], d5[2])) +
                      norm3_dev(d4[0], d4[1], d4[2]);
    return (A4 > 0.0) ? d.eta * cbrt(A1 / A4) : INFINITY;
}
__device__ __forceinline__ double criterion4(const Dev &d, const double a[3], const double j[3],
                                             const double a2[3], const double a3[3]) {
    const double an = norm3_dev(a[0], a[1], a[2]);
    const double jn = norm3_dev(j[0], j[1], j[2]);
    const double sn = norm3_dev(a2[0], a2[1], a2[2]);
    const double cn = norm3_dev(a3[0], a3[1], a3[2]);
    const double den = fma(jn, cn, sn * sn);
    return (den > 0.0) ? sqrt(d.eta * fma(an, sn, jn * jn) / den) : INFINITY;
}

// Corrector, interpolated derivatives, new power-of-two step; writes the
// state of particle i.  o = {a1[3], j1[3], s1[3], pot} evaluated at tn on the
// predicted state.
//
//   v1 = v0 + h/2 (a1 + a0) - h^2/10 (j1 - j0) + h^3/120 (s1 + s0)
//   x1 = x0 + h/2 (v1 + v0) - h^2/10 (a1 - a0) + h^3/120 (j1 + j0)
// The quintic through (a, j, s) at both ends has, at t1, with
// D = a1 - a0, Jp/Jm = j1 +/- j0, Sp/Sm = s1 +/- s0:
//   c5 = (6 D - 3 h Jp + h^2 Sm / 2) / h^5      (so a^(5) = 120 c5)
//   c4 = (h Sp / 4 - Jm / 2) / h^3
//   a^(5) = 120 c5,  a^(4) = 24 c4 + 60 h c5,  a^(3) = Sm/h + 12 h c4 + 10 h^2 c5
// New step: eta (A1/A4)^{1/3}, A1 = sqrt(|a||s|) + |j|, A4 = sqrt(|a3||a5|) + |a4|.
__device__ __forceinline__ void correct_particle(const Dev &d, int64_t i, double tn,
                                                 const double o[10]) {
    const int64_t n = d.n;
    const StepH H = step_powers(tn - d.t[i]);
    double x1[3], v1[3], d3[3], d4[3], d5[3];
    bool finite = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const Axis6 r = correct_axis6(H, d.x[k * n + i], d.v[k * n + i], d.a[k * n + i], d.j[k * n + i],
                                      d.s[k * n + i], o[k], o[3 + k], o[6 + k]);
        x1[k] = r.x1; v1[k] = r.v1; d3[k] = r.d3; d4[k] = r.d4; d5[k] = r.d5;
        finite = finite && isfinite(r.x1) && isfinite(r.v1) && isfinite(o[k]) && isfinite(o[3 + k]) &&
                 isfinite(o[6 + k]) && isfinite(r.d3);
    }
    const double dtc = criterion6(d, o, o + 3, o + 6, d3, d4, d5);
    const double dtn = block_step_quantize(d, dtc, d.dt[i], tn);
    if (!finite) atomicOr(d.err, kErrNonFinite);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        d.x[k * n + i] = x1[k];
        d.v[k * n + i] = v1[k];
        d.a[k * n + i] = o[k];
        d.j[k * n + i] = o[3 + k];
        d.s[k * n + i] = o[6 + k];
        d.c[k * n + i] = d3[k];
    }
    d.pot[i] = o[9];
    d.t[i] = tn;
    d.dt[i] = dtn;
}

// 4th-order Hermite corrector (Makino & Aarseth 1992), o = {a1, j1, -, pot}:
//   v1 = v0 + h/2 (a0 + a1) + h^2/12 (j0 - j1)
//   x1 = x0 + h/2 (v0 + v1) + h^2/12 (a0 - a1)
// The cubic through (a, j) at both ends gives at t1
//   a2 = (6 (a0 - a1) + 2 h (j0 + 2 j1)) / h^2,  a3 = (12 (a0 - a1) + 6 h (j0 + j1)) / h^3,
// kept in s and c; new step from Aarseth's criterion
//   dt = sqrt(eta (|a1||a2| + |j1|^2) / (|j1||a3| + |a2|^2)).
__device__ __forceinline__ void correct_particle4(const Dev &d, int64_t i, double tn,
                                                  const double o[10]) {
    const int64_t n = d.n;
    const StepH H = step_powers(tn - d.t[i]);
    double x1[3], v1[3], a2[3], a3[3];
    bool finite = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const Axis4 r = correct_axis4(H.h, H.inv, d.x[k * n + i], d.v[k * n + i], d.a[k * n + i], d.j[k * n + i],
                                      o[k], o[3 + k]);
        x1[k] = r.x1; v1[k] = r.v1; a2[k] = r.a2; a3[k] = r.a3;
        finite = finite && isfinite(r.x1) && isfinite(r.v1) && isfinite(o[k]) && isfinite(o[3 + k]) &&
                 isfinite(r.a3);
    }
    const double dtc = criterion4(d, o, o + 3, a2, a3);
    const double dtn = block_step_quantize(d, dtc, d.dt[i], tn);
    if (!finite) atomicOr(d.err, kErrNonFinite);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        d.x[k * n + i] = x1[k];
        d.v[k * n + i] = v1[k];
        d.a[k * n + i] = o[k];
        d.j[k * n + i] = o[3 + k];
        d.s[k * n + i] = a2[k];
        d.c[k * n + i] = a3[k];
    }
    d.pot[i] = o[9];
    d.t[i] = tn;
    d.dt[i] = dtn;
}

// ------------------------------------------------ the corrector by a CTA
// log2 of a positive normal double, to 2^-13 (the exponent's float rounding);
// ok: it is one.
__device__ __forceinline__ float log2_rough(double x, bool &ok) {
    const int hi = __double2hiint(x);
    const int e = hi >> 20;
    ok = ok && (unsigned)(e - 1) < 2046u;
    return (float)(e - 1023) + __log2f(__int_as_float(0x3f800000 | ((hi & 0xfffff) << 3)));
}
// log2(2^a + 2^b)
__device__ __forceinline__ float log2_add(float a, float b) {
    return fmaxf(a, b) + __log2f(1.0f + exp2f(-fabsf(a - b)));
}
__device__ __forceinline__ bool pow2_field(double x, int &e) {  // x = 2^(e - 1023)
    const int hi = __double2hiint(x);
    e = hi >> 20;
    return ((hi & 0xfffff) | __double2loint(x)) == 0 && e > 100 && e < 1900;
}

// block_step_quantize for a criterion's dt known as log2 dt = l to better than
// 2^-10: its result depends on floor(log2 dt) alone while the steps are powers
// of two.  false: l is too close to a whole number, or a step is no power of two.
__device__ __forceinline__ bool quantize_rough(const Dev &d, float l, double dt_old, double tn, double &dtn) {
    constexpr float kTol = 1.0f / 1024.0f;
    const float f = floorf(l);
    int eo, emin, emax;
    const bool pow2 = pow2_field(dt_old, eo) && pow2_field(d.dt_min, emin) && pow2_field(d.dt_max, emax);
    if (!pow2 || !(l - f > kTol) || !(l - f < 1.0f - kTol)) return false;
    const int ec = (int)f + 1023;
    int e = eo;
    if (ec < emin) {
        e = emin;
        atomicAdd(d.ctr_underflow, 1ull);
    } else if (ec < eo) {
        e = ec;
    } else if (ec > eo) {
        const double q = tn * __hiloint2double((2045 - eo) << 20, 0);  // tn / (2 dt_old), exact
        if (q == trunc(q)) e = eo + 1;
    }
    e = min(max(e, emin), emax);
    dtn = __hiloint2double(e << 20, 0);
    return true;
}

// The corrector of the nv particles of an i-tile, by the whole CTA: four lanes a
// particle, one a coordinate, the particles dealt out over the warps.  red holds
// the sums, [q][ld]; index(il) gives particle il's global index or -1.  An FP64
// instruction occupies a warp's scheduler for 64 clocks whatever its lanes do,
// and this runs at the end of a step with the chip otherwise idle: one thread a
// particle was a chain of about 330 of them (eight square roots, three
// divisions, a cube root), 15 us of every block step.  A coordinate's share is
// about 55; the criterion's dt is needed only as a power of two, so its roots
// are taken as rough logarithms on the FP32 units and the FP64 form is kept for
// results within 2^-10 of a power of two (1 in 500), zeros and the non-finite.
// The same doubles as correct_particle / correct_particle4.
template <bool kOrder4, class Index>
__device__ __forceinline__ void correct_tile(const Dev &d, int nv, double tn, const double *red, int ld,
                                             Index index) {
    const int64_t n = d.n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int k = lane & 3, c = min(k, 2), q0 = lane & ~3;
    for (int base = 0; base < nv; base += 8 * warps) {
        const int il = base + (lane >> 2) * warps + warp;
        const int64_t gi = il < nv ? index(il) : -1;
        const bool live = gi >= 0;
        if (!__any_sync(0xffffffffu, live)) continue;
        const int64_t i = live ? gi : 0;
        const double *o = red + (live ? il : 0);
        const double a1 = o[c * ld], j1 = o[(3 + c) * ld], s1 = o[(6 + c) * ld];
        const double dt_old = d.dt[i];
        const StepH H = step_powers(live ? tn - d.t[i] : 1.0);
        double x1, v1, u[3], w[3], snew, cnew;  // the criterion's vectors, first and second three
        if constexpr (kOrder4) {
            const Axis4 r = correct_axis4(H.h, H.inv, d.x[c * n + i], d.v[c * n + i], d.a[c * n + i],
                                          d.j[c * n + i], a1, j1);
            x1 = r.x1; v1 = r.v1; snew = r.a2; cnew = r.a3;
            u[0] = a1; u[1] = j1; u[2] = r.a2;
            w[0] = w[1] = w[2] = r.a3;
            if (live && !(isfinite(x1) && isfinite(v1) && isfinite(a1) && isfinite(j1) && isfinite(r.a3)))
                atomicOr(d.err, kErrNonFinite);
        } else {
            const Axis6 r = correct_axis6(H, d.x[c * n + i], d.v[c * n + i], d.a[c * n + i], d.j[c * n + i],
                                          d.s[c * n + i], a1, j1, s1);
            x1 = r.x1; v1 = r.v1; snew = s1; cnew = r.d3;
            u[0] = a1; u[1] = j1; u[2] = s1;
            w[0] = r.d3; w[1] = r.d4; w[2] = r.d5;
            if (live && !(isfinite(x1) && isfinite(v1) && isfinite(a1) && isfinite(j1) && isfinite(s1) &&
                          isfinite(r.d3)))
                atomicOr(d.err, kErrNonFinite);
        }
        // lane c gathers vector c of each three (lane c' holds its coordinate c')
        // and forms the log2 of its square
        double su = 0.0, sw = 0.0;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int give = (c + 3 - r) % 3, from = q0 + (c + r) % 3;
            const double eu = give == 0 ? u[0] : give == 1 ? u[1] : u[2];
            const double ew = give == 0 ? w[0] : give == 1 ? w[1] : w[2];
            const double pu = __shfl_sync(0xffffffffu, eu, from), pw = __shfl_sync(0xffffffffu, ew, from);
            su = fma(pu, pu, su);
            sw = fma(pw, pw, sw);
        }
        bool ok = true;
        const float lu = log2_rough(su, ok), lw = log2_rough(sw, ok);
        float U[3], W[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            U[r] = __shfl_sync(0xffffffffu, lu, q0 + r);
            W[r] = __shfl_sync(0xffffffffu, lw, q0 + r);
        }
        ok = ((__ballot_sync(0xffffffffu, ok) >> q0) & 7u) == 7u;
        bool eta_ok = true;
        const float leta = log2_rough(d.eta, eta_ok);
        float l;
        if constexpr (kOrder4)
            l = 0.5f * (leta + log2_add(0.5f * (U[0] + U[2]), U[1]) - log2_add(0.5f * (U[1] + W[0]), U[2]));
        else
            l = leta + (log2_add(0.25f * (U[0] + U[2]), 0.5f * U[1]) -
                        log2_add(0.25f * (W[0] + W[2]), 0.5f * W[1])) * (1.0f / 3.0f);
        double dtn = dt_old;
        const bool done = !live || k != 0 || (ok && eta_ok && quantize_rough(d, l, dt_old, tn, dtn));
        if (__any_sync(0xffffffffu, !done)) {
            double V[6][3];
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    V[q][r] = __shfl_sync(0xffffffffu, u[q], q0 + r);
                    V[3 + q][r] = __shfl_sync(0xffffffffu, w[q], q0 + r);
                }
            if (!done) {
                double dtc;
                if constexpr (kOrder4) dtc = criterion4(d, V[0], V[1], V[2], V[3]);
                else dtc = criterion6(d, V[0], V[1], V[2], V[3], V[4], V[5]);
                dtn = block_step_quantize(d, dtc, dt_old, tn);
            }
        }
        if (live && k < 3) {
            d.x[c * n + i] = x1;
            d.v[c * n + i] = v1;
            d.a[c * n + i] = a1;
            d.j[c * n + i] = j1;
            d.s[c * n + i] = snew;
            d.c[c * n + i] = cnew;
            if (k == 0) {
                d.pot[i] = o[9 * ld];
                d.t[i] = tn;
                d.dt[i] = dtn;
            }
        }
    }
}

}  // namespace nb
