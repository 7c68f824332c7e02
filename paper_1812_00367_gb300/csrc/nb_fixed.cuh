// nb_fixed.cuh -- fixed-point arithmetic of the FP64 pair terms.
//
// GB300 retires 2 FP64 lanes per clock and SM, but 64 lanes of IMAD.WIDE
// (32 x 32 -> 64 bits, 64-bit addend), 64 of shifts and logic and 128 of FP32
// (measured).  One FP64 instruction therefore costs as much as 32 integer
// ones, and a 62 x 62 bit product is four IMAD.WIDE.  The pair terms keep the
// FP64 pipe for what needs its range per particle (the coordinate differences
// and the nine running sums) and evaluate the rest on the integer pipe: every
// component of r, v and a of a pair is a 62-bit integer with an exponent of its
// own (fx_vectors), the reciprocal square root is an SFU seed with one
// third-order step on integers, and w1, w2, q return to doubles by a shift.
//
// Accuracy (u = 2^-53; CPU tests).  Relative to a vector's norm, rms over pairs
// of any scale: acceleration term 0.4-0.5 u, jerk 0.6-0.8 u, snap 0.6-0.9 u,
// against 1.7 u, 2.2-2.9 u and 2.8-4.8 u of the same terms in doubles.  Each
// component relative to its own summands, in systems thin along an axis down to
// 1e-12, chains, bulk motion: 0.4-0.7 u against 1.1-2.9 u in doubles.  Range: as
// the doubles', except that a component of jerk or snap below 1e-285 is zero.
//
// The functions run on the host too (the check of the arithmetic against long
// double is a CPU test); there the SFU seed is a rounded reciprocal root.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define NB_HD __host__ __device__ __forceinline__
#else
#define NB_HD inline
#endif

namespace nb {

// A vector of three with one exponent: component k is w[k] 2^(e - 61), |w[k]| < 2^62.
struct Fx3 {
    int64_t w[3];
    int32_t e;
};
// A 64-bit factor as hi 2^32 + lo with a signed low half.
struct FxS {
    int32_t h, l;
};

// Block forms (fx_pack): exponents lie in [kFxMinExp, kFxMaxExp]; a block with a
// non-finite component (or one beyond 2^kFxMaxExp) carries kFxBad and turns
// the sums that use it into NaN.
constexpr int kFxMinExp = -900;
constexpr int kFxMaxExp = 300;
constexpr int kFxBad = 4096;

NB_HD int fx_clz(uint32_t x) {
#if defined(__CUDA_ARCH__)
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}
// Place of the highest bit that differs from the sign, -1 if there is none.
NB_HD int fx_top(int32_t h) {
#if defined(__CUDA_ARCH__)
    int r;
    asm("bfind.s32 %0, %1;" : "=r"(r) : "r"(h));
    return r;
#else
    const uint32_t x = (uint32_t)(h ^ (h >> 31));
    return x ? 31 - __builtin_clz(x) : -1;
#endif
}
NB_HD float fx_u2f_rz(uint32_t x) {
#if defined(__CUDA_ARCH__)
    return __uint2float_rz(x);
#else
    const int n = fx_clz(x);
    return (float)(n < 8 ? x & (0xFFFFFFFFu << (8 - n)) : x);
#endif
}
NB_HD float fx_fma_rz(float a, float b, float c) {
#if defined(__CUDA_ARCH__)
    return __fmaf_rz(a, b, c);
#else
    const double s = (double)a * (double)b + (double)c;  // exact for the operands used here
    float f = (float)s;
    if ((double)f > s) f = std::nextafter(f, 0.0f);
    return f;
#endif
}
NB_HD float fx_fmul(float a, float b) {  // not to be joined with an addition
#if defined(__CUDA_ARCH__)
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
NB_HD uint32_t fx_f2bits(float f) {
#if defined(__CUDA_ARCH__)
    return (uint32_t)__float_as_int(f);
#else
    uint32_t u;
    std::memcpy(&u, &f, 4);
    return u;
#endif
}
NB_HD float fx_bits2f(uint32_t u) {
#if defined(__CUDA_ARCH__)
    return __int_as_float((int)u);
#else
    float f;
    std::memcpy(&f, &u, 4);
    return f;
#endif
}
NB_HD int64_t fx_d2bits(double d) {
#if defined(__CUDA_ARCH__)
    return __double_as_longlong(d);
#else
    int64_t u;
    std::memcpy(&u, &d, 8);
    return u;
#endif
}
NB_HD double fx_bits2d(uint32_t hi, uint32_t lo) {
#if defined(__CUDA_ARCH__)
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t u = ((uint64_t)hi << 32) | lo;
    double d;
    std::memcpy(&d, &u, 8);
    return d;
#endif
}
NB_HD float fx_rsqrt_seed(float x) {
#if defined(__CUDA_ARCH__)
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return (float)(1.0 / std::sqrt((double)x));
#endif
}
// shifts with the count clamped at 63 (a count of 64 or more gives the sign)
NB_HD int64_t fx_sar(int64_t x, int n) {
#if defined(__CUDA_ARCH__)
    int64_t r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
#else
    return x >> (n > 63 ? 63 : n);
#endif
}
NB_HD uint64_t fx_shr(uint64_t x, int n) {
#if defined(__CUDA_ARCH__)
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
#else
    return n > 63 ? 0 : x >> n;
#endif
}
NB_HD uint64_t fx_shl(uint64_t x, int n) {
#if defined(__CUDA_ARCH__)
    uint64_t r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
#else
    return n > 63 ? 0 : x << n;
#endif
}
NB_HD int64_t fx_mul(int32_t a, int32_t b) { return (int64_t)a * (int64_t)b; }
NB_HD uint64_t fx_mulu(uint32_t a, uint32_t b) { return (uint64_t)a * (uint64_t)b; }
// a b + c: one IMAD.WIDE
NB_HD int64_t fx_mad(int32_t a, int32_t b, int64_t c) {
#if defined(__CUDA_ARCH__)
    int64_t r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (int64_t)((uint64_t)fx_mul(a, b) + (uint64_t)c);
#endif
}
NB_HD uint64_t fx_madu(uint32_t a, uint32_t b, uint64_t c) {
#if defined(__CUDA_ARCH__)
    uint64_t r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return fx_mulu(a, b) + c;
#endif
}
NB_HD int32_t fx_max3(int32_t a, int32_t b, int32_t c) {
    const int32_t m = a > b ? a : b;
    return m > c ? m : c;
}
NB_HD int32_t fx_imin3(int32_t a, int32_t b, int32_t c) {
    const int32_t m = a < b ? a : b;
    return m < c ? m : c;
}
NB_HD uint32_t fx_min3(uint32_t a, uint32_t b, uint32_t c) {
    const uint32_t m = a < b ? a : b;
    return m < c ? m : c;
}
// The factors 1 and 2 as run-time values: x.hi is added to a 64-bit sum by
// one IMAD.WIDE with them, where a constant factor would be turned into a
// sign extension and a carry chain (three instructions).
struct FxK {
    int32_t one, two;
};
NB_HD int32_t fx_hi(int64_t x) { return (int32_t)(x >> 32); }
NB_HD uint32_t fx_hiu(uint64_t x) { return (uint32_t)(x >> 32); }
NB_HD FxS fx_split(int64_t w) {
    FxS s;
    s.l = (int32_t)(uint32_t)w;
    s.h = fx_hi(w) + (int32_t)((uint32_t)w >> 31);
    return s;
}
constexpr int64_t kFxHalf = (int64_t)1 << 31;
// a b / 2^64 to within about a unit (the product of the low halves, below a
// quarter unit, is left out; the rest is rounded to nearest)
NB_HD int64_t fx_mulhi(FxS a, FxS b, FxK K) {
    const int64_t c = fx_mad(a.l, b.h, fx_mad(a.h, b.l, kFxHalf));
    return fx_mad(fx_hi(c), K.one, fx_mul(a.h, b.h));
}
// a^2 / 2^64, as fx_mulhi
NB_HD int64_t fx_sqrhi(FxS a, FxK K) {
    const int64_t c = fx_mad(a.h, a.l, kFxHalf);
    return fx_mad(fx_hi(c), K.two, fx_mul(a.h, a.h));
}
// a b / 2^64 for unsigned factors of at most 2^63, floor to within two units
NB_HD uint64_t fx_mulhi_u(uint64_t a, uint64_t b, FxK K) {
    const uint32_t ah = fx_hiu(a), al = (uint32_t)a, bh = fx_hiu(b), bl = (uint32_t)b;
    const uint64_t u = fx_madu(al, bh, fx_mulu(ah, bl));
    return fx_madu(fx_hiu(u), (uint32_t)K.one, fx_mulu(ah, bh));
}
// a.b / 2^64 of two vectors, each cross sum rounded to nearest
NB_HD int64_t fx_dot(const FxS a[3], const FxS b[3], FxK K) {
    int64_t h = fx_mul(a[0].h, b[0].h), c1 = fx_mad(a[0].h, b[0].l, kFxHalf), c2 = fx_mad(a[0].l, b[0].h, kFxHalf);
    for (int k = 1; k < 3; ++k) {
        h = fx_mad(a[k].h, b[k].h, h);
        c1 = fx_mad(a[k].h, b[k].l, c1);
        c2 = fx_mad(a[k].l, b[k].h, c2);
    }
    return fx_mad(fx_hi(c2), K.one, fx_mad(fx_hi(c1), K.one, h));
}
// a.a / 2^64
NB_HD int64_t fx_norm2(const FxS a[3], FxK K) {
    int64_t h = fx_mul(a[0].h, a[0].h), c = fx_mad(a[0].h, a[0].l, kFxHalf);
    for (int k = 1; k < 3; ++k) {
        h = fx_mad(a[k].h, a[k].h, h);
        c = fx_mad(a[k].h, a[k].l, c);
    }
    return fx_mad(fx_hi(c), K.two, h);
}

// ------------------------------------------------ vectors with one exponent
// fx_decode, fx_root and the conversions serve the kernels; fx_pack,
// fx_diff_norm, fx_inside, fx_dot, fx_w1 and fx_w2 are the pair term with one
// exponent for a vector, which the CPU check of the arithmetic compares: as exact
// as the kernels' against a vector's norm, not component by component.
// A vector of doubles as integers of at most 61 bits (component k is
// w[k] 2^(e - 60)): exact for components down to 2^-8 of the largest,
// below that cut at 2^-60 of it.
NB_HD Fx3 fx_pack(double x, double y, double z) {
    const double d[3] = {x, y, z};
    Fx3 r;
    int em = 0;
    for (int k = 0; k < 3; ++k) {
        const int ek = (int)((uint64_t)fx_d2bits(d[k]) >> 52) & 0x7ff;
        em = ek > em ? ek : em;
    }
    int e = em - 1023;
    if (e < kFxMinExp) e = kFxMinExp;
    const bool bad = e > kFxMaxExp;
    for (int k = 0; k < 3; ++k) {
        const int64_t b = fx_d2bits(d[k]);
        const int ek = (int)((uint64_t)b >> 52) & 0x7ff;
        const uint64_t mant = (((uint64_t)b & 0xfffffffffffffull) | ((uint64_t)1 << 52)) << 8;
        const uint64_t a = (bad || ek == 0) ? 0 : fx_shr(mant, e - (ek - 1023));
        r.w[k] = b < 0 ? -(int64_t)a : (int64_t)a;
    }
    r.e = bad ? kFxBad : e;
    return r;
}
// A mass: |m| = mm 2^(e - 62), mm in [2^62, 2^63) or 0.
NB_HD void fx_pack_mass(double m, uint64_t &mm, int &e, uint32_t &sign) {
    const int64_t b = fx_d2bits(m);
    const int ek = (int)((uint64_t)b >> 52) & 0x7ff;
    // a vanishing mass: an exponent below every range, so that q becomes 0
    sign = ek == 0 ? 0u : (uint32_t)((uint64_t)b >> 32) & 0x80000000u;
    mm = ek == 0 ? 0 : ((((uint64_t)b & 0xfffffffffffffull) | ((uint64_t)1 << 52)) << 10);
    e = ek == 0x7ff ? 2 * kFxBad : (ek == 0 ? -2 * kFxBad : ek - 1023);
}

// ------------------------------------------------------- a pair's vectors
// Difference of two stored vectors, normalised to the largest component.
NB_HD Fx3 fx_diff_norm(const int64_t *wj, int ej, const int64_t *wi, int ei) {
    const int e = ej > ei ? ej : ei;
    const int sj = e - ej, si = e - ei;
    Fx3 r;
    uint32_t t = 0;
    for (int k = 0; k < 3; ++k) {
        r.w[k] = fx_sar(wj[k], sj) - fx_sar(wi[k], si);  // < 2^62
        const int32_t h = fx_hi(r.w[k]);
        t |= (uint32_t)(h ^ (h >> 31));
    }
    // the largest component's top bit to bit 61 (a difference below 2^-29 of
    // the vectors stays unnormalised: its error is that of the vectors' scale)
    const int n = fx_clz(t) - 2;
    for (int k = 0; k < 3; ++k) r.w[k] = (int64_t)fx_shl((uint64_t)r.w[k], n);
    r.e = e + 1 - n;
    return r;
}
// Three doubles as a block; emin: biased exponent the block's scale stays at
// or above (the softening's), already shifted to the exponent field.
NB_HD Fx3 fx_decode(const double d[3], uint32_t emin_field) {
    uint32_t h[3], a[3], em = emin_field;
    for (int k = 0; k < 3; ++k) {
        h[k] = (uint32_t)((uint64_t)fx_d2bits(d[k]) >> 32);
        a[k] = h[k] & 0x7fffffffu;
        em = a[k] > em ? a[k] : em;
    }
    const int e = (int)(em >> 20);
    Fx3 r;
    for (int k = 0; k < 3; ++k) {
        const uint32_t lo = (uint32_t)fx_d2bits(d[k]);
        const uint32_t mh = (h[k] & 0xfffffu) | 0x100000u;
        const uint64_t w = (((uint64_t)mh << 32) | lo) << 9;
        const int64_t s = (int64_t)(int32_t)h[k] >> 31;
        // one's complement: a negative component is off by one unit, 2^-61
        r.w[k] = (int64_t)fx_shr(w, e - (int)(a[k] >> 20)) ^ s;
    }
    r.e = e - 1023;
    return r;
}

// Whether r lies below the softening's scale.
NB_HD bool fx_inside(const double d[3], uint32_t emin_field) {
    uint32_t m = 0;
    for (int k = 0; k < 3; ++k) {
        const uint32_t a = (uint32_t)((uint64_t)fx_d2bits(d[k]) >> 32) & 0x7fffffffu;
        m = a > m ? a : m;
    }
    return m < emin_field;
}
// eps^2 = eps_x 2^(2 E - 58) with eps_x in [2^58, 2^60), so that r^2 + eps^2
// of a block of exponent >= E lies in [2^58, 2^62) units; emin_field =
// (E + 1023) << 20.  0 and 0 for eps^2 = 0 (or below the normal range).
NB_HD void fx_eps2(double eps2, uint64_t &eps_x, uint32_t &emin_field) {
    eps_x = 0;
    emin_field = 0;
    const int64_t b = fx_d2bits(eps2);
    const int ek = (int)((uint64_t)b >> 52) & 0x7ff;
    if (b <= 0 || ek == 0 || ek == 0x7ff) return;
    const int ex = ek - 1023, E = (ex - (ex & 1)) / 2;  // floor(ex / 2)
    eps_x = (((uint64_t)b & 0xfffffffffffffull) | ((uint64_t)1 << 52)) << (6 + (ex & 1));
    emin_field = (uint32_t)(E + 1023) << 20;
}

// --------------------------------------------------------- conversions
// w 2^base as a double (rounded to nearest), base + 1023 given biased.
NB_HD double fx_to_double(int64_t w, int base_biased) {
    const int64_t s = w >> 63;
    const uint64_t a = (uint64_t)(w ^ s);
    const float f = fx_fma_rz(fx_u2f_rz((uint32_t)(a >> 32)), 4294967296.0f, fx_u2f_rz((uint32_t)a));
    const int ef = (int)(fx_f2bits(f) >> 23);  // 127 + floor(log2 a); 0 for a = 0
    const uint64_t m = (fx_shl(a, 127 + 62 - ef) + 0x200) >> 10;  // leading one at bit 52
    uint32_t hi = (uint32_t)(m >> 32) + ((uint32_t)(ef + base_biased - 127 - 1) << 20);
    hi = ef == 0 ? 0u : hi;
    hi |= (uint32_t)(s >> 32) & 0x80000000u;
    return fx_bits2d(hi, (uint32_t)m);
}
// The same for a w whose magnitude has a bit in the high word (fx_high).
NB_HD double fx_to_double_high(int64_t w, int base_biased) {
    const int64_t s = w >> 63;
    const uint64_t a = (uint64_t)(w ^ s);
    const int n = fx_clz((uint32_t)(a >> 32));
    const uint64_t m = (fx_shl(a, n - 1) + 0x200) >> 10;  // leading one at bit 52
    const uint32_t hi = (uint32_t)(m >> 32) + ((uint32_t)(base_biased + 62 - n) << 20);
    return fx_bits2d(hi | ((uint32_t)(s >> 32) & 0x80000000u), (uint32_t)m);
}
// The high word of the magnitude (one's complement for negative w).
NB_HD uint32_t fx_high(int64_t w) {
    const int32_t h = (int32_t)(w >> 32);
    return (uint32_t)(h ^ (h >> 31));
}
// a positive q 2^base as a double; clamped to infinity / zero outside the range
NB_HD void fx_q_to_double(uint64_t q, int base_biased, uint32_t &hi, uint32_t &lo) {
    const int n = fx_clz((uint32_t)(q >> 32));  // the caller's q has its top bit in the high word
    const uint64_t m = (fx_shl(q, n - 1) + 0x200) >> 10;
    int e = base_biased + 63 - n;
    e = e < 0 ? 0 : (e > 0x7ff ? 0x7ff : e);
    // the leading one adds one to the exponent; without it (e = 0) a number
    // below the normal range remains, which stands for zero
    hi = e == 0 ? 0u : (uint32_t)(m >> 32) + ((uint32_t)(e - 1) << 20);
    lo = e == 0 ? 0u : (uint32_t)m;
}

// The scalar part that every pair term starts with.
struct FxRoot {
    uint64_t y;   // 1/sqrt(r^2 + eps^2) = y 2^(-62 - g), y in (2^62, 2^63]
    uint64_t y2;  // its square, y2 2^(-60 - 2 g)
    int g, s;     // s: the even normalising shift of r^2 (0 or 2)
};
// eps^2 = eps_x 2^(2 (e - 1023) - 58) at the block exponent field e it was
// formed for (emin_field); for larger blocks it is shifted down.
NB_HD FxRoot fx_root(const FxS R[3], int e, uint64_t eps_x, uint32_t emin_field, FxK K) {
    uint64_t X = (uint64_t)fx_norm2(R, K);  // r^2 in units of 2^(2 e - 58)
    X += fx_shr(eps_x, 2 * (e + 1023 - (int)(emin_field >> 20)));
    FxRoot o;
    o.s = X < ((uint64_t)1 << 60) ? 2 : 0;
    X = fx_shl(X, o.s);  // x = X 2^-62 in [1/4, 1)
    o.g = e + 2 - (o.s >> 1);
    // seed from the top 32 bits: y0 = Y0 2^-23 in [1, 2)
    float y0 = fx_rsqrt_seed((float)(uint32_t)(X >> 30));
    y0 = fminf(fmaxf(y0, 1.52587890625e-05f), 3.0517576306010596e-05f);
    const uint32_t Y0 = (fx_f2bits(y0) & 0x7fffffu) | 0x800000u;
    // residual e = 1 - x y0^2 in units of 2^-58, |e| < 2^-21
    const uint32_t Ys = Y0 << 7;
    const uint64_t Z = fx_mulu(Ys, Ys);
    const int64_t e58 = ((int64_t)1 << 58) - (int64_t)fx_mulhi_u(X, Z, K);
    // (1 - e)^(-1/2) = 1 + e/2 + 3/8 e^2 + ..., in units of 2^-61
    const int32_t eh = (int32_t)(e58 >> 14);
    const int64_t c61 = fx_mad((int32_t)(fx_mul(eh, eh) >> 31), 6, e58 << 2);
    const uint64_t p = fx_mulu(Y0, (uint32_t)c61) + ((uint64_t)(Y0 * (uint32_t)fx_hi(c61)) << 32);
    o.y = ((uint64_t)Y0 << 39) + (uint64_t)((int64_t)p >> 22);
    const uint32_t yh = fx_hiu(o.y), yl = (uint32_t)o.y;
    o.y2 = fx_madu(fx_hiu(fx_mulu(yh, yl)), (uint32_t)K.two, fx_mulu(yh, yh));
    return o;
}

// 1/sqrt(r^2 + eps^2) as a double; no number when r (block exponent e) is not
// finite, 2^-1022 when it is larger than that says.
NB_HD double fx_root_to_double(const FxRoot &t, int e) {
    const uint64_t m = (t.y + 0x200) >> 10;  // leading one at bit 52
    const int x = 1023 - 1 - t.g;
    uint32_t hi = (uint32_t)(m >> 32) + ((uint32_t)(x > 0 ? x : 0) << 20);
    hi = e >= 1024 ? 0x7ff80000u : hi;
    return fx_bits2d(hi, (uint32_t)m);
}
// 1/sqrt(r^2 + eps^2) as a pair of floats, 24 + 24 bits; no number outside
// [2^-102, 2^126], where a float's exponent or the low part's bits end.
NB_HD void fx_root_to_floats(const FxRoot &t, float &yh, float &yl) {
    const uint32_t x = (uint32_t)(127 - 23 - t.g);
    const float s = fx_bits2f(x - 2u <= 228u ? x << 23 : 0x7fc00000u);
    yh = fx_fmul((float)(uint32_t)(t.y >> 39), s);
    yl = fx_fmul((float)((uint32_t)(t.y >> 15) & 0xffffffu), fx_fmul(s, 5.9604644775390625e-08f));
}

// y^3 in units of 2^(-58 - 3 g)
NB_HD uint64_t fx_y3(const FxRoot &t, FxK K) { return fx_mulhi_u(t.y, t.y2, K); }
// q = |m| y^3, with the sign put back, as a double.
NB_HD double fx_q(uint64_t y3, int g, uint64_t mm, int em, uint32_t sign, bool zero, FxK K) {
    const uint64_t Q = fx_mulhi_u(mm, y3, K);  // in units of 2^(em - 56 - 3 g)
    uint32_t hi, lo;
    fx_q_to_double(Q, (zero ? -2 * kFxBad : em) - 3 * g - 56 + 1023, hi, lo);
    return fx_bits2d(hi | sign, lo);
}

// Pair terms up to the jerk: alpha and w1 = v - 3 alpha r.
struct FxW1 {
    int64_t al;    // alpha in units of 2^(ev - er - 58)
    int64_t an3;   // -3 alpha, same units
    int64_t w[3];  // w1 in units of 2^(ev - 59)
};
NB_HD FxW1 fx_w1(const FxS R[3], const FxS V[3], const int64_t v[3], const FxRoot &t, FxS Y2, FxK K) {
    const int64_t rv = (int64_t)fx_shl((uint64_t)fx_dot(R, V, K), t.s);
    FxW1 o;
    o.al = fx_mulhi(fx_split(rv), Y2, K);
    o.an3 = -3 * o.al;
    const FxS a3 = fx_split(o.an3);
    for (int k = 0; k < 3; ++k) o.w[k] = (v[k] >> 2) + (fx_mulhi(a3, R[k], K) << 4);
    return o;
}
// w2 = a - 6 alpha w1 - 3 beta r in units of 2^(ez - er - 52), ez returned.
NB_HD void fx_w2(const FxS R[3], int er, const FxS V[3], int ev, const Fx3 &A, const FxRoot &t, FxS Y2,
                 const FxW1 &u, int64_t w2[3], int &ez, FxK K) {
    // v.v and r.a at the larger of their scales 2 ev, er + ea
    const int64_t vv = fx_norm2(V, K);
    const FxS As[3] = {fx_split(A.w[0]), fx_split(A.w[1]), fx_split(A.w[2])};
    const int64_t ra = fx_dot(R, As, K);
    const int ev2 = 2 * ev, era = er + A.e;
    ez = ev2 > era ? ev2 : era;
    const int dz = ez - ev2, da = ez - era;
    const int64_t w = fx_sar(vv, dz) + fx_sar(ra, da);
    const int64_t ze3 = 3 * fx_mulhi(fx_split(w), Y2, K);  // 3 zeta, units 2^(ez - 2 er - 58 + s)
    // -3 alpha^2 in units of 2^(2 ev - 2 er - 54)
    const int64_t aa3 = fx_mulhi(fx_split(u.al << 2), fx_split(u.an3), K);
    // -3 beta, units 2^(ez - 2 er - 55)
    const FxS b3 = fx_split((fx_sar(aa3, dz) << 1) - fx_sar(ze3, 3 - t.s));
    const FxS a3 = fx_split(fx_sar(u.an3, dz));
    for (int k = 0; k < 3; ++k) {
        const FxS w1 = fx_split(u.w[k]);
        const int64_t c1 = fx_mad(a3.l, w1.h, fx_mad(a3.h, w1.l, kFxHalf));
        const int64_t c2 = fx_mad(b3.l, R[k].h, fx_mad(b3.h, R[k].l, kFxHalf));
        int64_t h = fx_mad(a3.h, w1.h, fx_sar(A.w[k], da + 9));
        h = fx_mad(b3.h, R[k].h, h);
        w2[k] = fx_mad(fx_hi(c2), K.one, fx_mad(fx_hi(c1), K.one, h));
    }
}

// ------------------------------------- a pair's vectors, component by component
// The pair term of the kernels.  Every component of r, v and a has an exponent of
// its own, every product of a dot is aligned to the largest of the dot's products
// only, and w1_k, w2_k are sums of products of normalised integers aligned to the
// largest of their own summands.  Each component of jerk and snap is therefore at
// least as exact against its own summands (|v_k| + 3 |alpha r_k|, |a_k| + 6 |alpha
// w1_k| + 3 |beta r_k|) as in doubles, however thin the system is along an axis.
// With one exponent for a vector a component 2^-k of its vector's norm had k - 5
// bits less than in doubles (z / x = 1e-6: jerk z 2.9e-12 instead of 2.3e-16); the
// exponents cost 112 of now 760 instructions a pair and warp (FP64, N = 65536, A =
// 1000: 2.17 -> 2.46 ms; all, each pair once: 90.4 -> 96.6 ms).  Differences of v
// and a in doubles instead of integers: 18 FP64 instructions instead of 12, 2.68
// and 110.6 ms, and a rounding of each difference that the integers do not have.
// Leading places by bfind.s32 on the signed high word instead of clz of its
// magnitude: 784 -> 760 instructions, 2.51 -> 2.46 ms.
struct FxC3 {
    int64_t w[3];  // component k is w[k] 2^(f[k] - 1023 - 61), 2^61 <= |w[k]| < 2^62, or 0
    int32_t f[3];  // exponent fields (below 0: under the doubles' range)
    int32_t e;     // the largest
};
// r from its doubles.  None of them is -0: the records hold no -0, so their
// differences are none.
NB_HD FxC3 fx_components(const double d[3]) {
    FxC3 o;
    for (int k = 0; k < 3; ++k) {
        const uint32_t h = (uint32_t)((uint64_t)fx_d2bits(d[k]) >> 32), lo = (uint32_t)fx_d2bits(d[k]);
        o.f[k] = (int32_t)((h >> 20) & 0x7ffu);
        const uint32_t mh = o.f[k] == 0 ? 0u : (h & 0xfffffu) | 0x100000u;
        // one's complement: a negative component is off by one unit, 2^-61
        o.w[k] = (int64_t)((((uint64_t)mh << 32) | lo) << 9) ^ ((int64_t)(int32_t)h >> 31);
    }
    o.e = fx_max3(o.f[0], o.f[1], o.f[2]);
    return o;
}
// A particle's velocity or acceleration as it is stored: component k is
// w[k] 2^(f[k] - 1023 - 60), 2^60 <= |w[k]| < 2^61, or 0.
struct FxP3 {
    int64_t w[3];
    int32_t f[3];  // exponent fields; 0x7ff: not finite
};
NB_HD FxP3 fx_pack_components(const double d[3]) {
    FxP3 o;
    for (int k = 0; k < 3; ++k) {
        const int64_t b = fx_d2bits(d[k]);
        o.f[k] = (int32_t)((uint64_t)b >> 52) & 0x7ff;
        const int64_t m = o.f[k] == 0 ? 0 : (int64_t)((((uint64_t)b & 0xfffffffffffffull) | ((uint64_t)1 << 52)) << 8);
        o.w[k] = b < 0 ? -m : m;
    }
    return o;
}
// Differences of kVecs stored vectors: exact where the doubles' would be rounded,
// except below 2^-60 of the larger component.  top[q]: the largest stored field.
template <int kVecs>
NB_HD void fx_differences(const FxP3 *j, const FxP3 *i, FxC3 *o, int32_t *top) {
    int m[kVecs][3];
    int t[kVecs][3], low = 31;
    for (int q = 0; q < kVecs; ++q) {
        for (int k = 0; k < 3; ++k) {
            m[q][k] = j[q].f[k] > i[q].f[k] ? j[q].f[k] : i[q].f[k];
            o[q].w[k] = fx_sar(j[q].w[k], m[q][k] - j[q].f[k]) - fx_sar(i[q].w[k], m[q][k] - i[q].f[k]);  // < 2^62
            t[q][k] = fx_top(fx_hi(o[q].w[k]));
        }
        const int l3 = fx_imin3(t[q][0], t[q][1], t[q][2]);
        low = low < l3 ? low : l3;
        top[q] = fx_max3(m[q][0], m[q][1], m[q][2]);
    }
    if (low >= 0) {
        for (int q = 0; q < kVecs; ++q)
            for (int k = 0; k < 3; ++k) {
                o[q].w[k] = (int64_t)fx_shl((uint64_t)o[q].w[k], 29 - t[q][k]);
                o[q].f[k] = m[q][k] + t[q][k] - 28;
            }
    } else {  // a component below 2^-29 of the particles' own (or zero)
        for (int q = 0; q < kVecs; ++q)
            for (int k = 0; k < 3; ++k) {
                const int64_t w = o[q].w[k];
                const int n = t[q][k] >= 0 ? 29 - t[q][k] : 30 + fx_clz((uint32_t)(w ^ (w >> 63)));
                o[q].w[k] = (int64_t)fx_shl((uint64_t)w, n);
                o[q].f[k] = w == 0 ? -8192 : m[q][k] + 1 - n;
            }
    }
    for (int q = 0; q < kVecs; ++q) o[q].e = fx_max3(o[q].f[0], o[q].f[1], o[q].f[2]);
}
// Fields below kFxLow stand for zero (results under 2^-900); terms whose
// scale reaches kFxHigh may leave the doubles' range: fx_to_double_any.
constexpr int kFxLow = 64, kFxHigh = 2030;
// The same conversion for any w and any scale: zero at the bottom, infinity (or
// no number) at the top.
NB_HD double fx_to_double_any(int64_t w, int m) {
    const int64_t s = w >> 63;
    const uint64_t a = (uint64_t)(w ^ s);
    if (a == 0 || m <= kFxLow) return 0.0;
    const int n = (a >> 32) ? fx_clz((uint32_t)(a >> 32)) : 32 + fx_clz((uint32_t)a);
    const uint64_t x = (fx_shl(a, n) >> 1) + 0x200;
    const int e = m - 57 + 62 - n;
    uint32_t hi = (uint32_t)(x >> 42) + ((uint32_t)(e > 2046 ? 2046 : e) << 20);
    return fx_bits2d(hi | ((uint32_t)(s >> 32) & 0x80000000u), (uint32_t)(x >> 10));
}
// From the differences r, v, a (a in the 6th-order form only): the root t, w1 =
// v - 3 alpha r and w2 = a - 6 alpha w1 - 3 beta r as doubles.  top: the largest
// stored field of v and a.
template <bool kOrder6>
NB_HD void fx_vectors(const double r[3], const FxC3 &V, const FxC3 &A, int top, uint64_t eps_x,
                      uint32_t emin_field, FxK K, FxRoot &t, double w1[3], double w2[3]) {
    const FxC3 R = fx_components(r);
    const int emin = (int)(emin_field >> 20);
    const int er = R.e > emin ? R.e : emin;
    FxS Rs[3], Vs[3];
    {
        FxS B[3];  // r as a block, for r^2
        for (int k = 0; k < 3; ++k) B[k] = fx_split(fx_sar(R.w[k], er - R.f[k]));
        t = fx_root(B, er - 1023, eps_x, emin_field, K);
    }
    for (int k = 0; k < 3; ++k) {
        Rs[k] = fx_split(R.w[k]);
        Vs[k] = fx_split(V.w[k]);
    }
    const FxS Y2 = fx_split((int64_t)t.y2);
    // alpha = al 2^(ea - 60), al in +-[2^60, 2^61)
    const int g0 = R.f[0] + V.f[0], g1 = R.f[1] + V.f[1], g2 = R.f[2] + V.f[2];
    const int G = fx_max3(g0, g1, g2);
    const int64_t rv = fx_sar(fx_mulhi(Rs[0], Vs[0], K), G - g0) + fx_sar(fx_mulhi(Rs[1], Vs[1], K), G - g1) +
                       fx_sar(fx_mulhi(Rs[2], Vs[2], K), G - g2);  // units 2^(G - 58), below 2^61.6
    int64_t al = fx_mulhi(fx_split(rv), Y2, K);                      // units 2^(G - 2 er + s - 58), below 2^59.6
    const int na = 28 - fx_top(fx_hi(al));
    al = (int64_t)fx_shl((uint64_t)al, na);
    const int ea = G - 2 * er + t.s + 2 - na;
    const FxS a3 = fx_split(-3 * al);
    int64_t u1[3];  // w1_k = u1[k] 2^(m1[k] - 1023 - 57)
    int m1[3];
    for (int k = 0; k < 3; ++k) {
        const int ep = ea + R.f[k];
        m1[k] = fx_max3(ep, V.f[k], kFxLow);
        u1[k] = fx_sar(V.w[k], 4 + m1[k] - V.f[k]) + fx_sar(fx_mulhi(a3, Rs[k], K), m1[k] - ep);
    }
    uint32_t high = fx_min3(fx_high(u1[0]), fx_high(u1[1]), fx_high(u1[2]));
    int64_t u2[3];
    int m2[3];
    if (kOrder6) {
        FxS As[3];
        for (int k = 0; k < 3; ++k) As[k] = fx_split(A.w[k]);
        // v.v + r.a, its six products aligned to the largest
        const int h0 = R.f[0] + A.f[0], h1 = R.f[1] + A.f[1], h2 = R.f[2] + A.f[2];
        const int H = fx_max3(h0, h1, h2);
        const int ez = 2 * V.e > H ? 2 * V.e : H;
        int64_t w = fx_sar(fx_mulhi(Rs[0], As[0], K), ez - h0) + fx_sar(fx_mulhi(Rs[1], As[1], K), ez - h1) +
                    fx_sar(fx_mulhi(Rs[2], As[2], K), ez - h2);
        for (int k = 0; k < 3; ++k) w += fx_sar(fx_sqrhi(Vs[k], K), ez - 2 * V.f[k]);
        // units 2^(ez - 58), below 2^62.6; 3 zeta in units 2^(eZ - 58)
        const int64_t z3 = 3 * fx_mulhi(fx_split(w), Y2, K);
        const int eZ = ez - 2 * er + t.s;
        const int64_t aa3 = fx_mulhi(a3, fx_split(al), K);  // -3 alpha^2, units 2^(2 ea - 56)
        const int eA = 2 * ea + 2;
        const int mB = eA > eZ ? eA : eZ;
        int64_t b3 = fx_sar(aa3, mB - eA + 1) - fx_sar(z3, mB - eZ + 1);  // -3 beta, units 2^(mB - 57)
        const int nb = 29 - fx_top(fx_hi(b3));
        b3 = (int64_t)fx_shl((uint64_t)b3, nb);  // below 2^62, units 2^(mB - 57 - nb)
        const FxS B3 = fx_split(b3);
        const int eb = mB + 3 - nb;
        for (int k = 0; k < 3; ++k) {
            const int f1 = ea + m1[k] + 5, f2 = eb + R.f[k];
            const int m = m2[k] = fx_max3(f1, f2, A.f[k] > kFxLow ? A.f[k] : kFxLow);
            u2[k] = fx_sar(A.w[k], 4 + m - A.f[k]) + fx_sar(fx_mulhi(a3, fx_split(u1[k]), K), m - f1) +
                    fx_sar(fx_mulhi(B3, Rs[k], K), m - f2);
        }
        top = top > ez - er ? top : ez - er;
        high = fx_min3(high, fx_high(u2[0]), fx_high(u2[1]));
        high = high < fx_high(u2[2]) ? high : fx_high(u2[2]);
    }
    high = top > kFxHigh ? 0u : high;
    if (high != 0) {
        for (int k = 0; k < 3; ++k) {
            w1[k] = fx_to_double_high(u1[k], m1[k] - 57);
            if (kOrder6) w2[k] = fx_to_double_high(u2[k], m2[k] - 57);
        }
    } else {  // a component below 2^-26 of its summands' scale (or zero), or the range's ends
        for (int k = 0; k < 3; ++k) {
            w1[k] = fx_to_double_any(u1[k], m1[k]);
            if (kOrder6) w2[k] = fx_to_double_any(u2[k], m2[k]);
        }
    }
}

}  // namespace nb
