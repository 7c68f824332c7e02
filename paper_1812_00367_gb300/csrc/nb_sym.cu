// nb_sym.cu -- the evaluation of a whole cluster by itself (every particle
// active), each pair once.
//
// Of a pair's terms only the mass and the sign differ between its two members
// (r, v, a change sign together; y, alpha, beta do not), so the all-active
// sums need half the pair terms: i's share is q_j (r, w1, w2), j's is
// -q_i (r, w1, w2).  For the FP64 and EX terms (the sums of the FP32 ones keep
// their order of additions) and the potential.  Rows are i-tiles of 128 particles (one per thread), columns
// j-tiles of 64; row I meets the columns from 2 I on.  The first two are the
// row's own particles and are summed one-sided as in k_eval; in the others lane
// l of a warp starts at particle l of the tile and walks round it, so that the
// lanes always hold different j's, and adds j's share into its warp's sums in
// shared memory.
//
// Bound: the FP64 pipe and the issue of integer instructions together (6th
// order: 21 DFMA a pair for both members, 336 SM clocks a warp, against 2 x 192;
// 876 instructions against 2 x 760; FP64 pipe 77 % and ALU 48 % busy).  Measured,
// one-sided -> each pair once, ms: N = 65536 6th order 151.4 -> 96.6, 4th order 88.2
// -> 64.2; N = 30011 31.9 -> 20.4 and 18.6 -> 13.6; potential N = 65536 32.0 -> 19.7
// (FP64 pipe 85 % busy); EX, bound by its packed FP32 operations (about 620 a pair
// for both members instead of 2 x 500), N = 65536 62.5 -> 43.4, 4th order 35.8 ->
// 26.6, N = 30011 13.2 -> 9.2 and 7.6 -> 5.6.  2 or 3 CTAs per SM instead of 4, FP64:
// 8 % slower.
//
// Order of the sums: units (row, column) are cut into equal ranges over a fixed
// grid (as stream-K); each range leaves one partial per row it touches and each
// unit one per column particle, in slots of its own; k_sym_reduce adds them in
// row order.  No atomics: results are reproducible.  The units are taken in
// bands whose columns' partials fit the evaluation's scratch (199 MB; 8 bands at N
// = 65536), one launch of each kernel a band.
#include "nb_eval.cuh"
#include "nb_sym.cuh"

namespace nb {
namespace {

// values per particle in the partials: sums first, the potential last
template <int MODE>
constexpr int sym_nv() {
    return MODE == kModePot ? 1 : (uses_order4_terms(MODE) ? 7 : 10);
}
// place of value v in the ten sums
template <int MODE>
__device__ __forceinline__ int sym_q(int v) {
    return v == sym_nv<MODE>() - 1 ? 9 : v;
}

template <int P, int MODE>
struct SymSmem {
    typename Prec<P>::J tile[kStages][kTJ / Prec<P>::kPerRec];
    // per warp: the sums of the tile's particles, one double each (FP64: the
    // potential as a float pair in its bits), EX: hi and lo of a record's two
    // particles in the room of two doubles
    alignas(16) double jsum[kTPB / 32][sym_nv<MODE>()][kTJ];
    uint64_t bar[kStages];
    long long u, u_end;  // next unit, end of the CTA's range
    long long tb, te;    // columns of the current piece
    int row, flag, fail;
};

// Both members' shares of one pair.
template <int MODE>
__device__ __forceinline__ void sym_pair(const Prec<NB_FP64>::I &i, const JFX &own, const JFX &jj, bool valid,
                                         Prec<NB_FP64>::Acc &c, double (*js)[kTJ], int k) {
    using T = Prec<NB_FP64>;
    constexpr bool k6 = !uses_order4_terms(MODE);
    T::Terms o;
    T::terms<k6>(i, jj, c, o);
    float yh, yl;
    fx_root_to_floats(o.t, yh, yl);
    T::pot_term(jj.mf, yh, yl, c.pf);
    const uint64_t y3 = fx_y3(o.t, i.K);
    T::add<k6>(fx_q(y3, o.t.g, jj.mm, jfx_em(jj), jfx_sign(jj), false, i.K), o, c);
    // -q_i: the sign bit turned
    const double nq = fx_q(y3, o.t.g, own.mm, jfx_em(own), jfx_sign(own) ^ 0x80000000u, !valid, i.K);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        js[q][k] = fma(nq, o.r[q], js[q][k]);
        js[3 + q][k] = fma(nq, o.w1[q], js[3 + q][k]);
        if constexpr (k6) js[6 + q][k] = fma(nq, o.w2[q], js[6 + q][k]);
    }
    double &pj = js[sym_nv<MODE>() - 1][k];  // the float pair of j's potential
    ff p{__int_as_float(__double2hiint(pj)), __int_as_float(__double2loint(pj))};
    T::pot_term(valid ? own.mf : make_float2(0.f, 0.f), yh, yl, p);
    pj = __hiloint2double(__float_as_int(p.hi), __float_as_int(p.lo));
}
// EX: one record, two pairs.
__device__ __forceinline__ void sym_add_ex(float4 *sum, ff2 a, ff2 b) {
    float4 v = *sum;  // (hi, hi, lo, lo) of the record's two particles
    ff2 acc{lo2(v), hi2(v)};
    ff_fma_acc_lazy(acc, a, b);
    *sum = make_float4(acc.hi.x, acc.hi.y, acc.lo.x, acc.lo.y);
}
template <int MODE>
__device__ __forceinline__ void sym_pair(const Prec<NB_EX>::I &i, ff2 nmi, const JEXP &jj, ff2 eps2,
                                         Prec<NB_EX>::Acc &c, float4 (*js)[kTJ / 2], int k) {
    using T = Prec<NB_EX>;
    constexpr bool k6 = !uses_order4_terms(MODE);
    ff2 r[3], v[3], a[3];
    T::rel(i, jj, r, v);
    const ff2 m{hi2(jj.q[1]), hi2(jj.q[3])};
    const ff2 y = rsqrt_ff(k6 ? ff_dot3_add_lazy(r, r, eps2) : ff_dot3_add(r, r, eps2));
    const ff2 y2 = ff_sqr_lazy(y);
    const ff2 my = ff_mul_lazy(m, y), myi = ff_mul_lazy(nmi, y);  // m_j y, -m_i y
    ff_add_lazy(c.p, my);
    {
        float4 &p = js[sym_nv<MODE>() - 1][k];
        ff2 acc{lo2(p), hi2(p)};
        ff_add_lazy(acc, myi);
        p = make_float4(acc.hi.x, acc.hi.y, acc.lo.x, acc.lo.y);
    }
    const ff2 q = ff_mul_lazy(my, y2), nq = ff_mul_lazy(myi, y2);
    const ff2 al = ff_mul_lazy(k6 ? ff_dot3_lazy(r, v) : ff_dot3(r, v), y2);
    const ff2 al3 = ff_mul_f_lazy(al, f2s(3.0f));
    ff2 be3, al6;
    if constexpr (k6) {
        a[0] = ff_sub(ff2{hi2(jj.q[5]), hi2(jj.q[7])}, i.a[0]);
        a[1] = ff_sub(ff2{lo2(jj.q[8]), lo2(jj.q[9])}, i.a[1]);
        a[2] = ff_sub(ff2{hi2(jj.q[8]), hi2(jj.q[9])}, i.a[2]);
        const ff2 ze = ff_mul_lazy(ff_dot3x2_lazy(v, v, r, a), y2);
        be3 = ff_mul_f_lazy(ff_sum_lazy(ff_sqr_lazy(al), ze), f2s(3.0f));
        al6 = ff2{add2(al3.hi, al3.hi), add2(al3.lo, al3.lo)};  // exact
    }
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        const ff2 w1 = ff_fnma_lazy(al3, r[t], v[t]);
        ff_fma_acc_lazy(c.a[t], q, r[t]);
        sym_add_ex(&js[t][k], nq, r[t]);
        ff_fma_acc_lazy(c.j[t], q, w1);
        sym_add_ex(&js[3 + t][k], nq, w1);
        if constexpr (k6) {
            const ff2 w2 = ff_fnma_lazy(be3, r[t], ff_fnma_lazy(al6, w1, a[t]));
            ff_fma_acc_lazy(c.s[t], q, w2);
            sym_add_ex(&js[6 + t][k], nq, w2);
        }
    }
}
__device__ __forceinline__ void sym_pot(const Prec<kPrecPot>::I &i, double mi, const J64 &jj,
                                        Prec<kPrecPot>::Acc &c, double (*js)[kTJ], int k) {
    const double y = Prec<kPrecPot>::root(i, jj);
    c.p = fma(jj.q[1].y, y, c.p);
    js[0][k] = fma(mi, y, js[0][k]);
}

template <int P, int MODE>
__global__ void __launch_bounds__(kTPB, 4) k_sym(const Dev d, const SymLaunch L) {
    using T = Prec<P>;
    using J = typename T::J;
    constexpr int NV = sym_nv<MODE>();
    constexpr int kRecs = kTJ / T::kPerRec;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    SymSmem<P, MODE> &S = *reinterpret_cast<SymSmem<P, MODE> *>(smem_raw);
    if (L.gate && *L.gate != 0) return;  // not the whole cluster in order
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const J *jc = reinterpret_cast<const J *>(d.jarr) + d.jofs[L.cluster] / T::kPerRec;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) mbar_init(&S.bar[s], 1);
        S.fail = 0;
        fence_mbar_init();
        S.u = L.u0 + sk_begin(L.units, gridDim.x, blockIdx.x);
        S.u_end = L.u0 + sk_begin(L.units, gridDim.x, blockIdx.x + 1);
    }
    uint32_t phase = 0, pending = 0;  // as in k_eval
    for (;;) {
        if (tid == 0) {
            S.row = -1;
            if (S.u < S.u_end) {
                const int row = sym_row(S.u, L.ntj);
                const long long first = sym_first(row, L.ntj);
                S.row = row;
                S.tb = 2LL * row + (S.u - first);
                S.te = min((long long)L.ntj, S.tb + (S.u_end - S.u));
            }
        }
        __syncthreads();
        if (S.row < 0) break;
        const int row = S.row;
        const int64_t tb = S.tb, te = S.te;
        const int64_t il = (int64_t)row * kTPB + tid;
        const bool valid = il < L.n;
        typename T::I me = T::load_i(jc, valid ? il : 0);
        if constexpr (P != NB_EX) T::prepare(me, d);
        const J own = jc[(valid ? il : 0) / T::kPerRec];
        ff2 nmi{f2s(0.f), f2s(0.f)};  // EX: -m_i
        if constexpr (P == NB_EX) {
            const float *f = reinterpret_cast<const float *>(&own) + (il & 1);
            if (valid) nmi = ff2{f2s(-f[2 * 3]), f2s(-f[2 * 7])};
        }
        typename T::Acc acc;
        T::zero(acc);
        if (tid == 0) {
            for (int s = 0; s < kStages && tb + s < te; ++s) {
                mbar_expect_tx(&S.bar[s], kRecs * sizeof(J));
                tma_load_1d(&S.tile[s][0], jc + (tb + s) * kRecs, kRecs * sizeof(J), &S.bar[s]);
                pending |= 1u << s;
            }
        }
        bool ok = true;
        for (int64_t tt = tb; tt < te; ++tt) {
            const int s = (int)((tt - tb) % kStages);
            if (ok) ok = mbar_wait_bounded(&S.bar[s], (phase >> s) & 1u);
            phase ^= 1u << s;
            const J *tl = &S.tile[s][0];
            const bool own_cols = tt < 2LL * row + 2;  // uniform over the CTA
            if (ok && own_cols) {
                const int js = (int)min(max(il - tt * kTJ, (int64_t)-1), (int64_t)kTJ);
                tile_pairs<P, MODE, true>(d, me, tl, js, 0, 1, acc);
            } else if (ok) {
                double (*js)[kTJ] = S.jsum[warp];
#pragma unroll
                for (int q = 0; q < NV; ++q) js[q][lane] = js[q][lane + 32] = 0.0;
                __syncwarp();
#pragma unroll 1
                for (int k0 = 0; k0 < kRecs; ++k0) {
                    const int k = (lane + k0) & (kRecs - 1);
                    if constexpr (P == NB_EX)
                        sym_pair<MODE>(me, nmi, tl[k], ff2{d.eps2_hi2, d.eps2_lo2}, acc,
                                       reinterpret_cast<float4(*)[kTJ / 2]>(js), k);
                    else if constexpr (P == kPrecPot) sym_pot(me, valid ? own.q[1].y : 0.0, tl[k], acc, js, k);
                    else sym_pair<MODE>(me, own, tl[k], valid, acc, js, k);
                    __syncwarp();  // the next lane takes this j over
                }
            }
            if constexpr (P != kPrecPot) T::tile_done(acc);
            if (!ok) S.fail = 1;
            __syncthreads();
            if (S.fail) break;
            if (tid == 0) {
                pending &= ~(1u << s);
                if (tt + kStages < te) {
                    mbar_expect_tx(&S.bar[s], kRecs * sizeof(J));
                    tma_load_1d(&S.tile[s][0], jc + (tt + kStages) * kRecs, kRecs * sizeof(J), &S.bar[s]);
                    pending |= 1u << s;
                }
            }
            if (!own_cols) {  // the warps' sums of the tile's particles, in warp order
                double *out = L.jpart + (S.u - L.u0 + (tt - tb)) * (int64_t)(NV * kTJ);
                for (int e = tid; e < NV * kTJ; e += kTPB) {
                    const int q = e / kTJ, k = e % kTJ;
                    double sum = 0.0;
#pragma unroll
                    for (int w = 0; w < kTPB / 32; ++w) {
                        if constexpr (P == NB_EX) {
                            const float *f = reinterpret_cast<const float *>(&S.jsum[w][q][0]) + 4 * (k >> 1) + (k & 1);
                            sum += (double)f[0] + (double)f[2];
                            continue;
                        }
                        const double v = S.jsum[w][q][k];
                        if (P == NB_FP64 && q == NV - 1)
                            sum += (double)__int_as_float(__double2hiint(v)) + (double)__int_as_float(__double2loint(v));
                        else
                            sum += v;
                    }
                    out[e] = sum;
                }
                __syncthreads();
            }
        }
        if (S.fail) {
            if (tid == 0) {
                atomicOr(d.err, kErrTimeout);
                for (int s = 0; s < kStages; ++s)
                    if (pending & (1u << s)) (void)mbar_wait_bounded(&S.bar[s], (phase >> s) & 1u);
            }
            return;
        }
        double o[10];
        if constexpr (P == NB_FP64) {
            T::template finish<!uses_order4_terms(MODE)>(acc, o);
            // a velocity or acceleration that is not finite spoils every other
            // particle's sums: the reduction is told (row 0 meets every particle
            // and lies in the first band, so no band's reduction comes too early)
            const int bad = acc.fv >= 0x7ff ? 3 : (acc.fa >= 0x7ff ? 2 : 0);
            if (bad) atomicOr(L.bad, bad);
        } else if constexpr (P == NB_EX) {
            T::finish(acc, nullptr, 0, o);
        } else {
            T::finish(acc, o);
        }
        double *part = L.ipart + (row - L.row0 + blockIdx.x) * (10 * kTPB) + tid;
#pragma unroll
        for (int q = 0; q < 10; ++q) part[q * kTPB] = o[q];
        __syncthreads();
        if (tid == 0) S.u += S.te - S.tb;
    }
}

// One j-tile's particles: what the earlier bands gave, the band's pieces of their
// own row, then the shares from the band's rows above, in row order.
constexpr int kSymRedTPB = 320;
template <int P, int MODE>
__global__ void __launch_bounds__(kSymRedTPB) k_sym_reduce(const Dev d, const SymLaunch L, int grid_sym) {
    constexpr int NV = sym_nv<MODE>();
    __shared__ double sums[10][kTJ];
    if (L.gate && *L.gate != 0) return;
    const int tile = (int)(2 * L.row0) + blockIdx.x, row = tile / 2, il0 = (tile & 1) * kTJ;
    const long long u1 = L.u0 + L.units, f0 = sym_first(row, L.ntj), f1 = sym_first(row + 1, L.ntj);
    const bool last = f1 <= u1;  // the particles' own row ends here: nothing more to come
    long long k0 = 0, k1 = -1;
    if (f0 < u1) {
        k0 = sk_owner(L.units, grid_sym, max(f0, (long long)L.u0) - L.u0);
        k1 = sk_owner(L.units, grid_sym, min(f1, u1) - L.u0 - 1);
    }
    // rows above with their unit of this column in the band: the first and the
    // last of them may be just outside
    auto unit = [&](long long r) { return sym_first(r, L.ntj) + (tile - 2 * r); };
    int r0 = (int)L.row0, r1 = min(row, sym_row(u1 - 1, L.ntj) + 1);
    if (r0 < r1 && unit(r0) < L.u0) ++r0;
    if (r0 < r1 && unit(r1 - 1) >= u1) --r1;
    double *so_far = L.sums + (int64_t)tile * (NV * kTJ);
    for (int e = threadIdx.x; e < NV * kTJ; e += kSymRedTPB) {
        const int v = e / kTJ, k = e % kTJ, q = sym_q<MODE>(v);
        double sum = L.u0 > 0 ? so_far[e] : 0.0;
        for (long long c = k0; c <= k1; ++c)
            sum += __ldcs(L.ipart + (row - L.row0 + c) * (10 * kTPB) + q * kTPB + il0 + k);
        double above = 0.0;
        for (int r = r0; r < r1; r += 8) {
            double t[8];
#pragma unroll
            for (int x = 0; x < 8; ++x)
                t[x] = r + x < r1 ? __ldcs(L.jpart + (unit(r + x) - L.u0) * (int64_t)(NV * kTJ) + e) : 0.0;
#pragma unroll
            for (int x = 0; x < 8; ++x) above += t[x];
        }
        // FP64's shares of the potential are sums of m y, its sum carries the sign
        sum = q == 9 && P != NB_EX ? sum - above : sum + above;
        if (!last) so_far[e] = sum;
        sums[q][k] = sum;
    }
    if (!last) return;
    __syncthreads();
    const int64_t il = (int64_t)tile * kTJ + threadIdx.x;
    if (threadIdx.x < kTJ && il < L.n) {
        double o[10];
        const double nan = __hiloint2double(0x7ff80000, 0);
        const int bad = P == NB_FP64 ? *L.bad : 0;
#pragma unroll
        for (int q = 0; q < 10; ++q) {
            const bool here = MODE == kModePot ? q == 9 : (!uses_order4_terms(MODE) || q < 6 || q == 9);
            o[q] = here ? sums[q][threadIdx.x] : 0.0;
        }
        if constexpr (P == NB_FP64) {
            const bool bad_x = !(isfinite(o[0]) && isfinite(o[1]) && isfinite(o[2]));
#pragma unroll
            for (int q = 0; q < 10; ++q)
                if ((bad_x || (q >= 3 && q < 6 && (bad & 1)) || (q >= 6 && q < 9 && bad)) &&
                    !(uses_order4_terms(MODE) && q >= 6 && q < 9))
                    o[q] = nan;
        }
        EvalLaunch E{};
        E.out = L.out;
        E.n_active = (int32_t)L.n;
        finalize_one<P, MODE>(d, E, L.cluster, d.offsets[L.cluster] + il, (int)il, o);
    }
}

// Whether active is off, off + 1, ..., off + n - 1 (gate stays 0).
__global__ void k_sym_check(const int32_t *active, int64_t n, int64_t off, int *gate) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n && active[i] != off + i) atomicOr(gate, 1);
}

template <int P, int MODE>
cudaError_t go(const Dev &d, const SymLaunch &L0, int grid, cudaStream_t st) {
    constexpr size_t smem = sizeof(SymSmem<P, MODE>);
    constexpr int NV = sym_nv<MODE>();
    SymLaunch L = L0;
    const int64_t bands = sym_bands(L.ntj, grid, NV, d.partial_cap);
    if (bands <= 0) return cudaErrorInvalidValue;
    L.ipart = d.partial;
    L.sums = L.ipart + sym_piece_doubles(L.ntj, grid);
    L.jpart = L.sums + sym_sum_doubles(L.ntj, NV);
    for (int64_t b = 0; b < bands; ++b) {
        L.u0 = sym_band_first(L.ntj, grid, bands, b);
        L.units = sym_band_first(L.ntj, grid, bands, b + 1) - L.u0;
        L.row0 = sym_row(L.u0, L.ntj);
        k_sym<P, MODE><<<grid, kTPB, smem, st>>>(d, L);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        k_sym_reduce<P, MODE><<<(unsigned)(L.ntj - 2 * L.row0), kSymRedTPB, 0, st>>>(d, L, grid);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}
template <int P, int MODE>
int resident() {  // CTAs per SM, after raising the shared-memory limit
    constexpr int smem = (int)sizeof(SymSmem<P, MODE>);
    int b = 0;
    if (cudaFuncSetAttribute(k_sym<P, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_sym<P, MODE>, kTPB, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return b;
}
}  // namespace

cudaError_t launch_sym_check(const int32_t *active, int64_t n, int64_t off, int *gate, cudaStream_t st) {
    k_sym_check<<<(unsigned)cdiv(n, 256), 256, 0, st>>>(active, n, off, gate);
    return cudaGetLastError();
}
cudaError_t launch_sym(const Dev &d, int mode, const SymLaunch &L, int grid, cudaStream_t st) {
    const bool ex = d.precision == NB_EX;
    switch (mode) {
    case kModeOut: return ex ? go<NB_EX, kModeOut>(d, L, grid, st) : go<NB_FP64, kModeOut>(d, L, grid, st);
    case kModeOut4: return ex ? go<NB_EX, kModeOut4>(d, L, grid, st) : go<NB_FP64, kModeOut4>(d, L, grid, st);
    case kModeInit1: return ex ? go<NB_EX, kModeInit1>(d, L, grid, st) : go<NB_FP64, kModeInit1>(d, L, grid, st);
    case kModeInit2: return ex ? go<NB_EX, kModeInit2>(d, L, grid, st) : go<NB_FP64, kModeInit2>(d, L, grid, st);
    case kModeInit4: return ex ? go<NB_EX, kModeInit4>(d, L, grid, st) : go<NB_FP64, kModeInit4>(d, L, grid, st);
    case kModePot: return go<kPrecPot, kModePot>(d, L, grid, st);
    default: return cudaErrorInvalidValue;
    }
}
int sym_values(int mode) { return mode == kModePot ? 1 : (uses_order4_terms(mode) ? 7 : 10); }
int sym_resident(int precision, int mode) {
    if (mode == kModePot) return resident<kPrecPot, kModePot>();
    if (precision != NB_FP64 && precision != NB_EX) return 0;
    const bool ex = precision == NB_EX;
    switch (mode) {
    case kModeOut: return ex ? resident<NB_EX, kModeOut>() : resident<NB_FP64, kModeOut>();
    case kModeOut4: return ex ? resident<NB_EX, kModeOut4>() : resident<NB_FP64, kModeOut4>();
    case kModeInit1: return ex ? resident<NB_EX, kModeInit1>() : resident<NB_FP64, kModeInit1>();
    case kModeInit2: return ex ? resident<NB_EX, kModeInit2>() : resident<NB_FP64, kModeInit2>();
    case kModeInit4: return ex ? resident<NB_EX, kModeInit4>() : resident<NB_FP64, kModeInit4>();
    default: return 0;
    }
}

}  // namespace nb
