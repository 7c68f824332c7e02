// nb_internal.cuh -- device-side data structures and primitives of libnb.
//
// Everything here is internal to the CUDA library; the public boundary is
// include/nb.h.  Sm_103a only.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/nb.h"
#include "nb_fixed.cuh"

namespace nb {

// ---------------------------------------------------------------- constants
#ifndef NB_EVAL_TPB
#define NB_EVAL_TPB 128       // threads per evaluation CTA
#endif
constexpr int kTPB = NB_EVAL_TPB;
constexpr int kTJ = 64;        // j-particles per shared-memory tile
// the whole-cluster evaluation's rows are two columns (nb_sym.cuh), its CTAs one row
static_assert(kTPB == 2 * kTJ, "evaluation CTA: 128 threads");
#ifndef NB_EVAL_STAGES
#define NB_EVAL_STAGES 4
#endif
#ifndef NB_EVAL_MIN_BLOCKS
#define NB_EVAL_MIN_BLOCKS 4  // resident evaluation CTAs per SM the compiler must allow
#endif
#ifndef NB_EVAL_UNROLL
#define NB_EVAL_UNROLL 2      // j-loop unrolling of the FP32 evaluation
#endif
#ifndef NB_EX_LAZY
// 1: the EX evaluation keeps its sums and intermediate products unnormalised
// (hi + lo with every error term kept; sums renormalised once per j-tile).
// Measured: 1.126x the pair rate at N = 65536, and the same maximum errors
// against FP64 at N = 2^20 (Kroupa masses, eps = 1e-5) to two digits.
#define NB_EX_LAZY 1
#endif
// FP32 evaluation: its own ring depth, residency and place of the FP64
// chunk totals (registers, or shared memory when NB_FP32_T64_SMEM)
#ifndef NB_FP32_STAGES
#define NB_FP32_STAGES NB_EVAL_STAGES
#endif
#ifndef NB_FP32_MIN_BLOCKS
#define NB_FP32_MIN_BLOCKS NB_EVAL_MIN_BLOCKS
#endif
#ifndef NB_EX_MIN_BLOCKS
#define NB_EX_MIN_BLOCKS NB_EVAL_MIN_BLOCKS
#endif
#ifndef NB_FP32X_MIN_BLOCKS
#define NB_FP32X_MIN_BLOCKS NB_EVAL_MIN_BLOCKS
#endif
#ifndef NB_EX4_MIN_BLOCKS
#define NB_EX4_MIN_BLOCKS 3
#endif
#ifndef NB_FP32_T64_SMEM
#define NB_FP32_T64_SMEM 1
#endif
constexpr int kStages = NB_EVAL_STAGES;  // TMA pipeline depth
constexpr int kEvalUnroll = NB_EVAL_UNROLL;
constexpr int kChunk = 2048;   // particles per select / predict chunk
constexpr int kSelTPB = 256;   // threads per select CTA
constexpr int kPredTPB = 64;   // threads per predict CTA
constexpr int kPlanTPB = 1024; // threads of the single planning CTA
constexpr int kGrpStride = 160;  // doubles of partial sums per group counter (nb_eval.cuh)
constexpr int kBuckets = 32;   // active-set size buckets (floor log2 A)
constexpr int kFp32FlushTiles = 32;  // FP32 path: j-tiles summed in FP32 before
                                     // promotion to FP64 (32 x 64 = 2048 j)

// device error word bits
constexpr uint32_t kErrNonFinite = 1u;
constexpr uint32_t kErrTimeout = 2u;
constexpr uint32_t kErrIndex = 4u;   // a caller-given index outside its cluster

// wait budget of a bounded device-side wait, nanoseconds
constexpr unsigned long long kWaitBudgetNs = 2000000000ull;

// Tag of the potential-only evaluation (FP64, energy diagnostics) beside the
// nb_precision values.
constexpr int kPrecPot = 64;

// ------------------------------------------------------------ packed j-data
// FP64 values (energy diagnostics, nb_predict's output): x, y, z, m, vx, vy,
// vz, ax, ay, az as five 16-byte pairs.
struct alignas(16) J64 {
    double2 q[5];  // (x,y) (z,m) (vx,vy) (vz,ax) (ay,az)
};
// FP64 evaluation: the position as doubles (none -0, nb_fixed.cuh), velocity and
// acceleration as integers with an exponent field each (FxP3), the mass as a
// 63-bit integer (|m| = mm 2^(em - 62)) and as a float pair.  112 bytes: lanes
// that share an i read records side by side, eight of them in different banks.
struct alignas(16) JFX {
    double x[3];
    uint64_t mm;
    int64_t v[3], a[3];
    float2 mf;      // (m_hi, m_lo) for the potential
    uint32_t f[3];  // exponent fields, two in a word: vx vy, vz ax, ay az
    int32_t ems;    // 2 em + (m < 0)
};
static_assert(sizeof(JFX) == 112, "JFX layout");
__device__ __forceinline__ int jfx_em(const JFX &j) { return j.ems >> 1; }
__device__ __forceinline__ uint32_t jfx_sign(const JFX &j) { return (uint32_t)j.ems << 31; }
__device__ __forceinline__ FxP3 jfx_v(const JFX &j) {
    return FxP3{{j.v[0], j.v[1], j.v[2]},
                {(int)(j.f[0] & 0xffffu), (int)(j.f[0] >> 16), (int)(j.f[1] & 0xffffu)}};
}
__device__ __forceinline__ FxP3 jfx_a(const JFX &j) {
    return FxP3{{j.a[0], j.a[1], j.a[2]},
                {(int)(j.f[1] >> 16), (int)(j.f[2] & 0xffffu), (int)(j.f[2] >> 16)}};
}
__device__ __forceinline__ JFX jfx_pack(const double x[3], const double v[3], const double a[3],
                                        double m) {
    JFX w;
    const FxP3 pv = fx_pack_components(v), pa = fx_pack_components(a);
    for (int k = 0; k < 3; ++k) {
        w.x[k] = x[k] + 0.0;  // -0 + 0 = +0
        w.v[k] = pv.w[k];
        w.a[k] = pa.w[k];
    }
    w.f[0] = (uint32_t)pv.f[0] | ((uint32_t)pv.f[1] << 16);
    w.f[1] = (uint32_t)pv.f[2] | ((uint32_t)pa.f[0] << 16);
    w.f[2] = (uint32_t)pa.f[1] | ((uint32_t)pa.f[2] << 16);
    int em;
    uint32_t sign;
    fx_pack_mass(m, w.mm, em, sign);
    const float hi = (float)m;
    w.mf = make_float2(hi, (float)(m - (double)hi));
    w.ems = 2 * em + (int32_t)(sign >> 31);
    return w;
}
// EX and FP32X: records of two particles whose values interleave like the FP32
// records below: value f of lane l of a record is its float 2 f + l, f in the
// order
//   xh, yh, zh, mh, xl, yl, zl, ml, vxh, vyh, vzh, axh, vxl, vyl, vzl, axl,
//   ayh, azh, ayl, azl
// so q[k] of a record holds (value 2k of lanes 0, 1; value 2k + 1 of lanes 0, 1).
// The last 16 bytes are padding: lanes that share an i read records side by
// side, and at a stride of 176 bytes eight of them meet 32 different banks (at
// 160 bytes pairs of them collide).
struct alignas(16) JEXP {  // a record of two particles
    float4 q[11];
};
constexpr int kJEXVals = 20;
// FP32: records of two particles whose values interleave, so that one 16-byte
// shared-memory load gives two two-lane operands of the packed FP32
// arithmetic.  Value f of lane l (the particle's index parity) of a record is
// its float 2 f + l, f in the order
// xh, yh, zh, m, xl, yl, zl, ax, vxh, vyh, vzh, ay, vxl, vyl, vzl, az:
//   q[0] = (xh0, xh1, yh0, yh1)  q[1] = (zh0, zh1, m0, m1)
//   q[2] = (xl0, xl1, yl0, yl1)  q[3] = (zl0, zl1, ax0, ax1)
//   q[4] = (vxh0, vxh1, vyh0, vyh1)  q[5] = (vzh0, vzh1, ay0, ay1)
//   q[6] = (vxl0, vxl1, vyl0, vyl1)  q[7] = (vzl0, vzl1, az0, az1)
// and 16 bytes of padding: at 128 bytes every record of a warp's lanes starts
// in the same bank (8 lanes an i: 8-fold conflicts; FP32, N = 16384, A = 1000:
// 240 us, with the padding 66 us).
struct alignas(16) J32P {  // a record of two particles
    float4 q[9];
};
constexpr int kJ32Vals = 16;
// Write particle jx's NV values (the orders above) into an array of
// two-particle records Rec (FP32: NV = 16, EX: NV = 20).
template <class Rec, int NV>
__device__ __forceinline__ void jpair_store(void *jarr, int64_t jx, const float v[NV]) {
    float *p = reinterpret_cast<float *>(reinterpret_cast<Rec *>(jarr) + (jx >> 1)) + (jx & 1);
#pragma unroll
    for (int f = 0; f < NV; ++f) p[2 * f] = v[f];
}

// ------------------------------------------------------------ planning data
struct ClusterPlan {
    int32_t gl;     // lanes cooperating on one i (1..32, power of two)
    int32_t split;  // number of j-ranges (S)
    int32_t tiles;  // i-tiles of kTPB / gl active particles
    int32_t active; // A for this step (0: idle)
    int64_t item0;  // first work item of the cluster
    int64_t tile0;  // first i-tile of the cluster (counter index)
    int64_t pslot0; // first partial-sum double (only clusters with split > 1 use them)
    int32_t streamk; // 1: single-cluster launch split stream-K style (split unused)
    int32_t pad_;
};

struct PlanEntry {  // per active-set bucket
    int32_t gl;
    int32_t target_items;  // desired work items per evaluation
};

// Everything a kernel needs, passed by value.
struct Dev {
    int64_t n;
    int32_t n_clusters;
    int32_t n_chunks;
    int32_t precision;
    int32_t grid_eval;  // persistent evaluation grid (CTAs)
    const int64_t *offsets;      // [nc+1] particle offsets
    const int64_t *jofs;         // [nc+1] padded j-array offsets
    const int32_t *chunk_cluster;// [n_chunks]
    const int64_t *chunk_begin;  // [n_chunks]
    const int64_t *chunk_end;    // [n_chunks]
    const int32_t *cluster_chunk0;  // [nc+1]
    // state (caller-owned), SoA [3][n]
    double *m, *x, *v, *a, *j, *s, *c, *t, *dt, *pot;
    // predicted j-arrays
    void *jarr;        // precision-specific (JFX / JEXP (EX, FP32X) / J32P)
    J64 *jarr64;       // FP64 copy (energy, nb_predict output)
    // select
    double *chunk_min;
    int32_t *chunk_cnt;
    double *tnext;     // [nc]
    int32_t *nact;     // [nc]
    int32_t *active;   // [n], cluster c's list at offsets[c]
    // plan
    ClusterPlan *plan; // [nc]
    int64_t *n_items;  // [1]
    unsigned long long *item_ctr;  // [1]: next work item (dynamic fetch), reset by k_plan
    const PlanEntry *table;  // [kBuckets]
    // reduction scratch
    double *partial;   // [max_items][10][kTPB]
    int64_t partial_cap;     // capacity in doubles (an item of Ti i's uses 10 Ti)
    int32_t *tile_cnt; // [max_tiles]
    // counters / flags
    unsigned long long *ctr_steps;
    double *ctr_inter;
    unsigned long long *ctr_underflow;
    uint32_t *err;
    int32_t *busy;     // [1]: clusters active in the last select
    double *t_end;     // [1]: clusters whose next block time exceeds it stay idle
    double *pot_tmp;   // [n] energy potential
    double *energy_part;  // [blocks][8]
    // parameters
    double eps2, eta, eta_init, dt_min, dt_max;
    // -1.0 as a run-time value: a - b = b*(-1) + a issued as an FMA, which
    // compilers cannot fold back (DADD runs at 84 % of the DFMA rate)
    double neg_one;
    // 6: NM08 6th order; 4: Makino & Aarseth 4th order.  Kept last: inserting
    // it among the fields above measured 2.8 % slower FP64 evaluation.
    int32_t order;
    int32_t streamk_off;  // NB_NO_STREAMK
    unsigned int *sel_ctr;  // [1]: chunks done in select pass 1 (the last one finishes the pass)
    // eps^2 as a float-float pair, both lanes equal: hi = fl(eps^2),
    // lo = fl(eps^2 - hi).  Formed on the host: the single-precision kernels
    // read them as parameters, where converting eps2 in the kernel costs
    // FP64-pipe conversions wherever the compiler re-forms the values.
    float2 eps2_hi2, eps2_lo2;
    // eps^2 = eps_x 2^(2 E - 58), eps_x in [2^58, 2^60], and its block's
    // exponent field (E + 1023) << 20 (nb_fixed.cuh); both 0 for eps = 0
    uint64_t eps_x;
    uint32_t eps_emin;
    FxK fxk;  // {1, 2} as run-time values (nb_fixed.cuh)
    int32_t *grp_cnt;  // [partial_cap / kGrpStride + 1]: pieces of a group done
    // several clusters: the active ones by first item (unused: INT64_MAX)
    int64_t *order_item0;    // [nc]
    int32_t *order_cluster;  // [nc]
};

// The small values host and device exchange, in one block: the host reads it
// with one copy.
struct Ctl {
    double t_end;       // clusters whose next block time exceeds it stay idle
    int32_t busy;       // clusters active in the last plan, or whether a step is due
    uint32_t err;       // device error word
    unsigned long long steps, underflow;  // counters
    double inter;
};

// eps^2 and its float-float pair (host side; every context and launch).
inline void set_eps2(Dev &d, double eps) {
    d.eps2 = eps * eps;
    const float hi = (float)d.eps2;
    const float lo = (float)(d.eps2 - (double)hi);
    d.eps2_hi2 = make_float2(hi, hi);
    d.eps2_lo2 = make_float2(lo, lo);
    fx_eps2(d.eps2, d.eps_x, d.eps_emin);
    d.fxk = FxK{1, 2};
}

// How one evaluation launch obtains its work.
struct EvalLaunch {
    int32_t direct;     // 1: single cluster, host-given list / plan
    int32_t cluster;    // direct mode
    int32_t n_active;   // direct mode
    int32_t gl;         // direct mode
    int32_t split;      // direct mode
    int32_t tiles;      // direct mode
    int32_t identity;   // active list is 0..A-1 of the cluster (init, energy)
    const int32_t *active;  // direct mode list (global indices)
    double *out;        // direct mode output [10][n_active]
    int32_t streamk;    // direct mode: stream-K ranges instead of split items
    int32_t jt0, jt1;   // direct mode: j-tiles [jt0, jt1) of the cluster (jt1 = 0: all)
    const int *gate;    // run only while *gate != 0 (NULL: always)
};

// Out/Step/Init1/Init2: 6th-order pair terms (a, jerk, snap); the *4 modes
// evaluate the 4th-order terms (a, jerk; snap slots stay 0); Pot: potential.
enum EvalMode {
    kModeOut = 0, kModeStep = 1, kModeInit1 = 2, kModeInit2 = 3, kModePot = 4,
    kModeOut4 = 5, kModeStep4 = 6, kModeInit4 = 7
};
constexpr bool is_order4_mode(int mode) { return mode >= kModeOut4; }
// Modes that sum only acceleration, jerk and potential (the 4th-order pair
// terms): the 4th-order modes, and the first start-up pass of the 6th-order
// scheme, whose only output that survives is the acceleration (pass 2 needs
// it for the relative accelerations; it recomputes a and jerk with snap).
constexpr bool uses_order4_terms(int mode) { return is_order4_mode(mode) || mode == kModeInit1; }

// ---------------------------------------------------------- small helpers
__host__ __device__ inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

constexpr int kMinTilesPerItem = 4;  // a j-range holds at least 4 x 64 j (FP64: 64, split_max)

// Stream-K decomposition of a single cluster's evaluation.  Its work is
// U = tiles x ntj units (one i-tile against one j-tile, all of equal cost);
// CTA k of G takes the contiguous unit range [U k / G, U (k+1) / G), so every
// CTA (and every SM) gets the same work to within one unit.  A range splits
// at i-tile boundaries into pieces; an i-tile covered by several CTAs gets one
// partial sum per CTA, added in CTA order by the last one to finish.
#ifndef NB_STREAMK
#define NB_STREAMK 1
#endif
#ifndef NB_STREAMK_MIN_UNITS
#define NB_STREAMK_MIN_UNITS 4
#endif
constexpr int kStreamKMinUnits = NB_STREAMK_MIN_UNITS;  // units per CTA below which splits are used
__host__ __device__ inline int64_t sk_begin(int64_t U, int64_t G, int64_t k) { return U * k / G; }
// CTA whose range holds unit p (the largest k with sk_begin(k) <= p; U >= G)
__host__ __device__ inline int64_t sk_owner(int64_t U, int64_t G, int64_t p) {
    return ((p + 1) * G + U - 1) / U - 1;
}
// most i-tiles one CTA's range can touch
__host__ __device__ inline int64_t sk_max_pieces(int64_t U, int64_t G, int64_t ntj) {
    return (cdiv(U, G) - 1) / ntj + 2;
}
// whether a launch of `tiles` i-tiles of Ti i's over ntj j-tiles on G CTAs
// runs stream-K: enough units per CTA, partial sums within the scratch
__host__ __device__ inline bool sk_use(int64_t tiles, int64_t Ti, int64_t ntj, int64_t G,
                                       int64_t partial_cap) {
    if (!NB_STREAMK || tiles <= 0) return false;
    const int64_t U = tiles * ntj;
    if (U < kStreamKMinUnits * G) return false;
    return G * sk_max_pieces(U, G, ntj) * 10 * Ti <= partial_cap;
}

// Lanes per i of a single cluster's launch: the table's choice for the
// active-set size, doubled (FP64, EX) while the launch has fewer units than
// stream-K wants (few active particles, or a small cluster).  EX pairs cost
// less: it doubles only where an even share still gives every lane of the grid
// eight pairs; below that the epilogue of the extra pieces costs more than the
// idle SMs.  FP32 and FP32X keep the table's lanes: the order of their single
// precision sums, and with it their rounding, follows the lanes.  Measured (us,
// one evaluation, table's lanes -> these): N = A = 1024 FP64 128 -> 59, EX 59 ->
// 47; N = A = 256 FP64 64 -> 15.
__host__ __device__ constexpr int sk_min_pairs(int precision) { return precision == NB_FP64 ? 0 : 8; }
// Units per CTA that the doubling aims at: with FP64's costly units a finer cut
// still pays (block steps of N = 16384: 24.04 -> 23.90 ms with 8 instead of 4).
__host__ __device__ constexpr int64_t sk_lane_units(int precision) {
    return precision == NB_FP64 ? 2 * kStreamKMinUnits : kStreamKMinUnits;
}
__host__ __device__ inline int sk_lanes(int gl, int64_t A, int64_t ntj, int64_t G, int precision) {
    if (precision != NB_FP64 && precision != NB_EX) return gl;
    if (A * ntj * kTJ < (int64_t)sk_min_pairs(precision) * G * kTPB) return gl;
    while (gl < 32 && cdiv(A, kTPB / gl) * ntj < sk_lane_units(precision) * G) gl *= 2;
    return gl;
}
// Most j-ranges a launch is split into: at least kMinTilesPerItem j-tiles
// each; the FP64 terms, whose pairs cost most, go down to one tile while that
// makes no more than 128 ranges.  Measured (us, FP64, N = 1024, A = 1): 20 ->
// 14; N = 16384, A = 4: 24.7 with at most 64 ranges, 22.7 with 128, 29 with 256.
__host__ __device__ inline int64_t split_max(int64_t ntj, int precision) {
    const int64_t s = ntj / kMinTilesPerItem > 1 ? ntj / kMinTilesPerItem : 1;
    const int64_t fine = ntj < 128 ? ntj : 128;
    return precision == NB_FP64 && s < fine ? fine : s;
}

// Number of j-ranges (split S) for `tiles` i-tiles over a cluster of `ntj`
// j-tiles.  Start from the bucket's target item count; make at most split_max
// ranges; for `grid` resident CTAs, take the
// smallest S in [S0/2, 2 S0] whose items fill the largest fraction of whole
// waves (equal-cost items: a last, partly filled wave leaves SMs idle).  The
// result depends on this cluster alone, so a cluster's plan (and therefore
// its rounding) is the same in a batch as on its own.
__host__ __device__ inline int64_t choose_split(int64_t tiles, int64_t ntj, int64_t target,
                                                int64_t grid, int precision = NB_EX) {
    const int64_t smax = split_max(ntj, precision);
    int64_t s0 = cdiv(target, tiles > 0 ? tiles : 1);
    s0 = s0 < 1 ? 1 : (s0 > smax ? smax : s0);
    if (grid <= 0) return s0;
    // efficiency items / (waves * grid), compared by cross-multiplication in
    // integers.  Within one wave count w the efficiency grows with S, so only
    // the largest S of each w can win: visit the wave counts of the window
    // (a few) instead of every S (a few hundred 64-bit divisions in the
    // planner's single thread); stepping w upwards and keeping only strict
    // improvements returns the smallest S of the best efficiency.
    int64_t best = s0, best_items = 0, best_slots = 1;
    const int64_t lo = s0 / 2 > 1 ? s0 / 2 : 1;
    const int64_t hi = 2 * s0 < smax ? 2 * s0 : smax;
    const int64_t t = tiles > 0 ? tiles : 1;
    const int64_t w_lo = cdiv(t * lo, grid), w_hi = cdiv(t * hi, grid);
    for (int64_t w = w_lo; w <= w_hi; ++w) {
        int64_t s = (w * grid) / t;  // the largest S with t S <= w grid
        s = s > hi ? hi : s;
        if (s < lo || t * s <= (w - 1) * grid) continue;  // no S of the window fills w waves
        const int64_t items = t * s, slots = w * grid;
        if (items * best_slots > best_items * slots) {
            best_items = items;
            best_slots = slots;
            best = s;
        }
    }
    return best;
}

// How an evaluation of A active particles over ntj j-tiles is launched, from its
// bucket's table entry: in the planner of the steps, for the host-planned
// evaluations, and in the autotuner, which times what the planner will run and
// stores lanes that this gives back unchanged.  streamk: the launch may use
// stream-K ranges (one cluster, NB_NO_STREAMK not set); otherwise the entry's lanes
// and split items, the same alone and in a batch.
struct EvalPlan {
    int32_t gl, split, tiles, streamk;
};
__host__ __device__ inline EvalPlan plan_eval(PlanEntry e, int64_t A, int64_t ntj, bool streamk, int64_t grid,
                                              int64_t partial_cap, int precision) {
    EvalPlan p;
    p.gl = streamk ? sk_lanes(e.gl, A, ntj, grid, precision) : e.gl;
    const int64_t tiles = cdiv(A, kTPB / p.gl);
    p.tiles = (int32_t)tiles;
    p.streamk = streamk && sk_use(tiles, kTPB / p.gl, ntj, grid, partial_cap) ? 1 : 0;
    p.split = p.streamk ? 1 : (int32_t)choose_split(tiles, ntj, e.target_items, grid, precision);
    return p;
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// ---------------------------------------------------------------- FP64 rsqrt
__device__ __forceinline__ double fma_rn_f64(double a, double b, double c) {
    double r;
    asm("fma.rn.f64 %0, %1, %2, %3;" : "=d"(r) : "d"(a), "d"(b), "d"(c));
    return r;
}
// SFU approximation of 1/sqrt (rsqrt.approx.ftz.f32), per lane for float2.
__device__ __forceinline__ float rsqrt_sfu(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 rsqrt_sfu(float2 x) {
    return make_float2(rsqrt_sfu(x.x), rsqrt_sfu(x.y));
}
// --------------------------------------------- packed two-lane FP32 (f32x2)
// sm_100 and later execute FP32 add / multiply / FMA on a pair of floats in
// one instruction (PTX add/sub/mul/fma.rn.f32x2): the same per-lane IEEE
// round-to-nearest results as the scalar instructions, half the issue slots.
__device__ __forceinline__ float2 f2s(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 ta, tb, tr;\n\tmov.b64 ta, {%2, %3};\n\tmov.b64 tb, {%4, %5};\n\t"
        "sub.rn.f32x2 tr, ta, tb;\n\tmov.b64 {%0, %1}, tr;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 lo2(float4 q) { return make_float2(q.x, q.y); }
__device__ __forceinline__ float2 hi2(float4 q) { return make_float2(q.z, q.w); }

// ------------------------------------------------------- float-float (EX)
// A value is hi + lo with |lo| <= ulp(hi)/2 (Dekker 1971; Knuth TAOCP 2;
// Hida, Li & Bailey 2001 for the double-double algorithms, here on floats).
// Every primitive is written once for a lane type T: float (one value) or
// float2 (two independent values, one per lane, each with the IEEE results
// of the float form, evaluated by the packed f32x2 instructions).
template <class T>
struct ffT {
    T hi, lo;
};
using ff = ffT<float>;
using ff2 = ffT<float2>;

__device__ __forceinline__ float o_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float o_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float o_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float o_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float o_neg(float a) { return -a; }
__device__ __forceinline__ float o_cst(float, float c) { return c; }
__device__ __forceinline__ float2 o_add(float2 a, float2 b) { return add2(a, b); }
__device__ __forceinline__ float2 o_sub(float2 a, float2 b) { return sub2(a, b); }
__device__ __forceinline__ float2 o_mul(float2 a, float2 b) { return mul2(a, b); }
__device__ __forceinline__ float2 o_fma(float2 a, float2 b, float2 c) { return fma2(a, b, c); }
__device__ __forceinline__ float2 o_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 o_cst(float2, float c) { return f2s(c); }

// exact: s + e = a + b (Knuth TwoSum)
template <class T>
__device__ __forceinline__ void two_sum(T a, T b, T &s, T &e) {
    s = o_add(a, b);
    const T bb = o_sub(s, a);
    e = o_add(o_sub(a, o_sub(s, bb)), o_sub(b, bb));
}
// exact: s + e = a - b (TwoSum of a and -b, the negation folded in)
template <class T>
__device__ __forceinline__ void two_diff(T a, T b, T &s, T &e) {
    s = o_sub(a, b);
    const T bb = o_sub(s, a);
    e = o_sub(o_sub(a, o_sub(s, bb)), o_add(b, bb));
}
// exact when |a| >= |b| (Dekker FastTwoSum)
template <class T>
__device__ __forceinline__ void fast_two_sum(T a, T b, T &s, T &e) {
    s = o_add(a, b);
    e = o_sub(b, o_sub(s, a));
}
template <class T>
__device__ __forceinline__ ffT<T> ff_renorm(T s, T e) {
    ffT<T> r;
    fast_two_sum(s, e, r.hi, r.lo);
    return r;
}
template <class T>
__device__ __forceinline__ ffT<T> ff_add(ffT<T> a, ffT<T> b) {
    T s, e;
    two_sum(a.hi, b.hi, s, e);
    e = o_add(e, o_add(a.lo, b.lo));
    return ff_renorm(s, e);
}
template <class T>
__device__ __forceinline__ ffT<T> ff_neg(ffT<T> a) { return ffT<T>{o_neg(a.hi), o_neg(a.lo)}; }
// a - b, normalised
template <class T>
__device__ __forceinline__ ffT<T> ff_sub(ffT<T> a, ffT<T> b) {
    T s, e;
    two_diff(a.hi, b.hi, s, e);
    e = o_add(e, o_sub(a.lo, b.lo));
    return ff_renorm(s, e);
}
// product, error terms folded with FMA (Dekker TwoProduct via FMA)
template <class T>
__device__ __forceinline__ ffT<T> ff_mul(ffT<T> a, ffT<T> b) {
    const T p = o_mul(a.hi, b.hi);
    T e = o_fma(a.hi, b.hi, o_neg(p));
    e = o_fma(a.hi, b.lo, e);
    e = o_fma(a.lo, b.hi, e);
    return ff_renorm(p, e);
}
template <class T>
__device__ __forceinline__ ffT<T> ff_mul_f(ffT<T> a, T b) {
    const T p = o_mul(a.hi, b);
    T e = o_fma(a.hi, b, o_neg(p));
    e = o_fma(a.lo, b, e);
    return ff_renorm(p, e);
}
template <class T>
__device__ __forceinline__ ffT<T> ff_sqr(ffT<T> a) {
    const T p = o_mul(a.hi, a.hi);
    T e = o_fma(a.hi, a.hi, o_neg(p));
    e = o_fma(o_add(a.hi, a.hi), a.lo, e);
    return ff_renorm(p, e);
}
// acc += a * b, product and sum kept exact to float-float accuracy
template <class T>
__device__ __forceinline__ void ff_fma_acc(ffT<T> &acc, ffT<T> a, ffT<T> b) {
    const T p = o_mul(a.hi, b.hi);
    T pe = o_fma(a.hi, b.hi, o_neg(p));
    pe = o_fma(a.hi, b.lo, pe);
    pe = o_fma(a.lo, b.hi, pe);
    T s, e;
    two_sum(acc.hi, p, s, e);
    e = o_add(e, o_add(acc.lo, pe));
    acc = ff_renorm(s, e);
}
// a - b*c: the product's error terms folded by FMA, one renormalisation
template <class T>
__device__ __forceinline__ ffT<T> ff_fnma(ffT<T> b, ffT<T> c, ffT<T> a) {
    const T p = o_mul(b.hi, c.hi);
    T pe = o_fma(b.hi, c.hi, o_neg(p));
    pe = o_fma(b.hi, c.lo, pe);
    pe = o_fma(b.lo, c.hi, pe);
    T s, e;
    two_diff(a.hi, p, s, e);
    e = o_add(e, o_sub(a.lo, pe));
    return ff_renorm(s, e);
}
// dot products: high parts summed with exact TwoSum, all second-order terms
// gathered in one value, one renormalisation at the end.
template <class T>
__device__ __forceinline__ ffT<T> ff_dot3(const ffT<T> a[3], const ffT<T> b[3]) {
    T p0 = o_mul(a[0].hi, b[0].hi), p1 = o_mul(a[1].hi, b[1].hi), p2 = o_mul(a[2].hi, b[2].hi);
    T lo = o_fma(a[0].hi, b[0].hi, o_neg(p0));
    lo = o_add(o_fma(a[1].hi, b[1].hi, o_neg(p1)), lo);
    lo = o_add(o_fma(a[2].hi, b[2].hi, o_neg(p2)), lo);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo = o_fma(a[k].hi, b[k].lo, lo);
        lo = o_fma(a[k].lo, b[k].hi, lo);
    }
    T s, e;
    two_sum(p0, p1, s, e);
    lo = o_add(lo, e);
    two_sum(s, p2, s, e);
    lo = o_add(lo, e);
    return ff_renorm(s, lo);
}

// Lazy forms: the sum's high part takes the exact TwoSum, the low part
// gathers every error term, and renormalisation is left to the caller (once
// per j-tile for accumulators).  |lo| may reach a few ulps of |hi|; every
// consumer below folds lo into first-order terms only.
template <class T>
__device__ __forceinline__ void ff_fma_acc_lazy(ffT<T> &acc, ffT<T> a, ffT<T> b) {
    const T p = o_mul(a.hi, b.hi);
    T pe = o_fma(a.hi, b.hi, o_neg(p));
    pe = o_fma(a.hi, b.lo, pe);
    pe = o_fma(a.lo, b.hi, pe);
    T s, e;
    two_sum(acc.hi, p, s, e);
    acc.hi = s;
    acc.lo = o_add(acc.lo, o_add(e, pe));
}
template <class T>
__device__ __forceinline__ ffT<T> ff_mul_lazy(ffT<T> a, ffT<T> b) {
    const T p = o_mul(a.hi, b.hi);
    T e = o_fma(a.hi, b.hi, o_neg(p));
    e = o_fma(a.hi, b.lo, e);
    e = o_fma(a.lo, b.hi, e);
    return ffT<T>{p, e};
}
template <class T>
__device__ __forceinline__ ffT<T> ff_mul_f_lazy(ffT<T> a, T b) {
    const T p = o_mul(a.hi, b);
    T e = o_fma(a.hi, b, o_neg(p));
    e = o_fma(a.lo, b, e);
    return ffT<T>{p, e};
}
template <class T>
__device__ __forceinline__ ffT<T> ff_sqr_lazy(ffT<T> a) {
    const T p = o_mul(a.hi, a.hi);
    T e = o_fma(a.hi, a.hi, o_neg(p));
    e = o_fma(o_add(a.hi, a.hi), a.lo, e);
    return ffT<T>{p, e};
}
template <class T>
__device__ __forceinline__ ffT<T> ff_sum_lazy(ffT<T> a, ffT<T> b) {
    T s, e;
    two_sum(a.hi, b.hi, s, e);
    return ffT<T>{s, o_add(e, o_add(a.lo, b.lo))};
}
template <class T>
__device__ __forceinline__ void ff_add_lazy(ffT<T> &acc, ffT<T> b) {
    T s, e;
    two_sum(acc.hi, b.hi, s, e);
    acc.hi = s;
    acc.lo = o_add(acc.lo, o_add(e, b.lo));
}
template <class T>
__device__ __forceinline__ ffT<T> ff_fnma_lazy(ffT<T> b, ffT<T> c, ffT<T> a) {
    const T p = o_mul(b.hi, c.hi);
    T pe = o_fma(b.hi, c.hi, o_neg(p));
    pe = o_fma(b.hi, c.lo, pe);
    pe = o_fma(b.lo, c.hi, pe);
    T s, e;
    two_diff(a.hi, p, s, e);
    return ffT<T>{s, o_add(e, o_sub(a.lo, pe))};
}
// 1/sqrt(r2) in float-float: SFU seed y0, residual e = 1 - r2 y0^2 from the
// exact square of y0 and FMA-exact products, then y0 (1 + e/2 + 3e^2/8).
// Lazy form: y0 + corr as it is (|corr| ~ 2^-22 |y0|).  Domain: the normal
// FP32 range of r2.hi.
template <class T>
__device__ __forceinline__ ffT<T> rsqrt_ff(ffT<T> r2) {
    const T y0 = rsqrt_sfu(r2.hi);
    const T p = o_mul(y0, y0);
    const T pe = o_fma(y0, y0, o_neg(p));
    const T u = o_mul(r2.hi, p);
    T ue = o_fma(r2.hi, p, o_neg(u));
    ue = o_fma(r2.hi, pe, ue);
    ue = o_fma(r2.lo, p, ue);
    const T e = o_sub(o_sub(o_cst(y0, 1.0f), u), ue);
    const T corr = o_mul(o_mul(y0, e), o_fma(e, o_cst(y0, 0.375f), o_cst(y0, 0.5f)));
    if constexpr (NB_EX_LAZY) return ffT<T>{y0, corr};
    else return ff_renorm(y0, corr);
}

// a.b, unnormalised (hi + lo with every error term in lo)
template <class T>
__device__ __forceinline__ ffT<T> ff_dot3_lazy(const ffT<T> a[3], const ffT<T> b[3]) {
    T p[3], lo;
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k] = o_mul(a[k].hi, b[k].hi);
    lo = o_fma(a[0].hi, b[0].hi, o_neg(p[0]));
#pragma unroll
    for (int k = 1; k < 3; ++k) lo = o_add(o_fma(a[k].hi, b[k].hi, o_neg(p[k])), lo);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo = o_fma(a[k].hi, b[k].lo, lo);
        lo = o_fma(a[k].lo, b[k].hi, lo);
    }
    T s = p[0], e;
#pragma unroll
    for (int k = 1; k < 3; ++k) {
        two_sum(s, p[k], s, e);
        lo = o_add(lo, e);
    }
    return ffT<T>{s, lo};
}
// a0.b0 + a1.b1, unnormalised
template <class T>
__device__ __forceinline__ ffT<T> ff_dot3x2_lazy(const ffT<T> a0[3], const ffT<T> b0[3],
                                                 const ffT<T> a1[3], const ffT<T> b1[3]) {
    T p[6];
    T lo = o_cst(a0[0].hi, 0.f);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[k] = o_mul(a0[k].hi, b0[k].hi);
        p[3 + k] = o_mul(a1[k].hi, b1[k].hi);
        lo = o_add(o_fma(a0[k].hi, b0[k].hi, o_neg(p[k])), lo);
        lo = o_add(o_fma(a1[k].hi, b1[k].hi, o_neg(p[3 + k])), lo);
        lo = o_fma(a0[k].hi, b0[k].lo, lo);
        lo = o_fma(a0[k].lo, b0[k].hi, lo);
        lo = o_fma(a1[k].hi, b1[k].lo, lo);
        lo = o_fma(a1[k].lo, b1[k].hi, lo);
    }
    T s = p[0], e;
#pragma unroll
    for (int k = 1; k < 6; ++k) {
        two_sum(s, p[k], s, e);
        lo = o_add(lo, e);
    }
    return ffT<T>{s, lo};
}
// a.b + c, unnormalised
template <class T>
__device__ __forceinline__ ffT<T> ff_dot3_add_lazy(const ffT<T> a[3], const ffT<T> b[3], ffT<T> c) {
    T p[3], lo = c.lo;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[k] = o_mul(a[k].hi, b[k].hi);
        lo = o_add(o_fma(a[k].hi, b[k].hi, o_neg(p[k])), lo);
        lo = o_fma(a[k].hi, b[k].lo, lo);
        lo = o_fma(a[k].lo, b[k].hi, lo);
    }
    T s = c.hi, e;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        two_sum(s, p[k], s, e);
        lo = o_add(lo, e);
    }
    return ffT<T>{s, lo};
}
// a.b + c, one renormalisation
template <class T>
__device__ __forceinline__ ffT<T> ff_dot3_add(const ffT<T> a[3], const ffT<T> b[3], ffT<T> c) {
    const ffT<T> r = ff_dot3_add_lazy(a, b, c);
    return ff_renorm(r.hi, r.lo);
}

// ------------------------------------------------------------ TMA / mbarrier
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
// 1-D bulk copy global -> shared (TMA engine), completion counted in bytes on bar.
// dst, src 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void tma_load_1d(void *dst, const void *src, uint32_t bytes,
                                            uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: false after kWaitBudgetNs without completion.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                                  unsigned long long budget_ns = kWaitBudgetNs) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = globaltimer_ns();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (globaltimer_ns() - t0 > budget_ns) return false;
    }
}

// ------------------------------------------------------------ launchers
// (implemented in the kernel translation units)
cudaError_t launch_select_min(const Dev &d, int look, cudaStream_t st);
cudaError_t launch_select_compact(const Dev &d, double unused, cudaStream_t st);
cudaError_t launch_predict(const Dev &d, int also64, int use_fixed_t, double t_fixed,
                           cudaStream_t st);
cudaError_t launch_pad(const Dev &d, cudaStream_t st);
cudaError_t launch_eval(const Dev &d, int mode, const EvalLaunch &L, int grid, cudaStream_t st);
cudaError_t launch_correct(const Dev &d, int64_t lo, int64_t hi, const int32_t *active,
                           int32_t n_active, double t_next, const double *ajs, cudaStream_t st);
cudaError_t launch_init_clear(const Dev &d, cudaStream_t st);
cudaError_t launch_energy(const Dev &d, int64_t begin, int64_t end, int blocks, cudaStream_t st);
int eval_occupancy(int precision, int mode);  // CTAs per SM

}  // namespace nb
