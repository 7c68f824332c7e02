// nb_sym.cuh -- launch description of the all-active evaluation that takes
// each pair once (nb_sym.cu), and the arithmetic of its units.
#pragma once

#include "nb_internal.cuh"

namespace nb {

// Row I (128 particles) meets the columns (64 particles) 2 I .. ntj - 1.  Units
// are numbered row by row; row I starts at unit sum_{r < I} (ntj - 2 r).
__host__ __device__ inline int64_t sym_first(int64_t row, int64_t ntj) { return row * (ntj + 1 - row); }
__host__ __device__ inline int64_t sym_rows(int64_t ntj) { return (ntj + 1) / 2; }
__host__ __device__ inline int64_t sym_units(int64_t ntj) { return sym_first(sym_rows(ntj), ntj); }
// row of unit u: the largest with sym_first(row) <= u
__host__ __device__ inline int sym_row(int64_t u, int64_t ntj) {
    const double b = (double)(ntj + 1);
    int64_t r = (int64_t)((b - sqrt(b * b - 4.0 * (double)u)) * 0.5);
    r = r < 0 ? 0 : r;
    while (r > 0 && sym_first(r, ntj) > u) --r;
    while (r + 1 < sym_rows(ntj) && sym_first(r + 1, ntj) <= u) ++r;
    return (int)r;
}

// Used from kSymMinUnits units per CTA on (N = 7,800 on a grid of 608), below which
// nb_evaluate of every particle keeps the sums of a block step bit for bit; up to
// kSymMaxUnits units (N = 113,000) for the pair terms, ten times as many (N =
// 357,000) for the potential, the sizes it was tried at.  It would pay from about one
// unit per CTA on (us, each pair once against one-sided; FP64: N = 3000 the same, 4000
// 488 / 628, 6000 944 / 1392, 8000 1560 / 2350, 12000 3395 / 5316; EX: 4000 233 /
// 293, 8000 714 / 995).
constexpr int64_t kSymMinUnits = 6;
constexpr int64_t kSymMaxUnits = 781250;

// Scratch: the evaluation's partial sums (Dev::partial), which nothing else uses
// meanwhile.  The units are taken in bands whose columns' partials fit there: they
// are 64 doubles a unit and value (5 KB, 1.3 GB at N = 65536 for all units at
// once).  Besides them it holds the rows' pieces and, between bands, the sums so
// far.  In doubles, for nv values on a grid of `grid` CTAs:
__host__ __device__ inline int64_t sym_piece_doubles(int64_t ntj, int64_t grid) {
    return (sym_rows(ntj) + grid) * 10 * kTPB;
}
__host__ __device__ inline int64_t sym_sum_doubles(int64_t ntj, int64_t nv) { return ntj * nv * kTJ; }
// Bands (0: the scratch is too small).  Their units are multiples of the grid, but
// for the last one's: a CTA's share of all bands together is then that of one
// launch (bands of whole rows left shares of 55 and 56 units: N = 65536 98.5 against
// 97.9 ms).  Every band has at least as many units as CTAs.
__host__ __device__ inline int64_t sym_bands(int64_t ntj, int64_t grid, int64_t nv, int64_t cap) {
    const int64_t fit = (cap - sym_piece_doubles(ntj, grid) - sym_sum_doubles(ntj, nv)) / (nv * kTJ);
    const int64_t most = fit / grid;  // units a CTA
    return fit < 0 || most < kSymMinUnits ? 0 : cdiv(cdiv(sym_units(ntj), grid), most);
}
// First unit of band b (b = bands: the number of units).
__host__ __device__ inline int64_t sym_band_first(int64_t ntj, int64_t grid, int64_t bands, int64_t b) {
    return b >= bands ? sym_units(ntj) : grid * (cdiv(sym_units(ntj), grid) * b / bands);
}

struct SymLaunch {
    int32_t cluster;
    int32_t ntj;      // columns
    int64_t n;
    int64_t u0, units, row0;  // the band: its first unit, its units, the row of the first
    double *jpart;    // [units of the band][values][64]
    double *ipart;    // [rows + grid][10][128]; slot row - row0 + CTA
    double *sums;     // [ntj][values][64]: what the earlier bands add up to
    int *gate;        // run only while *gate == 0 (NULL: always)
    int *bad;         // bit 0: a velocity, bit 1: an acceleration is not finite
    double *out;      // mode out: [10][n]
};

cudaError_t launch_sym_check(const int32_t *active, int64_t n, int64_t off, int *gate, cudaStream_t st);
// All bands, in the scratch d.partial.  L: cluster, ntj, n, gate, bad, out.
cudaError_t launch_sym(const Dev &d, int mode, const SymLaunch &L, int grid, cudaStream_t st);
int sym_values(int mode);  // values per particle in the partials
int sym_resident(int precision, int mode);  // CTAs per SM (0: not available)

}  // namespace nb
