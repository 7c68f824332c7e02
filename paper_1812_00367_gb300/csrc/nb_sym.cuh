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

// Used from kSymMinUnits units per CTA (below, the triangle's cut is too
// coarse) while the columns' partials fit kSymMaxBytes.
constexpr int64_t kSymMinUnits = 6;
constexpr int64_t kSymMaxBytes = 4000000000ll;
constexpr int64_t kSymUnitBytes = 10 * kTJ * (int64_t)sizeof(double);

struct SymLaunch {
    int32_t cluster;
    int32_t ntj;      // columns
    int64_t n, units;
    double *jpart;    // [units][values][64]
    double *ipart;    // [rows + grid][10][128]; slot row + CTA
    int *gate;        // run only while *gate == 0 (NULL: always)
    int *bad;         // bit 0: a velocity, bit 1: an acceleration is not finite
    double *out;      // mode out: [10][n]
};

cudaError_t launch_sym_check(const int32_t *active, int64_t n, int64_t off, int *gate, cudaStream_t st);
cudaError_t launch_sym(const Dev &d, int mode, const SymLaunch &L, int grid, cudaStream_t st);
int sym_resident(int precision, int mode);  // CTAs per SM (0: not available)

}  // namespace nb
