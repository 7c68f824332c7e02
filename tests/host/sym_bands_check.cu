// sym_bands_check.cu -- host-only checks of the bands of the all-active evaluation
// that takes each pair once (nb_sym.cuh): every unit in one band, the bands inside
// the scratch, every partial written once and read once by the reduction.  Runs on
// the CPU, makes no CUDA call.  Prints "ok <cases>" or the first violation.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../../paper_1812_00367_gb300/csrc/nb_sym.cuh"

using namespace nb;

#define CHECK(cond, ...)                                   \
    do {                                                   \
        if (!(cond)) {                                     \
            std::printf("FAIL %s: ", #cond);               \
            std::printf(__VA_ARGS__);                      \
            std::printf("\n");                             \
            std::exit(1);                                  \
        }                                                  \
    } while (0)

int main() {
    long cases = 0, split = 0;
    for (int64_t G : {152, 456, 608, 1064, 1216, 1368})
        for (int64_t ntj : {121, 128, 157, 300, 365, 366, 470, 1023, 1024, 1025, 1765})
            for (int64_t nv : {1, 7, 10}) {
                const int64_t total = sym_units(ntj);
                if (total < kSymMinUnits * G) continue;
                // the contexts' scratch (456 or more CTAs of the evaluation), and a small one
                for (int64_t cap : {32 * 608 * 10 * (int64_t)kTPB, 32 * 456 * 10 * (int64_t)kTPB, (int64_t)4000000}) {
                    const int64_t bands = sym_bands(ntj, G, nv, cap);
                    if (bands == 0) {
                        CHECK(cap == 4000000, "no room at the contexts' scratch: ntj %lld", (long long)ntj);
                        continue;
                    }
                    split += bands > 1;
                    const int64_t room = cap - sym_piece_doubles(ntj, G) - sym_sum_doubles(ntj, nv);
                    CHECK(sym_band_first(ntj, G, bands, 0) == 0, "first unit");
                    std::vector<int> adds(ntj, 0), last(ntj, 0), pieces(ntj, 0), found(ntj, 0);
                    int64_t share = 0;
                    for (int64_t b = 0; b < bands; ++b) {
                        const int64_t u0 = sym_band_first(ntj, G, bands, b), u1 = sym_band_first(ntj, G, bands, b + 1);
                        const int64_t U = u1 - u0, row0 = sym_row(u0, ntj);
                        CHECK(U >= G && u1 <= total, "units %lld for %lld CTAs", (long long)U, (long long)G);
                        CHECK(U * nv * kTJ <= room, "columns' partials of band %lld", (long long)b);
                        share += cdiv(U, G);
                        CHECK(b + 1 < bands || u1 == total, "last unit");
                        // pieces: one slot each
                        std::vector<int64_t> slot(sym_piece_doubles(ntj, G) / (10 * kTPB), -1);
                        for (int64_t k = 0; k < G; ++k) {
                            int64_t p = u0 + sk_begin(U, G, k);
                            const int64_t e = u0 + sk_begin(U, G, k + 1);
                            CHECK(e <= u1, "range");
                            while (p < e) {
                                const int64_t row = sym_row(p, ntj);
                                const int64_t tb = 2 * row + (p - sym_first(row, ntj));
                                const int64_t te = tb + (e - p) < ntj ? tb + (e - p) : ntj;
                                CHECK(row >= row0 && row - row0 + k < (int64_t)slot.size(), "slot");
                                CHECK(slot[row - row0 + k] < 0, "slot twice");
                                slot[row - row0 + k] = row;
                                ++pieces[2 * row];
                                if (2 * row + 1 < ntj) ++pieces[2 * row + 1];
                                p += te - tb;
                            }
                        }
                        // the reduction: tiles from 2 row0 on
                        for (int64_t tile = 2 * row0; tile < ntj; ++tile) {
                            const int64_t row = tile / 2, f0 = sym_first(row, ntj), f1 = sym_first(row + 1, ntj);
                            CHECK(!last[tile] || f1 <= u0 || row == row0, "tile %lld after its last band", (long long)tile);
                            if (f0 < u1 && f1 > u0)
                                for (int64_t k = sk_owner(U, G, (f0 > u0 ? f0 : u0) - u0);
                                     k <= sk_owner(U, G, (f1 < u1 ? f1 : u1) - u0 - 1); ++k) {
                                    CHECK(slot[row - row0 + k] == row, "slot of row %lld", (long long)row);
                                    ++found[tile];
                                }
                            auto unit = [&](int64_t r) { return sym_first(r, ntj) + (tile - 2 * r); };
                            int64_t r0 = row0, r1 = sym_row(u1 - 1, ntj) + 1;
                            if (row < r1) r1 = row;
                            if (r0 < r1 && unit(r0) < u0) ++r0;
                            if (r0 < r1 && unit(r1 - 1) >= u1) --r1;
                            for (int64_t r = 0; r < row; ++r)
                                CHECK((unit(r) >= u0 && unit(r) < u1) == (r >= r0 && r < r1), "rows of tile %lld", (long long)tile);
                            adds[tile] += (int)(r1 > r0 ? r1 - r0 : 0);
                            last[tile] += f1 <= u1;
                        }
                    }
                    CHECK(share == cdiv(total, G), "a CTA's share %lld", (long long)share);
                    for (int64_t t = 0; t < ntj; ++t)
                        CHECK(last[t] == 1 && adds[t] == t / 2 && found[t] == pieces[t], "tile %lld", (long long)t);
                    ++cases;
                }
            }
    CHECK(split > 20, "bands were hardly used: %ld", split);
    std::printf("ok %ld\n", cases);
    return 0;
}
