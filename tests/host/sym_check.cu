// sym_check.cu -- host-only checks of the units of the all-active evaluation
// that takes each pair once (nb_sym.cuh): every (row, column) pair in exactly
// one unit, row lookup, partial slots unique and inside the scratch.  Runs on
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
    long cases = 0;
    for (int64_t ntj : {1, 2, 3, 4, 5, 63, 64, 65, 121, 128, 157, 470, 1024, 1765}) {
        const int64_t R = sym_rows(ntj), U = sym_units(ntj);
        int64_t u = 0;
        for (int64_t r = 0; r < R; ++r) {
            CHECK(sym_first(r, ntj) == u, "first of row %lld", (long long)r);
            CHECK(2 * r < ntj, "empty row");
            u += ntj - 2 * r;
            CHECK(sym_row(sym_first(r, ntj), ntj) == r && sym_row(u - 1, ntj) == r, "row %lld", (long long)r);
        }
        CHECK(u == U, "units %lld", (long long)U);
        CHECK(2 * R >= ntj, "rows cover the columns");
        for (int64_t G : {1, 152, 456, 608, 760}) {
            if (U < G) continue;
            std::vector<char> unit(U, 0), slot(R + G, 0);
            for (int64_t k = 0; k < G; ++k) {
                int64_t p = sk_begin(U, G, k);
                const int64_t e = sk_begin(U, G, k + 1);
                while (p < e) {
                    const int64_t row = sym_row(p, ntj), tb = 2 * row + (p - sym_first(row, ntj));
                    const int64_t te = tb + (e - p) < ntj ? tb + (e - p) : ntj;
                    CHECK(tb >= 2 * row && tb < te && te <= ntj, "columns");
                    CHECK(row + k < R + G && !slot[row + k], "slot %lld", (long long)(row + k));
                    slot[row + k] = 1;
                    // the reduction finds this piece among its row's
                    CHECK(sk_owner(U, G, sym_first(row, ntj)) <= k && k <= sk_owner(U, G, sym_first(row + 1, ntj) - 1),
                          "owner");
                    for (int64_t t = tb; t < te; ++t) {
                        CHECK(!unit[p + (t - tb)], "unit twice");
                        unit[p + (t - tb)] = 1;
                        CHECK(sym_first(row, ntj) + (t - 2 * row) == p + (t - tb), "unit of a column");
                    }
                    p += te - tb;
                }
            }
            for (int64_t q = 0; q < U; ++q) CHECK(unit[q], "unit %lld left out", (long long)q);
            // no slot between a row's first and last piece is left unwritten
            for (int64_t r = 0; r < R; ++r)
                for (int64_t k = sk_owner(U, G, sym_first(r, ntj)); k <= sk_owner(U, G, sym_first(r + 1, ntj) - 1); ++k)
                    CHECK(slot[r + k], "slot of row %lld", (long long)r);
            ++cases;
        }
    }
    std::printf("ok %ld\n", cases);
    return 0;
}
