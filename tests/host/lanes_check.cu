// lanes_check.cu -- host-only checks of the planning rules for small launches
// (sk_lanes, split_max, choose_split): runs on the CPU, makes no CUDA call.
// Prints "ok <cases>" or the first violated property.
#include <cstdio>
#include <cstdlib>

#include "../../paper_1812_00367_gb300/csrc/nb_internal.cuh"

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
    const int precisions[] = {NB_FP64, NB_EX, NB_FP32, NB_FP32X};
    const long long ns[] = {1, 2, 63, 64, 65, 300, 1024, 4096, 10007, 65536, 1048576};
    for (int p : precisions)
        for (long long G : {152LL, 456LL, 608LL, 760LL})
            for (long long n : ns)
                for (long long A = 1; A <= n; A = A * 3 / 2 + 1)
                    for (int gl0 = 1; gl0 <= 32; gl0 *= 2) {
                        const int64_t ntj = cdiv(n, kTJ);
                        const int gl = sk_lanes(gl0, A, ntj, G, p);
                        // a power of two from the table's choice to a warp
                        CHECK(gl >= gl0 && gl <= 32 && (gl & (gl - 1)) == 0, "gl %d from %d", gl, gl0);
                        const int64_t tiles = cdiv(A, kTPB / gl), U = tiles * ntj;
                        // raised only while the launch has too few units, and then as far as needed
                        if (gl > gl0)
                            CHECK(cdiv(A, kTPB / (gl / 2)) * ntj < sk_lane_units(p) * G, "raised too far: %d", gl);
                        if (p == NB_FP64) CHECK(gl == 32 || U >= sk_lane_units(p) * G, "gl %d U %lld", gl, (long long)U);
                        // single-precision sums keep the table's lanes
                        if (p == NB_FP32 || p == NB_FP32X) CHECK(gl == gl0, "gl %d", gl);
                        // never for a share below the arithmetic's least
                        if (A * ntj * kTJ < (int64_t)sk_min_pairs(p) * G * kTPB) CHECK(gl == gl0, "gl %d", gl);
                        // splits: at least one range, each of at least one tile
                        const int64_t smax = split_max(ntj, p);
                        CHECK(smax >= 1 && smax <= (ntj > 1 ? ntj : 1), "smax %lld of %lld", (long long)smax, (long long)ntj);
                        if (p != NB_FP64) CHECK(smax == 1 || ntj / smax >= kMinTilesPerItem, "smax %lld", (long long)smax);
                        const int64_t S = choose_split(tiles, ntj, 8 * G, G, p);
                        CHECK(S >= 1 && S <= smax, "S %lld of %lld", (long long)S, (long long)smax);
                        ++cases;
                    }
    std::printf("ok %ld\n", cases);
    return 0;
}
