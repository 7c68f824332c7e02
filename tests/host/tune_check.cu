// tune_check.cu -- host-only checks of the plan shared by the planner, the
// host-planned evaluations and the autotuner (plan_eval): what the autotuner times
// and stores is what a later plan from the stored entry runs, with stream-K ranges
// and without.  Runs on the CPU, makes no CUDA call.  Prints "ok <cases>" or the
// first violated property.
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
    long cases = 0, raised = 0;
    for (int prec : {NB_FP64, NB_EX, NB_FP32, NB_FP32X})
        for (int64_t G : {456, 608, 760})
            for (int64_t n : {1, 64, 300, 1024, 4096, 10007, 65536})
                for (int64_t A = 1; A <= n; A = A * 3 / 2 + 1)
                    for (int gl = 1; gl <= 32; gl *= 2)
                        for (int64_t target : {G / 2, G, 8 * G, 16 * G})
                            for (int streamk = 0; streamk < 2; ++streamk) {
                                const int64_t ntj = cdiv(n, kTJ), cap = 32 * G * 10 * kTPB;
                                const PlanEntry e{gl, (int32_t)target};
                                const EvalPlan p = plan_eval(e, A, ntj, streamk != 0, G, cap, prec);
                                const EvalPlan q = plan_eval(PlanEntry{p.gl, e.target_items}, A, ntj, streamk != 0, G, cap, prec);
                                CHECK(p.gl == q.gl && p.split == q.split && p.tiles == q.tiles && p.streamk == q.streamk,
                                      "gl %d stored %d planned %d", gl, p.gl, q.gl);
                                CHECK((int64_t)p.tiles * (kTPB / p.gl) >= A, "tiles");
                                if (!streamk) {  // the entry's own lanes, split items
                                    CHECK(p.gl == gl && p.streamk == 0, "gl %d planned %d", gl, p.gl);
                                    CHECK(p.split == choose_split(p.tiles, ntj, target, G, prec), "split %d", p.split);
                                }
                                if (p.streamk) CHECK(p.split == 1, "split %d", p.split);
                                raised += p.gl > gl;
                                ++cases;
                            }
    CHECK(raised > 1000, "lanes hardly raised: %ld", raised);
    std::printf("ok %ld\n", cases);
    return 0;
}
