// Host-side check of the estimates that choose the kernels (no GPU).  Prints
// "ok" and exits 0, or the first violation and exits 1.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "lbhpde_internal.h"

static int fails = 0;
#define CHECK(c, ...)                                        \
    do {                                                     \
        if (!(c) && fails++ == 0) {                          \
            std::printf("FAIL %s:%d: ", __FILE__, __LINE__); \
            std::printf(__VA_ARGS__);                        \
            std::printf("\n");                               \
        }                                                    \
    } while (0)

static std::vector<lbk::Seg> members(int count, int N, int D) {
    lbk::Seg s{};
    s.N = N;
    s.D = D;
    return std::vector<lbk::Seg>(count, s);
}

int main() {
    const int sms = 152;
    // a cubic flux (degree 9 of D1Q5) takes 4 (9 + 3) + 1 operations a node where a quadratic one takes
    // 4 (5 + 3) + 1: FP64, where those are the cost of a step, in k_wave's estimate as in the others'
    for (int count : {16, 64, 128}) {
        const auto m5 = members(count, 1000, 5), m9 = members(count, 1000, 9);
        const double w5 = lbh::wave_cost(8, 5, 5, false, m5, sms), w9 = lbh::wave_cost(8, 5, 9, false, m9, sms);
        const double c5 = lbh::cta_cost(8, 5, 5, false, false, m5, sms), c9 = lbh::cta_cost(8, 5, 9, false, false, m9, sms);
        CHECK(w9 > 1.3 * w5 && w9 < 1.49 * w5, "%d members: k_wave %g and %g", count, w5, w9);
        CHECK(c9 > 1.3 * c5 && c9 < 1.49 * c5, "%d members: CTAs %g and %g", count, c5, c9);
    }
    // bounded FP64 members on k_bounded: the nodes a thread that measured least (within 3%) on a GPU of 152 SMs
    const struct {
        int b, count, lo, hi, K;
    } bounded[] = {{7, 304, 601, 601, 5}, {7, 304, 301, 301, 5}, {7, 152, 301, 301, 3}, {5, 152, 601, 601, 5}, {5, 304, 847, 847, 4},
                   {7, 304, 847, 847, 4}, {7, 152, 250, 1000, 4}, {5, 1500, 150, 601, 4}, {7, 504, 450, 450, 4}, {7, 304, 300, 1200, 4}};
    for (const auto &c : bounded) {
        std::vector<lbk::Seg> m = members(c.count, c.hi, c.b);
        for (int i = 0; i < c.count; ++i) {
            m[i].N = c.lo + (int)((long long)(c.hi - c.lo) * i / std::max(1, c.count - 1));
            m[i].pad = c.b == 5 ? 2 : 1;
        }
        const int K = lbh::bounded_nodes(c.b, m, sms);
        CHECK(K == c.K, "D1Q%d, %d members of %d to %d nodes: %d nodes a thread", c.b, c.count, c.lo, c.hi, K);
    }
    // FP64 windows of a chosen size, or one CTA a member and windows of the default size: what measured
    // least (both sides over 3% apart)
    const struct {
        int b, count, N;
        bool windows;
    } w64[] = {{7, 114, 581, false}, {7, 128, 643, false}, {7, 283, 340, false}, {7, 537, 341, false}, {5, 298, 1547, false}, {7, 21, 18787, false},
               {5, 100, 2048, true}, {7, 1, 300001, true}, {5, 1, 300001, true}, {7, 166, 1000, true}, {5, 80, 2406, true}};
    for (const auto &c : w64) {
        int threads = 0, T = 0;
        const bool got = lbh::windows_f64(c.b, c.b, 4, members(c.count, c.N, c.b), sms, &threads, &T);
        CHECK(got == c.windows, "D1Q%d, %d members of %d nodes: windows %d", c.b, c.count, c.N, got);
    }
    if (!fails) std::printf("ok\n");
    return fails ? 1 : 0;
}
