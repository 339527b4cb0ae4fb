// Host-side check of the strips of k_strip (no GPU): the segments of a member own its nodes in
// order, once each, no two segments of a warp share a lane, and, replaying steps with node numbers in
// place of values, each own node still holds a right value after the most steps a launch can take.
// Prints "ok" and exits 0, or the first violation and exits 1.
#include <algorithm>
#include <cstdio>
#include <random>
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

int main() {
    std::mt19937 g(11);
    size_t warps = 0, lanes = 0, own = 0;
    for (int t = 0; t < 200 && !fails; ++t) {
        const int b = g() % 2 ? 5 : 7, W = lbk::wmax(b), AA = b == 5 && g() % 2 ? 4 : 0;
        const int K = lbk::strip_K(b, AA), P = 32 * K, T = lbk::strip_steps(b, AA);
        std::vector<lbk::Seg> m;
        for (int i = 0, n = 1 + (int)(g() % 40); i < n; ++i) {
            lbk::Seg s{};
            const int top[4] = {40, 700, 3000, 9000};
            s.N = 2 * W + (int)(g() % top[g() % 4]);
            s.off = (long long)i << 20;
            m.push_back(s);
        }
        lbh::PackedStrip p;
        lbh::pack_strip(b, AA, AA ? 1 : (b == 5 ? 5 : 7), m, p);
        std::vector<std::vector<int>> count(m.size());
        for (size_t i = 0; i < m.size(); ++i) count[i].assign(m[i].N, 0);
        for (int w = 0; w < p.nwarps(); ++w) {
            const int s0 = w < p.nmix() ? p.first[w] : w - p.nmix(), s1 = w < p.nmix() ? p.first[w + 1] : s0 + 1, ns = s1 - s0;
            CHECK(w < p.nmix() || (p.segs[s0].lane0 == 0 && p.segs[s0].nlanes == 32), "warp %d: lanes of a whole segment", w);
            CHECK(ns >= 1 && ns <= lbk::kStripSegs, "warp %d: %d segments", w, ns);
            std::vector<long long> node(P, -1);  // member << 32 | node
            std::vector<int> good(P, 0);
            std::vector<bool> taken(32, false);
            for (int s = s0; s < s1; ++s) {
                const lbk::StripSeg &S = p.segs[s];
                const long long i = S.off >> 20;
                CHECK(S.lane0 >= 0 && S.nlanes > 0 && S.lane0 + S.nlanes <= 32, "warp %d: lanes %d + %d", w, S.lane0, S.nlanes);
                CHECK(S.vlo == lbk::strip_HL(b) * K && S.vhi > S.vlo && S.vhi <= S.nlanes * K, "warp %d: own [%d, %d)", w, S.vlo, S.vhi);
                for (int l = 0; l < S.nlanes; ++l) {
                    CHECK(!taken[S.lane0 + l], "warp %d: lane %d twice", w, S.lane0 + l);
                    taken[S.lane0 + l] = true;
                    ++lanes;
                }
                for (int q = 0; q < S.nlanes * K; ++q) {
                    const long long x = ((S.x0 + q) % S.N + S.N) % S.N;
                    node[S.lane0 * K + q] = i << 32 | x;
                    good[S.lane0 * K + q] = 1;
                    if (q >= S.vlo && q < S.vhi) ++count[i][x], ++own;
                }
            }
            for (int s = 0; s < T; ++s) {  // a position stays right while all it pulls from is right
                std::vector<int> was = good;
                for (int q = 0; q < P; ++q)
                    for (int e = -W; e <= W; ++e) {
                        const int r = q - e;
                        bool ok = was[q] && r >= 0 && r < P && was[r];
                        if (ok) {
                            const long long N = m[node[q] >> 32].N, x = node[q] & 0xffffffff;
                            ok = node[r] == ((node[q] >> 32) << 32 | (x - e + N) % N);
                        }
                        good[q] = good[q] && ok;
                    }
            }
            for (int s = s0; s < s1; ++s)
                for (int q = p.segs[s].vlo; q < p.segs[s].vhi; ++q)
                    CHECK(good[p.segs[s].lane0 * K + q], "b %d warp %d segment %d: own position %d after %d steps", b, w, s, q, T);
            ++warps;
        }
        for (size_t i = 0; i < m.size(); ++i)
            for (int x = 0; x < m[i].N; ++x) CHECK(count[i][x] == 1, "member %zu: node %d owned %d times", i, x, count[i][x]);
    }
    if (!fails) std::printf("ok %zu warps, %.1f%% of the lanes used\n", warps, 100.0 * lanes / (32.0 * warps));
    return fails ? 1 : 0;
}
