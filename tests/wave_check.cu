// Host-side check of the one-warp windows of k_wave (no GPU): every node belongs to exactly one
// window, every position stays inside the warp, and, replaying steps and trades with node numbers
// in place of values, each own node always pulls from the right nodes at the right step.  Prints
// "ok" and exits 0, or the first violation and exits 1.
#include <cstdio>
#include <cstdlib>
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

// what a position holds: node x of the state after `step` steps (step < 0: not a value of the solve)
struct Val {
    long long x;
    int step;
};

static void replay(const std::vector<lbk::WaveWin> &w, int b, int K, int G, int T, int nsteps, bool in_place) {
    const int W = lbk::wmax(b), H = T * W, P = lbk::wave_positions(K, G);
    std::vector<std::vector<Val>> pos(w.size(), std::vector<Val>(P, Val{-1, -1}));
    for (size_t i = 0; i < w.size(); ++i) {
        if (w[i].N == 0) continue;
        CHECK(H <= lbk::wave_pitch(K, G) || (w[i].left < 0 && w[i].right < 0), "window %zu: borders of %d", i, H);
        const int lo = w[i].left >= 0 ? w[i].vlo - H : w[i].vlo, hi = w[i].right >= 0 ? w[i].vhi + H : w[i].vhi;
        CHECK(lo >= 0 && hi <= P && w[i].vlo < w[i].vhi, "window %zu: positions [%d, %d) of %d", i, lo, hi, P);
        for (int p = lo; p < hi && p < P; ++p) pos[i][p] = Val{((long long)w[i].x0 + p + 4LL * w[i].N) % w[i].N, 0};
    }
    auto trade = [&](int step) {
        auto old = pos;
        for (size_t i = 0; i < w.size(); ++i) {
            for (int k = 0; k < H && w[i].N > 0; ++k) {
                if (w[i].left >= 0) {
                    const lbk::WaveWin &n = w[w[i].left];
                    CHECK(n.vhi - H >= n.vlo, "window %zu: its left neighbour owns fewer than %d nodes", i, H);
                    pos[i][k] = old[w[i].left][n.vhi - H + k];
                    CHECK(w[i].vlo == H, "window %zu: first own position %d", i, w[i].vlo);
                    CHECK(pos[i][k].step == step, "window %zu: copy of step %d, expected %d", i, pos[i][k].step, step);
                }
                if (w[i].right >= 0) pos[i][w[i].vhi + k] = old[w[i].right][w[w[i].right].vlo + k];
            }
        }
    };
    int done = 0;
    if (in_place && nsteps <= T) trade(0);
    while (done < nsteps) {
        const int n = std::min(T, nsteps - done);
        for (int s = 0; s < n; ++s) {
            for (size_t i = 0; i < w.size(); ++i) {
                if (w[i].N == 0) continue;
                auto old = pos[i];
                const bool nee = w[i].depth > 0;
                const long long N = w[i].N;
                for (int p = 0; p < P; ++p) {
                    if (old[p].step < 0) continue;
                    const bool outer = nee && (old[p].x < W || old[p].x >= N - W);
                    bool ok = true;
                    for (int e = -W; e <= W && !outer; ++e) {
                        const int q = p - e;
                        const long long want = nee ? old[p].x - e : (old[p].x - e + N) % N;
                        ok = ok && q >= 0 && q < P && old[q].step == old[p].step && old[q].x == want;
                    }
                    if (outer) {  // rebuilt from x_f after its own step: the same window, an own node
                        const long long xf = old[p].x < W ? W - 1 + w[i].depth : N - W - w[i].depth;
                        const long long q = xf - w[i].x0;
                        ok = q >= w[i].vlo && q < w[i].vhi && old[q].x == xf && old[q].step == old[p].step;
                        CHECK((old[p].x < W ? w[i].left : w[i].right) < 0, "window %zu: an outer node is a copy", i);
                    }
                    pos[i][p].step = ok ? old[p].step + 1 : -1;
                }
                for (int p = w[i].vlo; p < w[i].vhi; ++p)
                    CHECK(pos[i][p].step == done + s + 1 && pos[i][p].x == ((long long)w[i].x0 + p + 4 * N) % N,
                          "b %d K %d T %d N %lld window %zu position %d: step %d of node %lld, expected %d", b, K, T, N, i, p,
                          pos[i][p].step, pos[i][p].x, done + s + 1);
            }
        }
        done += n;
        if (done < nsteps) trade(done);
    }
}

int main() {
    std::mt19937 g(7);
    int planned = 0;
    for (int t = 0; t < 6000 && !fails; ++t) {
        const int b = g() % 2 ? 5 : 7, G = g() % 2 ? 1 : (g() % 2 ? 2 : (b == 5 ? 4 : 3));
        const int K = G > 1 ? 1 : 1 << (g() % 3), T = 1 + g() % (G > 1 ? 3 : 16), W = lbk::wmax(b);
        const int csize = g() % 2 ? 0 : 1 << (g() % 5), room = csize * lbk::kWaveWarps;
        const bool nee = g() % 2;
        std::vector<lbk::Seg> m;
        for (int i = 0, n = 1 + (int)(g() % 3); i < n; ++i) {
            lbk::Seg x{};
            x.pad = nee ? 1 + (int)(g() % 4) : 0;
            const int lo = nee ? 2 * (W + x.pad) : 2 * W;
            x.N = lo + (int)(g() % (g() % 2 ? 40 : 1500));
            m.push_back(x);
        }
        std::vector<lbk::WaveWin> w;
        if (!lbh::pack_wave(m, b, K, G, T, csize, w)) continue;
        ++planned;
        size_t at = 0;
        for (size_t i = 0; i < m.size(); ++i) {  // the windows of a member own its nodes in order, once each
            while (at < w.size() && w[at].N == 0) ++at;
            long long next = 0;
            const size_t first = at;
            for (; at < w.size() && w[at].N > 0 && w[at].mi == (int)i; ++at) {
                CHECK(w[at].x0 + w[at].vlo == next && w[at].N == m[i].N, "member %zu: window starts at node %d, expected %lld", i,
                      w[at].x0 + w[at].vlo, next);
                next = w[at].x0 + w[at].vhi;
                for (int nb : {w[at].left, w[at].right})
                    CHECK(nb < 0 || (nb >= (int)first && nb < (int)w.size() && w[nb].N > 0 && w[nb].mi == (int)i),
                          "window %zu: neighbour %d", at, nb);
                CHECK(csize == 0 || at / room == first / room, "member %zu spans two clusters", i);
                CHECK(w[at].vhi - w[at].vlo >= K || (w[at].left < 0 && w[at].right < 0), "window %zu: own nodes", at);
            }
            CHECK(next == m[i].N, "member %zu: windows end at node %lld of %d", i, next, m[i].N);
            CHECK((w[first].left < 0) == nee && (w[at - 1].right < 0) == nee, "member %zu: ends", i);
        }
        CHECK(w.size() % ((csize > 0 ? csize : 1) * lbk::kWaveWarps) == 0, "%zu places", w.size());
        replay(w, b, K, G, T, 1 + (int)(g() % (3 * T)), g() % 2);
    }
    CHECK(planned > 1000, "only %d plans", planned);
    if (!fails) std::printf("ok %d plans\n", planned);
    return fails ? 1 : 0;
}
