// Launch of k_span (bounded FP32 instances of one warp each).
#include <cuda_runtime.h>

#include <algorithm>

#include "lbhpde.h"
#include "lbhpde_internal.h"
#include "lbhpde_span.cuh"

namespace lbh {

int span_nodes(int N) { return ((N + 31) / 32 + 3) & ~3; }

// Depth 2, the compiled degree, one warp's registers (the two ends are in different lanes from 96
// nodes on).  A warp's step costs the same for all sizes of one K, so at least 0.6 of its positions
// are to hold nodes; k_ring_nee packs smaller members closer.  us a step, k_span against k_ring_nee:
// 20 000 members of 65 nodes 4.51 : 3.70 (refused), 100 4.57 : 4.62; 4000 of 129 1.53 : 1.42
// (refused), 160 1.53 : 1.72, 257 2.23 : 2.23; 10 000 of 257 4.97 : 6.30, 3000 of 1024 3.48 : 5.41.
// D1Q7, against k_bounded: 3000 of 160 2.10 : 3.53, 4000 of 760 6.86 : 13.6.
bool span_ok(size_t esz, int b, const lbk::Seg &s) {
    const bool form = b == 5 ? s.D <= 5 && s.pad == 2 && s.N >= 96 && s.N <= 1024
                             : s.D <= 7 && (s.pad == 1 || s.pad == 2) && s.N > 128 && s.N <= 768;
    return esz == 4 && s.A == 0 && form && 5 * s.N >= 3 * 32 * span_nodes(s.N);
}

// Not one for each number of nodes a lane: the code of one is tens of KB, and an SM that runs four or
// more of them side by side waits for instructions (GB300, us a step: 250 members of 1000 nodes 0.87,
// and 250 of 500 beside them 0.95, but 250 of each of 1000, 880, 700 and 500 3.1, as long as one after
// another).  Two side by side take the sum of what each takes of the schedulers, a warp alone on one
// at least its own time: with the largest number of nodes for all, or with a second one, whichever is
// less by this (us a step on D1Q5, which measured, of 608, 1000, 2000 and 4000 members: 32 nodes a
// lane 1.07, 1.63, 3.06, 5.2; 16 nodes 0.71, 0.97, 1.73, 2.77; 8 nodes 0.52, 0.64, 1.07, 1.72).
std::vector<std::pair<int, int>> span_launches(const std::vector<int> &nodes, int sms) {
    std::vector<std::pair<int, int>> out;
    if (nodes.empty()) return out;
    auto load = [&](int K, size_t n) { return (0.104 + 0.0209 * K) * (double)((n + 4 * sms - 1) / (4 * sms)); };
    const double alone = 0.42 + 0.0195 * nodes[0];
    double best = 0.95 * std::max(alone, load(nodes[0], nodes.size()));
    size_t at = 0;
    for (size_t q = 1; q < nodes.size(); ++q) {
        if (nodes[q] == nodes[q - 1]) continue;
        const double t = std::max(alone, load(nodes[0], q) + load(nodes[q], nodes.size() - q));
        if (t < best) best = t, at = q;
    }
    out.emplace_back(nodes[0], 0);
    if (at > 0) out.emplace_back(nodes[at], (int)at);
    return out;
}

namespace {
template <int B, int K>
int launch_span_t(const lbk::SpanInst *insts, int n, const void *in, void *out, const void *coefT, const double *phib,
                  long long stride, long long step0, int nsteps, cudaStream_t st) {
    lbk::k_span<B, K><<<n, 32, 0, st>>>((const float *)in, (float *)out, insts, (const float *)coefT, phib, stride, step0, nsteps);
    if (cudaGetLastError() != cudaSuccess) return LBHPDE_ERR_CUDA;
    return LBHPDE_OK;
}
}  // namespace

int launch_span(int b, int K, const lbk::SpanInst *insts, int n, const void *in, void *out, const void *coefT, const double *phib,
                long long stride, long long step0, int nsteps, cudaStream_t st) {
    if (n == 0 || nsteps <= 0) return LBHPDE_OK;
    switch (b * 100 + K) {
#define LBH_SPAN(Bc, Kc)  \
    case Bc * 100 + Kc:   \
        return launch_span_t<Bc, Kc>(insts, n, in, out, coefT, phib, stride, step0, nsteps, st);
        LBH_SPAN(5, 4) LBH_SPAN(5, 8) LBH_SPAN(5, 12) LBH_SPAN(5, 16) LBH_SPAN(5, 20) LBH_SPAN(5, 24) LBH_SPAN(5, 28) LBH_SPAN(5, 32)
        LBH_SPAN(7, 8) LBH_SPAN(7, 12) LBH_SPAN(7, 16) LBH_SPAN(7, 20) LBH_SPAN(7, 24)
#undef LBH_SPAN
    }
    return LBHPDE_ERR_UNSUPPORTED;
}

}  // namespace lbh
