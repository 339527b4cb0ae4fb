// Launch of k_span (bounded FP32 instances of one warp each).
#include <cuda_runtime.h>

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
