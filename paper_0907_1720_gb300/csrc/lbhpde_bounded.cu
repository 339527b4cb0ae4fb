// Launchers of the bounded-grid kernels (lbhpde_bounded.cuh): the resident kernel k_bounded,
// one instance per CTA, and the outer-node rebuild k_nee_fix that follows a streaming step.
#include <algorithm>
#include <cmath>

#include "lbhpde_bounded.cuh"
#include "lbhpde_internal.h"

namespace lbh {

namespace {

#define LBB_CK(call)                  \
    do {                              \
        cudaError_t e_ = (call);      \
        if (e_ != cudaSuccess) {      \
            (void)cudaGetLastError(); \
            return LBHPDE_ERR_CUDA;   \
        }                             \
    } while (0)

struct BoundedArgs {
    int ninst, nthreads;
    size_t smem;
    const lbk::BoundedInst *insts;
    const void *in;
    void *out;
    const void *coefT;
    const double *phib;
    long long stride, step0;
    int nsteps;
    cudaStream_t st;
    int K;
};

template <typename T, int B, int DC, int K = kBoundedK, int MAXT = kBoundedMaxT>
int launch_bounded_t(const BoundedArgs &a) {
    auto fn = lbk::k_bounded<T, B, K, MAXT, DC>;
    if (!allow_smem(fn)) return LBHPDE_ERR_CUDA;
    fn<<<a.ninst, a.nthreads, a.smem, a.st>>>((const T *)a.in, (T *)a.out, a.insts, (const T *)a.coefT, a.phib,
                                             a.stride, a.step0, a.nsteps);
    LBB_CK(cudaGetLastError());
    return LBHPDE_OK;
}

template <typename T, int B>
int launch_bounded_d(int dc, const BoundedArgs &a) {
    constexpr int DC = bounded_degree(B);
    if constexpr (sizeof(T) == 8) {  // FP64: the nodes a thread of the plan
        if (dc == DC && a.K == 3) return launch_bounded_t<T, B, DC, 3, kBoundedMaxTAny>(a);
        if (dc == DC && a.K == 5) return launch_bounded_t<T, B, DC, 5, kBoundedMaxTAny>(a);
        if (dc == DC && a.K == 6) return launch_bounded_t<T, B, DC, 6, kBoundedMaxTAny>(a);
    }
    if (a.K != kBoundedK) return LBHPDE_ERR_UNSUPPORTED;
    if (dc == DC) return launch_bounded_t<T, B, DC>(a);
    if (dc < 0) return launch_bounded_t<T, B, -1>(a);  // real-exponent members
    return launch_bounded_t<T, B, 0>(a);
}

}  // namespace

size_t bounded_smem(int b, size_t esz, int nthreads, int D, int nsteps) {
    const int W = lbk::wmax(b), NE = lbk::nedge(b), cs = lbk::crow(D);
    return (size_t(4) * NE * nthreads + size_t(2) * (b - 1) * cs + 16 + size_t(nsteps) * 2 * W * b) * esz;
}

int bounded_shift(int b, int N, int depth, int K) {
    const int W = lbk::wmax(b), maxt = K == kBoundedK ? kBoundedMaxT : kBoundedMaxTAny;
    const int kL = W - 1 + depth, kR = N - W - depth;
    for (int shift = 0; kL + shift < 32 * K; ++shift) {
        const bool right_in_one_warp = ((kR + shift) / K) / 32 == ((N - 1 + shift) / K) / 32;
        if (right_in_one_warp && N + shift <= K * maxt) return shift;
    }
    return -1;
}

// The scheduler with the most warps paces an SM (an FP64 operation of a warp holds it for 64 clocks),
// and a warp that is half empty costs as much as a full one: of the warps of the ceil(n / SMs)
// instances of an SM it holds a quarter, rounded up.  601 nodes on D1Q7, two instances an SM (GB300, us a
// step): 5 warps each at K = 4 21.5, 4 at K = 5 20.8; one instance 12.7 and 11.5; 301 nodes, two, 3 warps at
// K = 4 13.1, 2 at K = 5 11.6.
int bounded_nodes(int b, const std::vector<lbk::Seg> &m, int sms) {
    int best = kBoundedK;
    double least = 0;
    for (int K : {kBoundedK, 3, 5, 6}) {
        if (K < lbk::wmax(b)) continue;
        long long warps = 0;
        bool fits = true;
        for (const lbk::Seg &s : m) {
            const int shift = bounded_shift(b, s.N, s.pad, K);
            fits = fits && shift >= 0;
            warps += (s.N + shift + 32 * K - 1) / (32 * K);
        }
        if (!fits) continue;
        const long long ctas = ((long long)m.size() + sms - 1) / sms;  // instances of the fullest SM
        const double per = (double)warps / m.size() * ctas;
        const double c = std::ceil(per / 4.0 - 1e-9) * K;
        if (least == 0 || c < 0.97 * least) {
            least = c;
            best = K;
        }
    }
    return best;
}

int bounded_launch_steps(int b, size_t esz) {
    const int per_step = 2 * lbk::wmax(b) * b * (int)esz;  // bytes of staged boundary data per step
    return std::max(32, std::min(kBoundedMaxSteps, kBoundedStageBytes / per_step));
}

int launch_bounded(int b, size_t esz, int dc, int ninst, int nthreads, size_t smem, const lbk::BoundedInst *insts_d,
                   const void *in, void *out, const void *coefT, const double *phib, long long stride,
                   long long step0, int nsteps, cudaStream_t st, int K) {
    if (ninst == 0 || nsteps <= 0) return LBHPDE_OK;
    if (nthreads <= 0 || nthreads > (K == kBoundedK ? kBoundedMaxT : kBoundedMaxTAny) || nthreads % 32) return LBHPDE_ERR_ARG;
    const BoundedArgs a{ninst, nthreads, smem, insts_d, in, out, coefT, phib, stride, step0, nsteps, st, K};
    if (esz == 4) return b == 5 ? launch_bounded_d<float, 5>(dc, a) : launch_bounded_d<float, 7>(dc, a);
    return b == 5 ? launch_bounded_d<double, 5>(dc, a) : launch_bounded_d<double, 7>(dc, a);
}

int launch_nee_fix(int b, size_t esz, void *st, const lbk::Seg *segs, const int *members, int nmem,
                   const void *coefT, const double *phib, long long stride, long long step, cudaStream_t stream) {
    if (nmem == 0) return LBHPDE_OK;
    if (esz == 4) {
        if (b == 5)
            lbk::k_nee_fix<float, 5><<<nmem, 32, 0, stream>>>((float *)st, segs, members, (const float *)coefT, phib,
                                                              stride, step);
        else
            lbk::k_nee_fix<float, 7><<<nmem, 32, 0, stream>>>((float *)st, segs, members, (const float *)coefT, phib,
                                                              stride, step);
    } else {
        if (b == 5)
            lbk::k_nee_fix<double, 5><<<nmem, 32, 0, stream>>>((double *)st, segs, members, (const double *)coefT,
                                                               phib, stride, step);
        else
            lbk::k_nee_fix<double, 7><<<nmem, 32, 0, stream>>>((double *)st, segs, members, (const double *)coefT,
                                                               phib, stride, step);
    }
    LBB_CK(cudaGetLastError());
    return LBHPDE_OK;
}

}  // namespace lbh
