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

// An SM does the FP64 work of four warps at a time, a warp's alone takes as long as a quarter of four
// warps' (its own operations one after another), and a warp that is half empty costs as much as a full
// one.  So a step of the members an SM holds at once takes, in units of one position a lane, K times a
// quarter of their warps, at least K, and a little more where a quarter is no whole number, on top of a
// barrier and the ends.  How many it holds the registers say (and every CTA has the warps of the
// largest member); the rest follow in further rounds.  GB300, us a step at K = 4, 3, 5, 6: D1Q7, 304 of
// 601 nodes 21.7, 22.9, 20.9, 24.9; 304 of 301 13.3, 12.8, 11.7, 13.8; 160 of 847 (K = 5 and 6: one at a time)
// 29.3, -, 32.6, 37.5; 1500 of 150 to 601 78.0, 85.2, 82.9, 84.1; D1Q5, 152 of 301 5.35, 4.38, 6.49, 7.56.
int bounded_nodes(int b, const std::vector<lbk::Seg> &m, int sms) {
    int best = kBoundedK;
    double least = 0;
    for (int K : {kBoundedK, 3, 5, 6}) {
        if (K < lbk::wmax(b)) continue;
        // warps an SM holds (registers a thread: 128 at K = 4, 154 (D1Q5) and 192 at 3, 214 to 254 at 5 and 6)
        const int room = K == 4 ? 16 : (K == 3 && b == 5 ? 12 : 8);
        long long warps = 0;
        int wmost = 1;
        bool fits = true;
        for (const lbk::Seg &s : m) {
            const int shift = bounded_shift(b, s.N, s.pad, K);
            fits = fits && shift >= 0;
            const int w = (s.N + shift + 32 * K - 1) / (32 * K);
            warps += w;
            wmost = std::max(wmost, w);
        }
        if (!fits) continue;
        const int per_sm = (int)(((long long)m.size() + sms - 1) / sms);  // members of the fullest SM
        const int at_once = std::min(per_sm, std::max(1, room / wmost));
        const double mean = per_sm == 1 ? wmost : (double)warps / m.size();
        auto round = [&](int n) {
            const double q = n * mean / 4.0;
            return (b == 5 ? 1.03 : 0.65) + K * std::max(1.0, q + 0.29 * (std::ceil(q - 1e-9) - q));
        };
        const double c = per_sm / at_once * round(at_once) + (per_sm % at_once ? round(per_sm % at_once) : 0.0);
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
