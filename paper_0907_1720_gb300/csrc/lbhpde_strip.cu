// Packing and launch of k_strip (FP32 strips of one warp each).
#include <cuda_runtime.h>

#include <algorithm>

#include "lbhpde.h"
#include "lbhpde_internal.h"
#include "lbhpde_strip.cuh"

namespace lbh {

bool strip_ok(size_t esz, int b, int dc, const std::vector<lbk::Seg> &m, int *AA, int *DG) {
    *AA = *DG = 0;
    if (esz != 4 || m.empty()) return false;
    if (dc >= 0) {
        *DG = dc;
        return dc == (b == 5 ? 5 : 7) || (b == 5 && dc == 9);
    }
    // real exponents: one of the compiled row shapes in every member
    *AA = m[0].A;
    *DG = m[0].Dg;
    for (const lbk::Seg &s : m)
        if (s.A != *AA || s.Dg != *DG) return false;
    return b == 5 && *AA == 4 && (*DG == 1 || *DG == 5);
}

void pack_strip(int b, int AA, int DG, const std::vector<lbk::Seg> &m, PackedStrip &out) {
    out = PackedStrip{};
    out.b = b;
    out.AA = AA;
    out.DG = DG;
    const int K = lbk::strip_K(b, AA), HL = lbk::strip_HL(b), own = (32 - 2 * HL) * K;
    auto seg = [&](const lbk::Seg &s, long long at, int V, int lane0, int nlanes) {
        lbk::StripSeg S{};
        S.off = s.off;
        S.ld = s.ld;
        S.N = s.N;
        S.D = s.D;
        S.gcoef = s.coef;
        S.x0 = (int)(at - HL * K);
        S.vlo = HL * K;
        S.vhi = S.vlo + V;
        S.lane0 = lane0;
        S.nlanes = nlanes;
        S.nu = (float)s.nu;
        return S;
    };
    struct Rest {
        int i, V, nl;
    };
    std::vector<Rest> rest;
    for (size_t i = 0; i < m.size(); ++i) {
        long long at = 0;
        for (; at + own <= m[i].N; at += own) {
            out.segs.push_back(seg(m[i], at, own, 0, 32));
            ++out.nfull;
        }
        if (at < m[i].N) rest.push_back(Rest{(int)i, (int)(m[i].N - at), 2 * HL + (int)((m[i].N - at + K - 1) / K)});
    }
    // what is left of each instance: first fit, largest first, into warps of 32 lanes
    std::stable_sort(rest.begin(), rest.end(), [](const Rest &x, const Rest &y) { return x.nl > y.nl; });
    std::vector<std::vector<lbk::StripSeg>> warps;
    std::vector<std::vector<int>> by_free(33);  // open warps by their free lanes
    for (const Rest &r : rest) {
        int w = -1, fr = r.nl;
        while (fr <= 32 && by_free[fr].empty()) ++fr;
        if (fr <= 32) {
            w = by_free[fr].back();
            by_free[fr].pop_back();
        } else {
            w = (int)warps.size();
            warps.emplace_back();
            fr = 32;
        }
        warps[w].push_back(seg(m[r.i], m[r.i].N - r.V, r.V, 32 - fr, r.nl));
        if ((int)warps[w].size() < lbk::kStripSegs && fr - r.nl > 2 * HL) by_free[fr - r.nl].push_back(w);
    }
    for (const auto &w : warps) {
        out.first.push_back((int)out.segs.size());
        out.segs.insert(out.segs.end(), w.begin(), w.end());
    }
    out.first.push_back((int)out.segs.size());
}

namespace {

template <int B, int DC, int AA = 0, int DG = 0>
int launch_strip_t(const PackedStrip &p, const lbk::StripSeg *segs, const int *first, const void *in, void *out,
                   const void *coefT, int nsteps, cudaStream_t st) {
    auto fn = lbk::k_strip<B, DC, AA, DG>;
    const int smem = lbk::strip_smem(B, AA, DC);
    if (!allow_smem(fn)) return LBHPDE_ERR_CUDA;
    fn<<<p.nwarps(), 32, smem, st>>>((const float *)in, (float *)out, segs, first, p.nmix(), (const float *)coefT, nsteps);
    if (cudaGetLastError() != cudaSuccess) return LBHPDE_ERR_CUDA;
    return LBHPDE_OK;
}

}  // namespace

int launch_strip(const PackedStrip &p, const lbk::StripSeg *segs, const int *first, const void *in, void *out,
                 const void *coefT, int nsteps, cudaStream_t st) {
    if (p.nwarps() == 0 || nsteps <= 0) return LBHPDE_OK;
    if (in == out || nsteps > lbk::strip_steps(p.b, p.AA)) return LBHPDE_ERR_ARG;
    if (p.AA == 4 && p.DG == 1) return launch_strip_t<5, 9, 4, 1>(p, segs, first, in, out, coefT, nsteps, st);
    if (p.AA == 4 && p.DG == 5) return launch_strip_t<5, 29, 4, 5>(p, segs, first, in, out, coefT, nsteps, st);
    if (p.b == 5 && p.DG == 9) return launch_strip_t<5, 9>(p, segs, first, in, out, coefT, nsteps, st);
    return p.b == 5 ? launch_strip_t<5, 5>(p, segs, first, in, out, coefT, nsteps, st)
                    : launch_strip_t<7, 7>(p, segs, first, in, out, coefT, nsteps, st);
}

}  // namespace lbh
