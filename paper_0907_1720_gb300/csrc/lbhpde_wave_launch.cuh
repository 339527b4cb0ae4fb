// Planning and launch of k_wave (windows of one warp each, spread over the GPU); one translation unit
// per precision (LBH_WAVE_ESZ 4 or 8) includes it, and the FP64 one holds the planning.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <functional>

#include "lbhpde.h"
#include "lbhpde_internal.h"

namespace lbh {

namespace {

struct WaveArgs {
    const PackedWave *p;
    const lbk::WaveWin *wins;
    unsigned char *box;
    unsigned *ctrl;
    const void *in;
    void *out;
    const void *coefT;
    int nsteps;
    const void *ends;
    cudaStream_t st;
    int *room;  // asked for: the CTAs (or clusters) that the GPU holds at once, instead of a launch
};

template <typename T, int B, int K, int G, int DC, bool NEE>
int launch_wave_t(const WaveArgs &a) {
    auto fn = lbk::k_wave<T, B, K, G, DC, NEE>;
    const PackedWave &p = *a.p;
    if (!allow_smem(fn) ||
        (p.csize > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
        (void)cudaGetLastError();
        return LBHPDE_ERR_CUDA;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)p.ncta());
    cfg.blockDim = dim3(32 * lbk::kWaveWarps);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = a.st;
    cudaLaunchAttribute at[1];
    if (p.csize > 0) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)p.csize;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    } else {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (a.room) {
        const cudaError_t e = p.csize > 0 ? cudaOccupancyMaxActiveClusters(a.room, fn, &cfg)
                                          : cudaOccupancyMaxActiveBlocksPerMultiprocessor(a.room, fn, 32 * lbk::kWaveWarps, p.smem);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            return LBHPDE_ERR_CUDA;
        }
        return LBHPDE_OK;
    }
    if (cudaLaunchKernelEx(&cfg, fn, (const T *)a.in, (T *)a.out, a.wins, p.nused, (const T *)a.coefT, a.box, a.ctrl,
                           a.nsteps, p.tblk, p.csize, (const T *)a.ends, p.wsmem) != cudaSuccess) {
        (void)cudaGetLastError();
        return LBHPDE_ERR_CUDA;
    }
    return LBHPDE_OK;
}

template <typename T, int B, int K, int G, bool NEE>
int launch_wave_d(const WaveArgs &a) {
    constexpr int DC = B == 5 ? 5 : 7;
    if (a.p->dc == DC) return launch_wave_t<T, B, K, G, DC, NEE>(a);
    if constexpr (B == 5)
        if (a.p->dc == 9) return launch_wave_t<T, B, K, G, 9, NEE>(a);
    if constexpr (K == (sizeof(T) == 4 ? 2 : 1) && G == 1) {  // run-time degrees and real exponents
        if (a.p->dc == 0) return launch_wave_t<T, B, K, G, 0, NEE>(a);
        if (a.p->dc < 0) return launch_wave_t<T, B, K, G, -1, NEE>(a);
    }
    return LBHPDE_ERR_UNSUPPORTED;
}

template <typename T, int B, bool NEE>
int launch_wave_k(const WaveArgs &a) {
    const int K = a.p->K, G = a.p->G;
    if (K == 1 && G == 1) return launch_wave_d<T, B, 1, 1, NEE>(a);
    if (K == 2 && G == 1) return launch_wave_d<T, B, 2, 1, NEE>(a);
    if constexpr (sizeof(T) == 4) {
        if (K == 4 && G == 1) return launch_wave_d<T, B, 4, 1, NEE>(a);
    } else {
        if (K == 1 && G == 2) return launch_wave_d<T, B, 1, 2, NEE>(a);
        if (K == 1 && G == (B == 5 ? 4 : 3)) return launch_wave_d<T, B, 1, (B == 5 ? 4 : 3), NEE>(a);
    }
    return LBHPDE_ERR_UNSUPPORTED;
}

template <typename T>
int launch_wave_b(const WaveArgs &a) {
    if (a.p->b == 5) return a.p->nee ? launch_wave_k<T, 5, true>(a) : launch_wave_k<T, 5, false>(a);
    return a.p->nee ? launch_wave_k<T, 7, true>(a) : launch_wave_k<T, 7, false>(a);
}

template <typename T, int B>
int launch_ends_t(void *ends, const lbk::Seg *segs, const int *members, int nmem, const void *coefT, const double *phib,
                  long long stride, long long step0, int nsteps, cudaStream_t st) {
    const long long n = (long long)nmem * nsteps * 2 * lbk::wmax(B);
    lbk::k_wave_ends<T, B><<<(unsigned)((n + 127) / 128), 128, 0, st>>>((T *)ends, segs, members, nmem, (const T *)coefT, phib, stride,
                                                                       step0, nsteps);
    if (cudaGetLastError() != cudaSuccess) return LBHPDE_ERR_CUDA;
    return LBHPDE_OK;
}

}  // namespace

int launch_wave_f32(const void *a);
int launch_wave_f64(const void *a);

#if LBH_WAVE_ESZ == 4
int launch_wave_f32(const void *a) { return launch_wave_b<float>(*(const WaveArgs *)a); }
#else
int launch_wave_f64(const void *a) { return launch_wave_b<double>(*(const WaveArgs *)a); }

namespace {
int wave_dispatch(const WaveArgs &a) { return a.p->esz == 4 ? launch_wave_f32(&a) : launch_wave_f64(&a); }
}  // namespace

int launch_wave(const PackedWave &p, const lbk::WaveWin *wins, unsigned char *box, unsigned *ctrl, void *st, const void *coefT,
                int nsteps, const void *ends, cudaStream_t stream) {
    if (nsteps <= 0) return LBHPDE_OK;
    const WaveArgs a{&p, wins, box, ctrl, st, st, coefT, nsteps, ends, stream, nullptr};
    return wave_dispatch(a);
}

int launch_wave_ends(const PackedWave &p, void *ends, const lbk::Seg *segs, const int *members, const void *coefT,
                     const double *phib, long long stride, long long step0, int nsteps, cudaStream_t st) {
    if (p.esz == 4)
        return p.b == 5 ? launch_ends_t<float, 5>(ends, segs, members, p.nmem, coefT, phib, stride, step0, nsteps, st)
                        : launch_ends_t<float, 7>(ends, segs, members, p.nmem, coefT, phib, stride, step0, nsteps, st);
    return p.b == 5 ? launch_ends_t<double, 5>(ends, segs, members, p.nmem, coefT, phib, stride, step0, nsteps, st)
                    : launch_ends_t<double, 7>(ends, segs, members, p.nmem, coefT, phib, stride, step0, nsteps, st);
}

bool pack_wave(const std::vector<lbk::Seg> &m, int b, int K, int G, int T, int csize, std::vector<lbk::WaveWin> &out) {
    out.clear();
    const int W = lbk::wmax(b), H = T * W, cap = lbk::wave_positions(K, G), room = csize * lbk::kWaveWarps;
    int used = 0;  // windows in the open cluster
    for (size_t mi = 0; mi < m.size(); ++mi) {
        const lbk::Seg &s = m[mi];
        const bool nee = s.pad > 0;
        // own nodes of an inner window, of the two at the ends of a bounded grid, of a single one
        const int vin = cap - 2 * H, vend = nee ? cap - H : vin, vone = nee ? cap : vin;
        long long nw = 1;
        if (s.N > vone) {
            if (vin < 1) return false;
            nw = nee ? 2 + std::max<long long>(0, ((long long)s.N - 2 * vend + vin - 1) / vin) : ((long long)s.N + vin - 1) / vin;
        }
        if (nw > (csize > 0 ? room : 1 << 16)) return false;
        if (csize > 0) {
            if (used + nw > room) {  // the next cluster
                out.resize((out.size() + room - 1) / room * room);
                used = 0;
            }
            used += (int)nw;
        }
        const int w0 = (int)out.size();
        long long at = 0;
        for (long long i = 0; i < nw; ++i) {
            const bool lend = nee && i == 0, rend = nee && i == nw - 1;
            // nodes in equal parts, the end windows taking up to H more each
            long long V;
            if (nw == 1) {
                V = s.N;
            } else {
                const long long extra = nee ? std::min<long long>(H, s.N / (2 * nw)) : 0;
                const long long inner = s.N - 2 * extra;
                V = inner * (i + 1) / nw - inner * i / nw + ((lend || rend) ? extra : 0);
            }
            if (V > (lend && rend ? vone : (lend || rend ? vend : vin))) return false;
            // the copies a neighbour takes come from this window alone, and are inner nodes; an end's
            // extrapolation node belongs to the window; no lane holds copies of both sides
            if (nw > 1 && V < H + ((lend || rend) ? W : 0)) return false;
            if (!nee && (V < H || V < K)) return false;
            if (V < K && !(lend && rend)) return false;
            if ((lend || rend) && V < W + s.pad) return false;
            lbk::WaveWin I{};
            I.off = s.off;
            I.ld = s.ld;
            I.N = s.N;
            I.D = s.D;
            I.gcoef = s.coef;
            I.vlo = lend ? 0 : H;
            I.vhi = I.vlo + (int)V;
            I.x0 = (int)(at - I.vlo);
            I.left = lend ? -1 : w0 + (int)(i == 0 ? nw - 1 : i - 1);
            I.right = rend ? -1 : w0 + (int)(i == nw - 1 ? 0 : i + 1);
            I.mi = (int)mi;
            I.depth = s.pad;
            I.A = s.A;
            I.Dg = s.Dg;
            I.nu = s.nu;
            out.push_back(I);
            at += V;
        }
    }
    const int per = (csize > 0 ? csize : 1) * lbk::kWaveWarps;
    out.resize((out.size() + per - 1) / per * per);  // whole CTAs and clusters; the places left over are unused
    return true;
}

namespace {

// What a step costs, in SM clocks (GB300, sweeps of 64 to 250 000 nodes over every form below): a
// window alone on its scheduler takes `a` a step and X a trade (Xg through L2, Xc inside a
// cluster), so a + X / T; the ends of a bounded grid take `end` more.  FP64: a is the FP64
// instruction count times 64 plus the shuffles.  FP32: latency, and instruction issue at K = 4.  With
// q windows on a scheduler: q a and, in FP64, whose trades then hide, 0.4 X / T.
struct WaveForm {
    int esz, b, K, G;
    double a, Xg, Xc, end;
};
const WaveForm kWaveForms[] = {
    {8, 5, 1, 4, 800, 1400, 800, 650},    {8, 5, 1, 2, 1350, 1500, 700, 850},   {8, 5, 1, 1, 2270, 1200, 600, 850},
    {8, 5, 2, 1, 4480, 2100, 950, 900},   {8, 7, 1, 3, 1750, 1750, 850, 650},   {8, 7, 1, 2, 2400, 1900, 870, 930},
    {8, 7, 1, 1, 4000, 1800, 650, 1150},  {8, 7, 2, 1, 8150, 2450, 1290, 1150}, {4, 5, 1, 1, 115, 1650, 600, 330},
    {4, 5, 2, 1, 180, 2030, 780, 330},    {4, 5, 4, 1, 270, 2000, 940, 400},    {4, 7, 1, 1, 190, 1620, 600, 450},
    {4, 7, 2, 1, 215, 2250, 920, 480},    {4, 7, 4, 1, 480, 2500, 1150, 650},
};
// A real exponent's power and rows on top of that: K = 2 in FP32 (unrolled row shapes, others),
// K = 1 in FP64.
constexpr double kWaveReal32 = 450, kWaveReal32Any = 3000, kWaveReal64 = 8500;

// FP operations of a step and node
double wave_ops(int b, int D) { return (b - 1) * (D + 1 + 2) + 1; }

struct WavePick {
    int K, G, T, C;
    double cost;
};

// windows of one member (as pack_wave), 0: it does not divide that way
long long wave_windows(const lbk::Seg &s, int W, int cap, int T) {
    const int H = T * W, vin = cap - 2 * H;
    const bool nee = s.pad > 0;
    if (nee && s.N <= cap) return 1;
    if (vin < 1) return 0;
    return nee ? 2 + std::max<long long>(0, ((long long)s.N - 2 * (cap - H) + vin - 1) / vin) : ((long long)s.N + vin - 1) / vin;
}

}  // namespace

namespace {

// A step of k_ring on the members it holds (FP32 D1Q5), in SM clocks, by the plan it gets (GB300).  Whole
// waves and a tail: 3400 a wave.  CTAs by size class, four of 128 threads an SM, two of 256 or one of 512:
// by the warps of the fullest SM's schedulers, one to four [107 members of 1095 nodes, a CTA on an SM,
// 1600; 249 of 1635, two, 1760; 318 CTAs of 960 nodes, three, 2540; 565 of 1287, four, 2740; 85 of 4021
// in CTAs of 256 threads 2050, 231 of 2710 2290; 107 of 4184 in CTAs of 512 2600, 81 of 6638 3260].  A
// warp takes the writes past its members' ends once for each remainder of 16 [1318 members of 43 to 173
// nodes 3930, 431 of 133 to 534 2600, 303 of 455 to 1821 2080; equal members of any size 1600 to 1700].
double ring_cost(const std::vector<lbk::Seg> &m, int sms) {
    std::vector<Member> res, cls[kRingClasses];
    long long nodes = 0;
    bool equal = true;
    for (const lbk::Seg &s : m)
        if (s.N <= 512 * kRingK) {
            res.push_back(Member{s, 0, 1});
            nodes += s.N;
            equal = equal && s.N % kRingK == res[0].seg.N % kRingK;
        }
    if (res.empty()) return 0;
    const double waves = nodes / (512.0 * kRingK * sms), rest = waves - std::floor(waves);
    if (waves >= 1) return 3400 * (std::floor(waves) + (rest > 0.25 ? 1.0 : (rest > 0 ? 0.6 : 0.0)));
    split_ring_classes(4, 5, kRingK, res, cls);
    std::vector<int> load(sms, 0);  // warps, the largest CTAs first, each to the emptiest SM (a heap)
    for (int c = kRingClasses - 1; c >= 0; --c) {
        Packed p;
        if (cls[c].empty() || pack_ring(5, 4, kRingK, 5, cls[c], p, ring_class_threads(4, 5, kRingK, c)) != LBHPDE_OK) continue;
        long long thr = 0;
        for (const lbk::OnchipInst &I : p.insts) thr += I.nthr;
        const int warps = (int)((thr + 32LL * p.ncta() - 1) / (32LL * p.ncta()));
        for (int i = 0; i < p.ncta(); ++i) {
            std::pop_heap(load.begin(), load.end(), std::greater<int>());
            load.back() += warps;
            std::push_heap(load.begin(), load.end(), std::greater<int>());
        }
    }
    const int most = *std::max_element(load.begin(), load.end());
    const double part[5] = {0, 1650, 1950, 2600, 3300};
    const double ends = equal ? 0.0 : (150 + 480 * 512.0 * res.size() / nodes) * std::max(1, most / 16);
    // (what does not fit at once starts as the first CTAs end [612 CTAs of 128 threads 4360, 369 of 256 4490])
    return most / 16 * part[4] + (most > 16 ? 0.65 : 1.0) * part[(most % 16 + 3) / 4] + ends;
}

}  // namespace

// The step of the CTA-wide kernels on a group's members, in SM clocks (GB300; measured in brackets).
//   A CTA alone: a barrier and an exchange, then its nodes at the rate of one SM (KdV on 400 nodes
//   [580 FP32, 8080 FP64], 2048-node FP64 windows [36 200]).
//   FP32 windows: D1Q5 650 and then 7.2e11 node-updates/s (real exponents: 450, 6.3e11 of their operations) [616 000 nodes 2470, 10^6 3670, 1.32 10^6 4310,
//   2^21 6390], D1Q7 1840 a wave of 152 windows [400 000 nodes 3620, 10^6 7060].
//   FP32 D1Q5 residents of a group that fills the GPU: ring_cost; windows beside them overlap.
//   Bounded: 601 nodes FP64 [16 400 D1Q5, 29 800 D1Q7], FP32 D1Q7 [2400]; streamed, two launches a
//   step: FP64 [55 000, 84 900], FP32 [23 400, 29 700].
double cta_cost(size_t esz, int b, int dc, bool nee, bool real, const std::vector<lbk::Seg> &m, int sms) {
    int D = 0;
    long long total = 0;
    for (const lbk::Seg &s : m) {
        D = std::max(D, s.D);
        total += s.N;
    }
    const double ops = wave_ops(b, dc > 0 ? dc : D), rate = esz == 8 ? 2.0 / 1.08 : 128.0 / 1.35;
    const bool q5 = esz == 4 && b == 5, ring = q5 && dc >= 0 && !nee && total >= 32LL * kRingK * sms;
    const int cap = esz == 8 ? (b == 5 ? 2048 : 1024) : (ring ? 512 * kRingK : (b == 5 ? 4096 : 2048));
    const int window = q5 ? 1024 : cap;
    double worst = 0, resident = 0, windows = 0;
    for (const lbk::Seg &s : m) {
        double t;
        if (nee && s.N > kBoundedK * kBoundedMaxT)
            t = esz == 8 ? (b == 5 ? 55000 : 84900) : (b == 5 ? 23400 : 29700);
        else if (nee)
            t = s.N * ops / rate + (esz == 8 ? (b == 5 ? 5600 : 10000) : 1500);
        else if (real && esz == 8)
            t = 94000;  // streamed [45 us a step at 100 nodes, 65 at 1000 to 50 000]
        else
            t = (s.N <= cap ? s.N : window) * ops / rate + (esz == 8 ? 1500 : 520) + (real ? 1200 : 0);
        (s.N <= cap || nee ? resident : windows) += s.N;
        worst = std::max(worst, t);
    }
    double all = (resident + windows) * ops / (rate * sms);
    if (esz == 4 && !nee) {
        // (a degree k_ring has not compiled takes single multiply-adds)
        const double res = ring ? ring_cost(m, sms) * ops / wave_ops(5, 5) * (dc == 5 ? 1.0 : 1.5) : resident * ops / (60.0 * sms);
        const double win = windows == 0 ? 0 : (b == 5 ? (real ? 450 + windows * ops / (66.0 * sms) : 650 + windows * ops / (75.0 * sms)) : 1840 * std::ceil(windows / (1856.0 * sms)) * ops / wave_ops(7, 7));
        all = ring ? std::max({res, win, res > 0 && win > 0 ? 0.6 * res + 0.9 * win : 0.0}) : res + win;
        if (ring) worst = 0;  // (ring_cost has it)
    }
    return std::max(worst, all);
}

// A step of k_strip: one warp on a scheduler, two, and every further wave of two (GB300: D1Q5 400 000
// nodes 2200, 800 000 3500, 2^24 37 800; D1Q7 400 000 2840, 800 000 4800, 2^24 75 400), and more where
// warps hold several segments or move nodes singly (D1Q5, warps of one or two equal members 2200, of three
// or of unequal ones 2470, of four 2730).
double strip_cost(const PackedStrip &p, int sms) {
    const int b = p.b, AA = p.AA, DG = p.DG, nwarps = p.nwarps();
    bool unequal = false;
    for (const lbk::StripSeg &S : p.segs) unequal = unequal || (S.N - p.segs[0].N) % 4 != 0;
    const double held = p.nmix() ? (double)(p.segs.size() - p.nfull) / p.nmix() : 0.0;  // segments of a mixed warp
    const double mix = b == 5 ? 270 * std::max({held - 2, unequal ? 1.0 : 0.0, 0.0}) : 0.0;
    const double s = AA > 0 ? (DG == 1 ? 2.0 : 4.9) : wave_ops(b, DG) / wave_ops(b, b == 5 ? 5 : 7);  // the power and the rows (2^24 nodes: 76 000 and 180 000)
    const double one = AA > 0 ? s * 2100 : (b == 5 ? s * (2200 + mix) : s * 2840), two = AA > 0 ? s * 3440 : (b == 5 ? s * (3480 + 0.4 * mix) : s * 4800), more = s * (b == 5 ? 2570 : 3620);
    const double waves = nwarps / (8.0 * sms);
    if (waves <= 0.5) return one;
    if (waves <= 1.0) return two;
    const double full = std::floor(waves), rest = waves - full;
    return two + (full - 1) * more + (rest == 0 ? 0.0 : (rest <= 0.5 ? 0.54 * more : more));
}

namespace {

// The forms, depths and placements of k_wave for a batch, and the modelled cost of a step of each.
std::vector<WavePick> wave_picks(size_t esz, int b, int dc, bool nee, const std::vector<lbk::Seg> &m, int sms) {
    const int W = lbk::wmax(b);
    int D = 0;
    bool real = false, fixed = true;
    for (const lbk::Seg &x : m) {
        D = std::max(D, x.D);
        real = real || x.A > 0;
        if (x.A > 0 && !lbk::wave_fixed_rows(b, x.A, x.Dg)) fixed = false;
    }
    // (the forms' costs are those of degree 5 on D1Q5, 7 on D1Q7)
    const double scale = real ? 1.0 : wave_ops(b, dc > 0 ? dc : D) / wave_ops(b, b == 5 ? 5 : 7);
    std::vector<WavePick> picks;
    for (const WaveForm &f : kWaveForms) {
        if (f.esz != (int)esz || f.b != b) continue;
        if (dc <= 0 && (f.G > 1 || f.K != (esz == 4 ? 2 : 1))) continue;
        for (int T : {1, 2, 3, 4, 6, 8, 12, 16})
            for (int C : {0, 1, 2, 4, 8, 16}) {
                long long ctas = 0, used = 0;
                const long long room = (long long)C * lbk::kWaveWarps;
                bool ok = true;
                for (const lbk::Seg &x : m) {
                    const long long nw = wave_windows(x, W, lbk::wave_positions(f.K, f.G), T);
                    ok = ok && nw > 0 && (C == 0 || nw <= room);
                    if (!ok) break;
                    if (C > 0 && used + nw > room) {
                        ctas += C;
                        used = 0;
                    }
                    used += nw;
                }
                if (!ok) continue;
                ctas += C > 0 ? C : (used + lbk::kWaveWarps - 1) / lbk::kWaveWarps;
                // clusters are placed in whole processing clusters: fewer SMs hold them
                const long long q = (ctas + (C > 1 ? sms * 4 / 5 : sms) - 1) / (C > 1 ? sms * 4 / 5 : sms);
                if (q > 4) continue;
                const double X = (C > 0 ? f.Xc + (nee ? 300 : 0) : f.Xg) * (q > 1 && esz == 8 ? 0.4 : 1.0);
                const double extra = (nee ? f.end : 0) + (real ? (esz == 8 ? kWaveReal64 : (fixed ? kWaveReal32 : kWaveReal32Any)) : 0);
                picks.push_back(WavePick{f.K, f.G, T, C, q * (f.a * scale + extra) + X / T});
            }
    }
    return picks;
}

}  // namespace

double wave_cost(size_t esz, int b, int dc, bool nee, const std::vector<lbk::Seg> &m, int sms) {
    double least = HUGE_VAL;
    for (const WavePick &k : wave_picks(esz, b, dc, nee, m, sms)) least = std::min(least, k.cost);
    return least;
}

bool plan_wave(size_t esz, int b, int dc, bool nee, const std::vector<lbk::Seg> &m, int sms, PackedWave &out) {
    out = PackedWave{};
    long long total = 0;
    int D = 0;
    bool real = false;
    for (const lbk::Seg &x : m) {
        total += x.N;
        D = std::max(D, x.D);
        real = real || x.A > 0;
    }
    if (total > (1 << 19)) return false;  // the other kernels fill the GPU
    std::vector<WavePick> picks = wave_picks(esz, b, dc, nee, m, sms);
    std::stable_sort(picks.begin(), picks.end(), [](const WavePick &x, const WavePick &y) { return x.cost < y.cost; });
    double other = cta_cost(esz, b, dc, nee, real, m, sms);
    int AA = 0, DG = 0;
    if (!nee && strip_ok(esz, b, dc, m, &AA, &DG)) {
        PackedStrip p;
        pack_strip(b, AA, DG, m, p);
        other = std::min(other, strip_cost(p, sms));
    }
    for (const WavePick &k : picks) {
        if (k.cost > 0.85 * other) return false;
        out.esz = (int)esz;
        out.b = b;
        out.dc = dc;
        out.nee = nee;
        out.K = k.K;
        out.G = k.G;
        out.tblk = k.T;
        out.csize = k.C;
        out.nmem = (int)m.size();
        out.cost = k.cost;
        out.other = other;
        if (!pack_wave(m, b, k.K, k.G, k.T, k.C, out.wins)) continue;
        out.nused = (int)std::count_if(out.wins.begin(), out.wins.end(), [](const lbk::WaveWin &w) { return w.N > 0; });
        out.wsmem = ((nee ? lbk::wave_end_elems(b, k.T) : 0) + (dc > 0 ? 0 : lbk::wave_coef_elems(b, D)) + 3) & ~3;
        const size_t boxes = (size_t)lbk::wave_box_bytes((int)esz, b, k.K, k.G);
        out.smem = (size_t(out.wsmem) * esz + (k.C > 0 ? boxes : 0)) * lbk::kWaveWarps;
        out.box_bytes = k.C > 0 ? 0 : boxes * out.wins.size();
        if (out.smem > kMaxSmem) continue;
        int room = 0;
        WaveArgs a{};
        a.p = &out;
        a.room = &room;
        if (wave_dispatch(a) != LBHPDE_OK) continue;
        if (k.C > 0 ? room > 0 : out.ncta() <= (long long)room * sms) return true;
    }
    return false;
}
#endif

}  // namespace lbh
