// Small and medium grids spread over the GPU (a2-a6, many steps per launch): each warp advances a
// window of one instance on its own, by warp shuffles, and trades the window's borders with its two
// neighbours every few steps.
//
// A grid that does not fill the GPU is bound by the latency of one step after another, not by any
// rate: in one CTA (k_onchip) a step pays shared-memory stores, a CTA barrier and loads, and, in
// double precision, the FP64 lanes of a single SM (two multiply-adds a clock, half a one for each of
// its four schedulers).  Here a window of 32 K positions belongs to one warp, and windows go to as
// many schedulers as there are.  A window holds its instance's nodes [x, x + V) and, on either side,
// copies of the H = T max|e| nodes next to them.  For T steps the warp needs no other warp: a stale
// edge value moves inward max|e| positions a step and so stays inside the copies.  Then the windows
// trade the H nodes next to each cut.
//
// In FP64 a multiply-add holds its scheduler's FP64 lanes for 64 cycles whatever the number of
// active lanes, so a window may be narrower and its populations split over G groups of 32 / G lanes:
// each lane then relaxes (B - 1) / G of a node's populations (all groups carry its phi), which cuts
// the FP64 instructions of a step from 33 to 19 (D1Q5, G = 2) or from 61 to 34 (D1Q7).
//
// A trade writes into boxes of the reader: every 32-bit half of a value travels in one 8-byte word
// beside the trade's number, so a reader knows a word is the awaited one from the word itself, and
// no fence, flag or barrier is needed.  Boxes are double buffered by the parity of the trade's
// number: a window writes trade i + 2 only after it has read its neighbours' i + 1, which they wrote
// after reading i.  Two places for the boxes:
//   cluster: all windows of an instance sit in one thread-block cluster, and a box lies in the
//     reader's shared memory (the writer stores through distributed shared memory, the reader polls
//     its own).  Clusters are independent of one another.
//   grid: boxes in global memory (L2), for instances over as many SMs as they take.  All windows
//     must be on the GPU together (a cooperative launch).  The trades' numbers run on from launch to
//     launch in device memory (ctrl[0]), so a captured launch can be replayed.  A window reads its
//     first copies from the state that its neighbours overwrite at the end: a fence before its first
//     trade and one after its last make every such read come before the write.
// Every wait is bounded: a window whose wait runs out marks ctrl[2], takes no further step, trades
// nothing more and writes NaN.  Its neighbours wait for its next trade in vain and do the same, so
// no value of a solve that a window has left counts as a result, and the readouts report it.
//
// The update of a node is that of k_onchip and k_stream (and, at the ends of a bounded grid, of
// k_bounded and k_nee_fix) operation by operation, so every result is theirs bit for bit.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbhpde_kernels.cuh"

namespace lbk {

struct WaveWin {
    long long off, ld;  // placement of the instance's state (as Seg)
    int N, D;           // N = 0: an unused place of a cluster
    int gcoef;          // coefficient block in global memory (as Seg::coef)
    int x0;             // node of position 0 (periodic: may be negative, taken modulo N)
    int vlo, vhi;       // own positions [vlo, vhi): traded at the cuts and written back
    int left, right;    // the windows next to this one (periodic: may be itself); -1: a grid end
    int mi, depth;      // bounded: member index among the plan's, extrapolation depth
    int A, Dg;          // real exponents (as Seg)
    double nu;
};

constexpr int kWaveWarps = 4;            // windows a CTA: one per scheduler
#ifndef LBK_WAVE_WAIT_LIMIT  // (a test of a wait that runs out compiles the kernel with fewer)
#define LBK_WAVE_WAIT_LIMIT (1 << 22)
#endif
constexpr int kWaveWaitLimit = LBK_WAVE_WAIT_LIMIT;  // polls of a wait, at most (seconds)

// One traded value: 8 bytes in FP32 (value, number), 16 in FP64 (half, number, half, number).
// Generic addresses: global memory or (distributed) shared memory.  Predicated, not branched: most
// lanes take part in a few of the accesses of a trade only.
template <typename T> struct WaveWord;
template <> struct WaveWord<float> {
    static constexpr int kBytes = 8;
    static __device__ __forceinline__ void put(bool on, unsigned char *p, float x, unsigned tag) {
        const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(x);
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %0, 0;\n\t@q st.relaxed.gpu.u64 [%1], %2;\n\t}" ::"r"((int)on),
                     "l"(p), "l"(w)
                     : "memory");
    }
    // x stays as it is and the answer is true where `on` is false
    static __device__ __forceinline__ bool get(bool on, const unsigned char *p, float &x, unsigned tag) {
        unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(x);
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %1, 0;\n\t@q ld.relaxed.gpu.u64 %0, [%2];\n\t}"
                     : "+l"(w)
                     : "r"((int)on), "l"(p)
                     : "memory");
        x = __uint_as_float((unsigned)w);
        return (unsigned)(w >> 32) == tag;
    }
};
template <> struct WaveWord<double> {
    static constexpr int kBytes = 16;
    static __device__ __forceinline__ void put(bool on, unsigned char *p, double x, unsigned tag) {
        const unsigned long long t = (unsigned long long)tag << 32, b = (unsigned long long)__double_as_longlong(x);
        const unsigned long long lo = t | (unsigned)b, hi = t | (unsigned)(b >> 32);
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %0, 0;\n\t@q st.relaxed.gpu.v2.u64 [%1], {%2, %3};\n\t}" ::"r"((int)on),
                     "l"(p), "l"(lo), "l"(hi)
                     : "memory");
    }
    static __device__ __forceinline__ bool get(bool on, const unsigned char *p, double &x, unsigned tag) {
        const unsigned long long t = (unsigned long long)tag << 32, b = (unsigned long long)__double_as_longlong(x);
        unsigned long long lo = t | (unsigned)b, hi = t | (unsigned)(b >> 32);
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t@q ld.relaxed.gpu.v2.u64 {%0, %1}, [%3];\n\t}"
                     : "+l"(lo), "+l"(hi)
                     : "r"((int)on), "l"(p)
                     : "memory");
        x = __longlong_as_double((long long)((hi << 32) | (unsigned)lo));
        return (unsigned)(lo >> 32) == tag && (unsigned)(hi >> 32) == tag;
    }
};

// Positions of a window, the pitch of a box row (H < half the positions, since own nodes remain) and
// the bytes of a window's boxes: two parities, two sides, b rows.
__host__ __device__ constexpr int wave_positions(int K, int G) { return 32 / G * K; }
__host__ __device__ constexpr int wave_pitch(int K, int G) { return wave_positions(K, G) / 2; }
__host__ __device__ constexpr int wave_box_bytes(int esz, int b, int K, int G) { return 4 * b * wave_pitch(K, G) * 2 * esz; }
// Row shapes of real-exponent models with unrolled code in k_wave.
__host__ __device__ constexpr bool wave_fixed_rows(int b, int A, int Dg) { return b == 5 ? A == 4 && (Dg == 1 || Dg == 5) : A == 6 && Dg == 1; }
// Coefficients staged in shared memory per window where the degree is known at run time only:
// P_j and f^eq_j rows of D + 1.
__host__ __device__ constexpr int wave_coef_elems(int b, int D) { return 2 * (b - 1) * (D + 1); }
// phi_b and f^eq_j(phi_b) of the steps between two trades, for the two ends: [T][2W][B]
__host__ __device__ constexpr int wave_end_elems(int b, int tblk) { return tblk * 2 * wmax(b) * b; }

// The relaxation of a lane's populations for a real-exponent model whose row count (AA + 1) and row
// degree DG are known at compile time (as relax_rows); false for other shapes.
template <typename T, int JG, int K, int AA, int DG>
__device__ __forceinline__ bool wave_rows(int A, int Dg, const T *r, int pitch, const T (&phi)[K], const T (&w)[K],
                                          T (&v)[JG][K], T omw) {
    if (A != AA || Dg != DG) return false;
#pragma unroll
    for (int i = 0; i < JG; ++i) {
        T acc[K];
        gen_evalN<T, DG, K, AA>(r + i * pitch, AA, DG, phi, w, acc);
#pragma unroll
        for (int k = 0; k < K; ++k) v[i][k] = fma_t(omw, v[i][k], acc[k]);
    }
    return true;
}

// phi_b and f^eq_j(phi_b), j = 1..B-1, of nsteps steps of every bounded member, ends[member][step]
// [2W][B], ahead of a k_wave launch: they depend on the prescribed values only, and inside k_wave
// they would hold up the two windows that every other one waits for.
template <typename T, int B>
__global__ void k_wave_ends(T *__restrict__ ends, const Seg *__restrict__ segs, const int *__restrict__ members, int nmem,
                            const T *__restrict__ coefs, const double *__restrict__ phib, long long stride,
                            long long step0, int nsteps) {
    constexpr int W = wmax(B);
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long per = (long long)nsteps * (2 * W);
    if (q >= per * nmem) return;
    const int m = members[q / per];
    const Seg s = segs[m];
    const T x = (T)phib[(long long)m * stride + step0 * (2 * W) + q % per];
    const T *fe = coefs + s.coef + (B - 1) * (s.D + 1);
    const T w = s.A > 0 ? nu_pow<T>(x, s.nu) : T(0);
    ends[q * B] = x;
#pragma unroll
    for (int j = 1; j < B; ++j) {
        const T *c = fe + (j - 1) * (s.D + 1);
        T acc;
        if (s.A > 0) {
            acc = gen_eval<T>(c, s.A, s.Dg, x, w);
        } else {
            acc = c[s.D];
            for (int p = s.D - 1; p >= 0; --p) acc = fma_t(acc, x, c[p]);
        }
        ends[q * B + j] = acc;
    }
}

// nused: windows with N > 0; tblk: steps between trades; csize: CTAs of a cluster (0: boxes in global memory at `box`, numbers
// from ctrl).  Dynamic shared memory: the CTA's boxes (cluster), then per window wsmem elements: the
// ends' values (NEE) and the coefficient rows (DC <= 0).
template <typename T, int B, int K, int G, int DC, bool NEE>
__global__ void __launch_bounds__(32 * kWaveWarps)
    k_wave(const T *st_in, T *st_out, const WaveWin *__restrict__ wins, int nused, const T *__restrict__ coefs,
           unsigned char *box, unsigned *ctrl, int nsteps, int tblk, int csize, const T *__restrict__ endtab, int wsmem) {
    static_assert(G == 1 || (K == 1 && (B - 1) % G == 0), "split windows hold one position a lane");
    constexpr int W = wmax(B);
    constexpr int NC = DC > 0 ? DC + 1 : 1;
    constexpr int JG = (B - 1) / G;   // populations of a lane: j = 1 + g JG + i
    constexpr int P = 32 / G;         // lanes of a group
    constexpr int PITCH = wave_pitch(K, G);
    constexpr int WB = WaveWord<T>::kBytes;
    constexpr int SIDE = B * PITCH * WB;  // bytes of one side's box
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int w = blockIdx.x * kWaveWarps + wid;
    const WaveWin I = wins[w];  // one for every warp of the grid
    const bool used = I.N > 0;
    const int H = tblk * W;
    const int g = G > 1 ? lane / P : 0;
    const int pos = (G > 1 ? lane % P : lane) * K;  // first position of the lane
    const bool in = G == 1 || g < G;                // G = 3: two lanes are left over

    // this window's boxes and its neighbours' (each side's: two parities of B rows)
    unsigned char *mine, *tol, *tor;
    unsigned tag = 0;
    if (csize > 0) {
        unsigned char *const b0 = smem_raw + wid * (4 * SIDE);
        for (int q = lane; q < 4 * SIDE / 16; q += 32) reinterpret_cast<uint4 *>(b0)[q] = make_uint4(0, 0, 0, 0);
        mine = b0;
        auto of = [&](int win) -> unsigned char * {
            unsigned long long a = (unsigned long long)(smem_raw + (win % kWaveWarps) * (4 * SIDE)), r;
            asm("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(win / kWaveWarps % csize));
            return (unsigned char *)r;
        };
        tol = used && I.left >= 0 ? of(I.left) : mine;
        tor = used && I.right >= 0 ? of(I.right) : mine;
    } else {
        mine = box + (long long)w * (4 * SIDE);
        tol = used && I.left >= 0 ? box + (long long)I.left * (4 * SIDE) : mine;
        tor = used && I.right >= 0 ? box + (long long)I.right * (4 * SIDE) : mine;
        if (used) tag = *(volatile unsigned *)ctrl;
    }
    const unsigned base = tag;
    T *const ends = reinterpret_cast<T *>(smem_raw + (csize > 0 ? kWaveWarps * 4 * SIDE : 0)) + (size_t)wid * wsmem;
    T *const srow = ends + (NEE ? wave_end_elems(B, tblk) : 0);

    // coefficients of P_j in registers (compile-time degree, zero-padded), else in shared memory
    T c[JG][NC];
    const int crows = (B - 1) * (I.D + 1);
    if constexpr (DC > 0) {
#pragma unroll
        for (int i = 0; i < JG; ++i)
#pragma unroll
            for (int p = 0; p <= DC; ++p)
                c[i][p] = used && in && p <= I.D ? coefs[I.gcoef + (g * JG + i) * (I.D + 1) + p] : T(0);
    } else {
        if (used)
            for (int q = lane; q < 2 * crows; q += 32) srow[q] = coefs[I.gcoef + q];
        __syncwarp();
    }
    const T omw = used ? coefs[I.gcoef + 2 * crows] : T(0);
    // the ends of a bounded grid: lane l evaluates the f^eq row 1 + l % (B - 1)
    const int myrow = lane % (B - 1);
    T qr[NEE ? NC : 1];
    if constexpr (NEE && DC > 0) {
#pragma unroll
        for (int p = 0; p <= DC; ++p) qr[p] = used && p <= I.D ? coefs[I.gcoef + crows + myrow * (I.D + 1) + p] : T(0);
    }
    auto feq_mine = [&](T x) -> T {  // f^eq of this lane's row at x (as row_eval / gen_eval)
        if constexpr (DC > 0) {
            T acc = qr[DC];
#pragma unroll
            for (int p = DC - 1; p >= 0; --p) acc = fma_t(acc, x, qr[p]);
            return acc;
        } else {
            const T *r = srow + crows + myrow * (I.D + 1);
            if constexpr (DC < 0) {
                if (I.A > 0) return gen_eval<T>(r, I.A, I.Dg, x, nu_pow<T>(x, I.nu));
            }
            T acc = r[I.D];
            for (int p = I.D - 1; p >= 0; --p) acc = fma_t(acc, x, r[p]);
            return acc;
        }
    };

    // state of the lane's positions; positions outside the window and its copies are 0
    const int plo = I.left >= 0 ? I.vlo - H : I.vlo, pend = I.right >= 0 ? I.vhi + H : I.vhi;
    T phi[K], v[JG][K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int p = pos + k;
        const bool ok = used && in && p >= plo && p < pend;
        long long x = (long long)I.x0 + p;
        if (ok) {
            x %= I.N;
            x += x < 0 ? I.N : 0;
        }
        phi[k] = ok ? st_in[I.off + x] : T(0);
#pragma unroll
        for (int i = 0; i < JG; ++i) v[i][k] = ok ? st_in[I.off + (long long)(1 + g * JG + i) * I.ld + x] : T(0);
    }
    // split windows: the lane a population comes from (itself past the group's edge)
    int from[G > 1 ? JG : 1];
    if constexpr (G > 1) {
#pragma unroll
        for (int i = 0; i < JG; ++i) {
            const int q = pos - vel(1 + g * JG + i);
            from[i] = in && q >= 0 && q < P ? g * P + q : lane;
        }
    }

    // one step of every position of the window; s: the step since the last trade
    auto step = [&](int s) {
        T d[K];
#pragma unroll
        for (int k = 0; k < K; ++k) d[k] = T(0);
        if constexpr (G == 1) {
#pragma unroll
            for (int j = 1; j < B; ++j) {
                const int e = vel(j);
                T nv[K];
#pragma unroll
                for (int k = 0; k < K; ++k) {  // position p - e: register r of the lane `up` below or `dn` above
                    const int q = k - e;
                    if (q < 0) {
                        const int up = (-q + K - 1) / K;
                        nv[k] = __shfl_up_sync(0xffffffffu, v[j - 1][q + up * K], up);
                    } else if (q >= K) {
                        const int dn = q / K;
                        nv[k] = __shfl_down_sync(0xffffffffu, v[j - 1][q - dn * K], dn);
                    } else {
                        nv[k] = v[j - 1][q];
                    }
                }
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    d[k] += nv[k] - v[j - 1][k];
                    v[j - 1][k] = nv[k];
                }
            }
        } else {
            T df[JG];
#pragma unroll
            for (int i = 0; i < JG; ++i) {
                const T nv = __shfl_sync(0xffffffffu, v[i][0], from[i]);
                df[i] = nv - v[i][0];
                v[i][0] = nv;
            }
#pragma unroll
            for (int j = 1; j < B; ++j) d[0] += __shfl_sync(0xffffffffu, df[(j - 1) % JG], (j - 1) / JG * P + pos);
        }
#pragma unroll
        for (int k = 0; k < K; ++k) phi[k] += d[k];
        if constexpr (DC > 0) {
#pragma unroll
            for (int i = 0; i < JG; ++i) {
                if constexpr (std::is_same<T, float>::value && K % 2 == 0) {
                    float2 a2[K / 2];
#pragma unroll
                    for (int k = 0; k < K / 2; ++k) a2[k] = make_float2(c[i][DC], c[i][DC]);
#pragma unroll
                    for (int p = DC - 1; p >= 0; --p)
#pragma unroll
                        for (int k = 0; k < K / 2; ++k)
                            a2[k] = __ffma2_rn(a2[k], make_float2(phi[2 * k], phi[2 * k + 1]), make_float2(c[i][p], c[i][p]));
#pragma unroll
                    for (int h = 0; h < K / 2; ++h) {
                        const bool right = G == 1 && vel(1 + i) > 0;
                        const int k = right ? K / 2 - 1 - h : h;
                        if (right) v[i][2 * k + 1] = fma_t(omw, v[i][2 * k + 1], a2[k].y);
                        v[i][2 * k] = fma_t(omw, v[i][2 * k], a2[k].x);
                        if (!right) v[i][2 * k + 1] = fma_t(omw, v[i][2 * k + 1], a2[k].y);
                    }
                } else {
                    T acc[K];
#pragma unroll
                    for (int k = 0; k < K; ++k) acc[k] = c[i][DC];
#pragma unroll
                    for (int p = DC - 1; p >= 0; --p)
#pragma unroll
                        for (int k = 0; k < K; ++k) acc[k] = fma_t(acc[k], phi[k], c[i][p]);
#pragma unroll
                    for (int k = 0; k < K; ++k) v[i][k] = fma_t(omw, v[i][k], acc[k]);
                }
            }
        } else {
            T wp[K];
            bool real = false, relaxed = false;
            if constexpr (DC < 0) {
                real = I.A > 0;
                if (real) {
#pragma unroll
                    for (int k = 0; k < K; ++k) wp[k] = nu_pow<T>(phi[k], I.nu);
                    // the rows of class (1) with Pi_k = phi: n alone and with a quadratic term on
                    // D1Q5, n alone on D1Q7 (a run-time shape takes 1.9 us a step, these 0.36: FP32,
                    // 1000 nodes)
                    const T *r = srow + g * JG * (I.D + 1);
                    if constexpr (B == 5)
                        relaxed = wave_rows<T, JG, K, 4, 1>(I.A, I.Dg, r, I.D + 1, phi, wp, v, omw) ||
                                  wave_rows<T, JG, K, 4, 5>(I.A, I.Dg, r, I.D + 1, phi, wp, v, omw);
                    else
                        relaxed = wave_rows<T, JG, K, 6, 1>(I.A, I.Dg, r, I.D + 1, phi, wp, v, omw);
                }
            }
#pragma unroll
            for (int i = 0; i < JG && !relaxed; ++i) {
                const T *r = srow + (g * JG + i) * (I.D + 1);
                T acc[K];
                if (real) {
                    gen_evalN<T, -1, K>(r, I.A, I.Dg, phi, wp, acc);
                } else {
                    const T cD = r[I.D];
#pragma unroll
                    for (int k = 0; k < K; ++k) acc[k] = cD;
                    for (int p = I.D - 1; p >= 0; --p) {
                        const T cp = r[p];
#pragma unroll
                        for (int k = 0; k < K; ++k) acc[k] = fma_t(acc[k], phi[k], cp);
                    }
                }
#pragma unroll
                for (int k = 0; k < K; ++k) v[i][k] = fma_t(omw, v[i][k], acc[k]);
            }
        }
        if constexpr (NEE) {
            // the outer nodes of each grid end: the window that holds one holds its x_f too
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                if ((side ? I.right : I.left) >= 0) continue;  // uniform in the warp
                const int pf = (side ? I.N - W - I.depth : W - 1 + I.depth) - I.x0;
                const int src = pf / K, kf = pf % K;  // the lane of x_f (in its group), its register
                // lane l takes population 1 + l % (B - 1) of x_f, and with it the non-equilibrium part
                T ph = phi[0];
#pragma unroll
                for (int k = 1; k < K; ++k) ph = k == kf ? phi[k] : ph;
                const T f = feq_mine(__shfl_sync(0xffffffffu, ph, src));
                T vf = T(0);
#pragma unroll
                for (int i = 0; i < JG; ++i) {
                    T x = v[i][0];
#pragma unroll
                    for (int k = 1; k < K; ++k) x = k == kf ? v[i][k] : x;
                    x = __shfl_sync(0xffffffffu, x, myrow / JG * P + src);
                    vf = myrow % JG == i ? x : vf;
                }
                // lane (l, row) the rebuilt value of outer node l
                const T *e = ends + (s * 2 + side) * W * B;
                const int ol = lane < W * (B - 1) ? lane / (B - 1) : 0;
                const T val = e[ol * B + 1 + myrow] + (vf - f);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const int x = I.x0 + pos + k;
                    int l = side ? x - (I.N - W) : x;
                    const bool outer = in && l >= 0 && l < W;
                    l = outer ? l : 0;
                    phi[k] = outer ? e[l * B] : phi[k];
#pragma unroll
                    for (int i = 0; i < JG; ++i) {
                        const int r = G > 1 ? (in ? g * JG + i : 0) : i;
                        const T nv = __shfl_sync(0xffffffffu, val, l * (B - 1) + r);
                        v[i][k] = outer ? nv : v[i][k];
                    }
                }
            }
        }
    };
    // the ends' values of the next n steps into shared memory (asynchronous copies)
    const bool has_end = NEE && used && (I.left < 0 || I.right < 0);
    auto fetch_ends = [&](long long s0, int n) {
        if constexpr (NEE) {
            if (!has_end) return;
            __syncwarp();
            const T *src = endtab + ((long long)I.mi * nsteps + s0) * (2 * W * B);
            const unsigned dst = (unsigned)__cvta_generic_to_shared(ends);
            for (int q = lane; q < n * 2 * W * B; q += 32)
                asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst + q * (unsigned)sizeof(T)), "l"(src + q),
                             "n"((int)sizeof(T))
                             : "memory");
        }
    };
    auto ends_ready = [&] {
        if constexpr (NEE) {
            if (!has_end) return;
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
        }
    };

    // what this lane writes and reads in a trade: bit k of the masks; boxes are [parity][side][B][PITCH],
    // side 0 what came from the left neighbour, side 1 from the right
    unsigned publ = 0, pubr = 0, take = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int p = pos + k;
        const bool on = used && in;
        if (on && I.left >= 0 && p >= I.vlo && p < I.vlo + H) publ |= 1u << k;
        if (on && I.right >= 0 && p >= I.vhi - H && p < I.vhi) pubr |= 1u << k;
        if (on && ((I.left >= 0 && p < I.vlo && p >= plo) || (I.right >= 0 && p >= I.vhi && p < pend))) take |= 1u << k;
    }
    unsigned char *const wl = tol + SIDE + (pos - I.vlo + g * JG * PITCH) * WB;
    unsigned char *const wr = tor + (pos - (I.vhi - H) + g * JG * PITCH) * WB;
    const unsigned char *const rd =
        (pos < I.vlo && I.left >= 0 ? mine + (pos - plo) * WB : mine + SIDE + (pos - I.vhi) * WB) + g * JG * PITCH * WB;
    bool dead = false;
    auto trade = [&] {
        ++tag;
        const long long par = (tag & 1) ? 2 * SIDE : 0;
        // row 0 is phi; a group's rows follow it at g JG (row 0 of groups g > 0 is not theirs)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool l = publ >> k & 1, r = pubr >> k & 1;
            WaveWord<T>::put(l && (G == 1 || g == 0), wl + par + k * WB, phi[k], tag);
            WaveWord<T>::put(r && (G == 1 || g == 0), wr + par + k * WB, phi[k], tag);
#pragma unroll
            for (int i = 0; i < JG; ++i) {
                WaveWord<T>::put(l, wl + par + ((1 + i) * PITCH + k) * WB, v[i][k], tag);
                WaveWord<T>::put(r, wr + par + ((1 + i) * PITCH + k) * WB, v[i][k], tag);
            }
        }
        const unsigned char *const rp = rd + par;
        for (int tries = 0;; ++tries) {
            bool ok = true;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const bool t = take >> k & 1;
                ok &= WaveWord<T>::get(t, rp + k * WB - (G > 1 ? g * JG * PITCH * WB : 0), phi[k], tag);
#pragma unroll
                for (int i = 0; i < JG; ++i) ok &= WaveWord<T>::get(t, rp + ((1 + i) * PITCH + k) * WB, v[i][k], tag);
            }
            if (__all_sync(0xffffffffu, ok)) break;
            if (tries >= kWaveWaitLimit) {
                dead = true;  // uniform: the vote and the count are
                if (lane == 0) atomicExch(ctrl + 2, 1u);
                break;
            }
        }
    };
    auto cluster_sync = [&] {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    };

    // the lanes' accesses before it come before the lanes' after it, also as other windows see them
    auto fence = [&] {
        __syncwarp();
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        __syncwarp();
    };

    // every first copy is read before anybody writes over it: cluster: (every box is empty, too) by
    // the barrier; grid: before this window's first trade, which its neighbours await before they write
    if (csize > 0)
        cluster_sync();
    else
        fence();
    const bool alone = !used || (I.left < 0 && I.right < 0);  // a whole bounded grid: nothing to trade
    int done = 0;
    if (used) {
        fetch_ends(0, min(tblk, nsteps));
        // grid: the state is updated in place, so nobody may write before its neighbours have read
        // their first copies: at least one trade comes before
        if (csize == 0 && nsteps <= tblk && !alone) trade();
        while (done < nsteps && !dead) {
            const int n = min(tblk, nsteps - done);
            ends_ready();
            for (int s = 0; s < n; ++s) step(s);
            done += n;
            if (done < nsteps) {
                fetch_ends(done, min(tblk, nsteps - done));
                if (!alone) trade();
            }
        }
        ends_ready();  // (a window that gave up has copies under way)
        if (csize == 0) fence();  // the neighbours' trades, so their reads, come before these writes
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int p = pos + k;
            if (in && p >= I.vlo && p < I.vhi) {
                long long x = (long long)I.x0 + p;
                x %= I.N;
                x += x < 0 ? I.N : 0;
                if (g == 0) st_out[I.off + x] = dead ? T(NAN) : phi[k];
#pragma unroll
                for (int i = 0; i < JG; ++i) st_out[I.off + (long long)(1 + g * JG + i) * I.ld + x] = dead ? T(NAN) : v[i][k];
            }
        }
    }
    if (csize > 0) {
        cluster_sync();  // no CTA ends while a neighbour may still write into its boxes
    } else if (used) {
        // the last window to finish moves the trades' numbers on for the next launch, after every
        // window has read them (they all have before their fence above)
        if (lane == 0 && atomicAdd(ctrl + 1, 1u) == (unsigned)(nused - 1)) {
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            ctrl[1] = 0;
            ctrl[0] = base + (unsigned)((nsteps - 1) / tblk) + 1u;
        }
    }
}

}  // namespace lbk
