// Periodic FP32 grids that fill the GPU (a2-a6, several steps per launch): every warp advances a
// strip of 32 K positions on its own, by warp shuffles, for up to HL K / max|e| steps between one
// load from HBM and one store, with no barrier and no exchange through shared memory.
//
// The bound is the FP32 pipes (33 operations a node and step on D1Q5, 61 on D1Q7).  What held the
// CTA-wide kernels below 71% of them was not the barrier but the mix: a packed multiply-add takes
// both halves of a scheduler's FP32 pipes, a single one either half, and many warps at different
// places leave halves idle between the two (a copy of this kernel with 4 warps of 16 nodes a lane
// on a scheduler reached 70%, with 2 warps of 32 nodes 80%).  So a lane holds as many nodes as the
// registers take (K = 32 on D1Q5, 24 on D1Q7: 236 and 251 registers, no spills), 8 warps share an
// SM, and the CTA is one warp, so that one loads while the others compute.
//
// A strip is one or several segments: consecutive lanes that hold V own nodes of one instance, HL
// lanes of copies before and HL K nodes of copies after them (node x0 + p at position p, modulo N: the
// unrolled periodic grid).  The lane next to a segment's end reads what its neighbour lane happens
// to hold; a wrong value moves inward max|e| positions a step and stays inside the copies.  Long
// instances are cut into whole-warp segments; what is left of each (and short instances) shares
// warps with others, so that ragged sizes cost lanes, not warps.
//
// State goes between HBM and registers through shared memory (16-byte asynchronous copies,
// coalesced; rows of a lane at an odd 16-byte stride, so neither side has bank conflicts): direct
// 16-byte loads of a lane's own nodes, 128 bytes apart, were 14% slower on D1Q5.  Segments whose
// lanes wrap around the grid's end or end inside a 16-byte piece move those lanes' nodes singly.
//
// Each node's update is k_onchip's, operation by operation (bit for bit the same results).
// GB300: 2^24 nodes, 256 steps: D1Q5 9.3e11 node-updates/s (76% of the FP32 pipes; k_onchip's windows
// 7.0e11), D1Q7 4.6e11 (70%; 3.3e11); u^1.5 u_x (a power and five rows a node) 4.6e11 (3.9e11).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "lbhpde_kernels.cuh"

namespace lbk {

struct StripSeg {
    long long off, ld;  // placement of the instance's state (as Seg), the same in both buffers
    int N, D;
    int gcoef;          // coefficient block in global memory (as Seg::coef)
    int x0;             // node of the segment's position 0 (may be negative: taken modulo N)
    int vlo, vhi;       // own positions [vlo, vhi), written back; vlo = HL K
    int lane0, nlanes;  // lanes [lane0, lane0 + nlanes)
    float nu;           // real-exponent models: the exponent
};

constexpr int kStripSegs = 4;  // segments a warp, at most
// Models: AA = 0: f^eq of the compiled degree DC; AA > 0: real exponents, P_j = sum_{a<=AA} (phi^nu)^a
// sum_{i<=DG} c[a (DG + 1) + i] phi^i (D1Q5; the shapes of class (1) with Pi_k = phi).
__host__ __device__ constexpr int strip_K(int B, int AA) { return B == 5 ? 32 : 24; }
__host__ __device__ constexpr int strip_HL(int B) { return B == 5 ? 1 : 2; }
// steps a launch can take: the copies cover steps * max|e| nodes
__host__ __device__ constexpr int strip_steps(int B, int AA) { return strip_HL(B) * strip_K(B, AA) / wmax(B); }
// shared memory of a warp: the staging rows, then the coefficient rows of its segments (degree D, or
// (AA + 1)(DG + 1) - 1 for a flattened real-exponent row)
__host__ __device__ constexpr int strip_pitch(int K) { return K / 4 + 1; }  // 16-byte pieces of a lane
__host__ __device__ constexpr int strip_smem(int B, int AA, int D) {
    return (B * 32 * strip_pitch(strip_K(B, AA)) * 4 + kStripSegs * cblock(B, D)) * 4;
}

// One step of a lane's K nodes: pull from its own registers and the lanes beside it, phi, relaxation.
template <int B, int DC, int AA, int DG, int K, int CH>
__device__ __forceinline__ void strip_step(float (&phi)[K], float (&v)[B - 1][K], const float *c0, float omw, float nu) {
    constexpr int CS = crow(DC);
    float d[K];
#pragma unroll
    for (int k = 0; k < K; ++k) d[k] = -0.f;  // the identity of the addition: the first one folds away
#pragma unroll
    for (int j = 1; j < B; ++j) {
        const int e = vel(j), a = e > 0 ? e : -e;
        float(&u)[K] = v[j - 1];
        float in[3];  // what crosses the lane's edge
#pragma unroll
        for (int i = 0; i < a; ++i)
            in[i] = e > 0 ? __shfl_up_sync(0xffffffffu, u[K - a + i], 1) : __shfl_down_sync(0xffffffffu, u[i], 1);
        if (a == 2) {
            // the pair (k, k + 1) pulls from an aligned pair: difference and sum in one packed
            // operation each (a multiply-add by -1 rounds as the subtraction)
#pragma unroll
            for (int i = 0; i < K; i += 2) {
                const int k = e > 0 ? K - 2 - i : i, q = k - e;
                const float2 nv = q >= 0 && q < K ? make_float2(u[q], u[q + 1]) : make_float2(in[0], in[1]);
                const float2 df = __ffma2_rn(make_float2(u[k], u[k + 1]), make_float2(-1.f, -1.f), nv);
                const float2 dd = __fadd2_rn(make_float2(d[k], d[k + 1]), df);
                d[k] = dd.x, d[k + 1] = dd.y, u[k] = nv.x, u[k + 1] = nv.y;
            }
        } else {
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const int k = e > 0 ? K - 1 - i : i, q = k - e;
                const float nv = q < 0 ? in[q + a] : (q >= K ? in[q - K] : u[q]);
                d[k] += nv - u[k];
                u[k] = nv;
            }
        }
    }
#pragma unroll
    for (int k = 0; k < K; k += 2) {
        const float2 p2 = __fadd2_rn(make_float2(phi[k], phi[k + 1]), make_float2(d[k], d[k + 1]));
        phi[k] = p2.x, phi[k + 1] = p2.y;
    }
    float wp[AA > 0 ? K : 1];  // phi^nu
    if constexpr (AA > 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) wp[k] = nu_pow<float>(phi[k], nu);
    }
    // A right-moving population relaxes from its last node down, a left-moving one from its first
    // node up: node k's new value may then take the register that held k before the pull, whose old
    // value (a neighbour's source) has been used.  In ascending order for all, a move a node went
    // to the FP32 pipes (8.6e11 node-updates/s on D1Q5 against 9.3e11, 4.45e11 against 4.66e11 on D1Q7).
#pragma unroll
    for (int j = 1; j < B; ++j) {
        const float *c = c0 + (j - 1) * CS;
#pragma unroll
        for (int b0 = 0; b0 < K; b0 += CH) {
            const int i0 = vel(j) > 0 ? K - CH - b0 : b0;
            float2 acc[CH / 2];
            if constexpr (AA == 0) {
                const float cD = c[DC];
#pragma unroll
                for (int i = 0; i < CH / 2; ++i) acc[i] = make_float2(cD, cD);
#pragma unroll
                for (int p = DC - 1; p >= 0; --p) {
                    const float cp = c[p];
#pragma unroll
                    for (int i = 0; i < CH / 2; ++i)
                        acc[i] = __ffma2_rn(acc[i], make_float2(phi[i0 + 2 * i], phi[i0 + 2 * i + 1]), make_float2(cp, cp));
                }
            } else {
                // Horner in phi within a row, in w = phi^nu across rows (as gen_evalN)
#pragma unroll
                for (int a = AA; a >= 0; --a) {
                    float2 h[CH / 2];
                    const float cD = c[a * (DG + 1) + DG];
#pragma unroll
                    for (int i = 0; i < CH / 2; ++i) h[i] = make_float2(cD, cD);
#pragma unroll
                    for (int p = DG - 1; p >= 0; --p) {
                        const float cp = c[a * (DG + 1) + p];
#pragma unroll
                        for (int i = 0; i < CH / 2; ++i)
                            h[i] = __ffma2_rn(h[i], make_float2(phi[i0 + 2 * i], phi[i0 + 2 * i + 1]), make_float2(cp, cp));
                    }
#pragma unroll
                    for (int i = 0; i < CH / 2; ++i)
                        acc[i] = a == AA ? h[i] : __ffma2_rn(acc[i], make_float2(wp[i0 + 2 * i], wp[i0 + 2 * i + 1]), h[i]);
                }
            }
#pragma unroll
            for (int h = 0; h < CH / 2; ++h) {
                const int i = vel(j) > 0 ? CH / 2 - 1 - h : h;
                const int k0 = i0 + 2 * i;
                if (vel(j) > 0) v[j - 1][k0 + 1] = __fmaf_rn(omw, v[j - 1][k0 + 1], acc[i].y);
                v[j - 1][k0] = __fmaf_rn(omw, v[j - 1][k0], acc[i].x);
                if (vel(j) < 0) v[j - 1][k0 + 1] = __fmaf_rn(omw, v[j - 1][k0 + 1], acc[i].y);
            }
        }
    }
}

template <int B, int DC, int AA = 0, int DG = 0>
__global__ void __launch_bounds__(32, 8)
    k_strip(const float *__restrict__ st_in, float *__restrict__ st_out, const StripSeg *__restrict__ segs,
            const int *__restrict__ first, int nmix, const float *__restrict__ coefs, int nsteps) {
    constexpr int K = strip_K(B, AA), KQ = K / 4, PQ = strip_pitch(K);
    constexpr int CS = crow(DC), CB = cblock(B, DC);
    constexpr int CH = AA > 0 ? 8 : 4;  // nodes a Horner chunk (others: equal or 1% slower)
    static_assert(K % CH == 0 && CH % 2 == 0 && K <= 32, "packed pairs; a node a lane where a lane's nodes are moved singly");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *const stage = reinterpret_cast<float4 *>(smem_raw);  // [B][32][PQ]
    float *const sc = reinterpret_cast<float *>(stage + B * 32 * PQ);
    const int lane = threadIdx.x;
    // the first nmix warps hold several segments or a part of a warp (they take longest), the others
    // one whole segment each: warp nmix + i segment i
    const int w = blockIdx.x;
    // Where the lane's positions lie, looked up before the steps and again after them (the registers
    // belong to the state): its segment, first node, place of that in row 0, and whether its K nodes
    // are consecutive and on a 16-byte boundary.
    struct Place {
        int mine, x, N;
        long long at, ld;
        bool fast;
    };
    auto place = [&](int again) {
        const int s0 = w < nmix ? first[w + again] : w - nmix, ns = w < nmix ? first[w + 1 + again] - s0 : 1;
        Place q{-1, 0, 1, 0, 0, false};
        for (int s = 0; s < ns; ++s) {
            const StripSeg &S = segs[s0 + s + again];
            if (lane >= S.lane0 && lane < S.lane0 + S.nlanes) {
                q.mine = s;
                q.N = S.N;
                q.x = S.x0 + (lane - S.lane0) * K;
                if (q.x < 0 || q.x >= q.N) {
                    q.x %= q.N;
                    q.x += q.x < 0 ? q.N : 0;
                }
                q.at = S.off + q.x;
                q.ld = S.ld;
                q.fast = q.x + K <= q.N && (q.x & 3) == 0;
            }
        }
        return q;
    };
    float phi[K], v[B - 1][K];
    int mine;
    float nu = 1.f;
    {
    const Place pl = place(0);
    mine = pl.mine;
    const int x = pl.x, N = pl.N;
    const long long at = pl.at, ld = pl.ld;
    const bool fast = pl.fast;
    const unsigned sbase = (unsigned)__cvta_generic_to_shared(stage);
#pragma unroll
    for (int q = 0; q < KQ; ++q) {  // piece f of the strip belongs to lane f / KQ
        const int f = q * 32 + lane, L = f / KQ, r = f % KQ;
        const long long a = __shfl_sync(0xffffffffu, at, L), l = __shfl_sync(0xffffffffu, ld, L);
        if (__shfl_sync(0xffffffffu, (int)fast, L)) {
#pragma unroll
            for (int j = 0; j < B; ++j)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sbase + ((j * 32 + L) * PQ + r) * 16),
                             "l"(st_in + a + j * l + 4 * r)
                             : "memory");
        }
    }
    const int s0 = w < nmix ? first[w] : w - nmix, ns = w < nmix ? first[w + 1] - s0 : 1;
    if (AA > 0 && mine >= 0) nu = segs[s0 + mine].nu;
    for (int s = 0; s < ns; ++s) {  // (while the state is under way)
        const StripSeg &S = segs[s0 + s];
        for (int q = lane; q < (B - 1) * CS; q += 32) {
            const int j = q / CS, p = q % CS;
            sc[s * CB + q] = p <= S.D ? coefs[S.gcoef + j * (S.D + 1) + p] : 0.f;
        }
        if (lane == 0) sc[s * CB + (B - 1) * CS] = coefs[S.gcoef + 2 * (B - 1) * (S.D + 1)];
    }
    // the nodes of a lane that wraps or is not aligned: one a lane of the whole warp; idle lanes: 0
    for (unsigned m = __ballot_sync(0xffffffffu, mine >= 0 && !fast); m; m &= m - 1) {
        const int L = __ffs(m) - 1;
        const long long a = __shfl_sync(0xffffffffu, at, L), l = __shfl_sync(0xffffffffu, ld, L);
        const int xl = __shfl_sync(0xffffffffu, x, L), n = __shfl_sync(0xffffffffu, N, L);
        if (lane < K) {
            const int y = (xl + lane) % n;
#pragma unroll
            for (int j = 0; j < B; ++j)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sbase + (j * 32 + L) * PQ * 16 + lane * 4),
                             "l"(st_in + a - xl + y + j * l)
                             : "memory");
        }
    }
    if (mine < 0) {
#pragma unroll
        for (int j = 0; j < B; ++j)
#pragma unroll
            for (int q = 0; q < KQ; ++q) stage[(j * 32 + lane) * PQ + q] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
#pragma unroll
    for (int j = 0; j < B; ++j) {
        float *d = j ? v[j ? j - 1 : 0] : phi;
#pragma unroll
        for (int q = 0; q < KQ; ++q) {
            const float4 t = stage[(j * 32 + lane) * PQ + q];
            d[4 * q] = t.x, d[4 * q + 1] = t.y, d[4 * q + 2] = t.z, d[4 * q + 3] = t.w;
        }
    }
    }
    const float *const c0 = sc + (mine >= 0 ? mine : 0) * CB;
    const float omw = c0[(B - 1) * CS];

#pragma unroll 1
    for (int s = 0; s < nsteps; ++s) strip_step<B, DC, AA, DG, K, CH>(phi, v, c0, omw, nu);

    // own positions of the lane: [lo, hi) of its K; whole 16-byte pieces go out coalesced, the rest
    // (a lane that wraps or is not aligned, an own range that ends inside a piece) node by node
    int lo = 0, hi = 0;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < B; ++j) {
        const float *d = j ? v[j ? j - 1 : 0] : phi;
#pragma unroll
        for (int q = 0; q < KQ; ++q)
            stage[(j * 32 + lane) * PQ + q] = make_float4(d[4 * q], d[4 * q + 1], d[4 * q + 2], d[4 * q + 3]);
    }
    int again;  // 0, but not to the compiler: the lookup is made anew
    asm volatile("mov.u32 %0, 0;" : "=r"(again));
    const Place pl = place(again);
    const int x = pl.x, N = pl.N;
    const long long at = pl.at, ld = pl.ld;
    const bool fast = pl.fast;
    if (pl.mine >= 0) {
        const StripSeg &S = segs[(w < nmix ? first[w] : w - nmix) + pl.mine];
        const int p0 = (lane - S.lane0) * K;
        lo = max(S.vlo - p0, 0);
        hi = min(S.vhi - p0, K);
        if (hi < lo) hi = lo;
    }
    const int vhi = fast ? hi & ~3 : 0;  // whole pieces (vlo is a lane's first position)
    __syncwarp();
#pragma unroll
    for (int q = 0; q < KQ; ++q) {
        const int f = q * 32 + lane, L = f / KQ, r = f % KQ;
        const long long a = __shfl_sync(0xffffffffu, at, L), l = __shfl_sync(0xffffffffu, ld, L);
        const int b = __shfl_sync(0xffffffffu, lo, L), e = __shfl_sync(0xffffffffu, vhi, L);
        if (4 * r >= b && 4 * r + 4 <= e) {
#pragma unroll
            for (int j = 0; j < B; ++j)
                *reinterpret_cast<float4 *>(st_out + a + j * l + 4 * r) = stage[(j * 32 + L) * PQ + r];
        }
    }
    const float *const own = reinterpret_cast<const float *>(stage);
    for (unsigned m = __ballot_sync(0xffffffffu, max(lo, vhi) < hi); m; m &= m - 1) {
        const int L = __ffs(m) - 1;
        const long long a = __shfl_sync(0xffffffffu, at, L), l = __shfl_sync(0xffffffffu, ld, L);
        const int xl = __shfl_sync(0xffffffffu, x, L), n = __shfl_sync(0xffffffffu, N, L);
        const int b = __shfl_sync(0xffffffffu, max(lo, vhi), L), e = __shfl_sync(0xffffffffu, hi, L);
        if (lane >= b && lane < e) {
            const int y = (xl + lane) % n;
#pragma unroll
            for (int j = 0; j < B; ++j) st_out[a - xl + y + j * l] = own[(j * 32 + L) * PQ * 4 + lane];
        }
    }
}

}  // namespace lbk
