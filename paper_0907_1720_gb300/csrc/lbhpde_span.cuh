// Bounded FP32 instances of up to 1024 nodes (D1Q5, depth 2) or 768 (D1Q7, depth 1 or 2), one warp each
// for every step of a launch (the boundary rule of lbhpde_bounded.cuh).
//
// A lane holds K nodes in registers (node x at lane x / K, register x % K; K = 4 to 32, at least the
// smallest multiple of 4 that holds the instance; 8 to 24 on D1Q7), its neighbours' edges come by shuffle, and nothing is
// shared with other warps: no barrier, no exchange buffer, no copies.  The bound is the FP32 pipes
// (and below 300 nodes the ends, which cost a warp the same at any size); in k_ring_nee, whose
// 512-thread CTAs hold 13 instances of 601 nodes, every step waits at a barrier, and in k_bounded
// (D1Q7), whose CTA holds one, two warps of five besides at the ends' work.  GB300, 601 nodes, us a
// step: D1Q5 5928 instances 4.37 (8.2e11 node-updates/s, 67% of the FP32 pipes) against 5.92, 608
// instances 0.66 against 1.99; D1Q7 5928 instances 8.2 (4.3e11, 66%) against 16.4, 608 1.16 against 2.43.
//
// After each step the max|e| outer nodes of either end take f^eq_j(phi_b) + [s_j(x_f) - f^eq_j(phi(x_f))].
// x_f's state comes by shuffle from its lane; on D1Q5 lane (side, l, j) of 2 x 2 x 4 = 16 evaluates one
// population of one outer node, on D1Q7 lane (side, j) the bracket of one population, and the
// owners fetch theirs by shuffle.  The left end sits at fixed registers of lane 0; the right end's
// depend on N % K, the same for the whole warp: one compile-time case of a jump.  phi_b and
// f^eq_j(phi_b) of 8 steps at a time (5 on D1Q7) are evaluated by all lanes, a value each, from
// boundary values loaded that many steps earlier.  What positions past the last node hold reaches
// the outer nodes only, which the rebuild overwrites.
//
// Each node's update is k_bounded's, operation by operation.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbhpde_strip.cuh"

namespace lbk {

struct SpanInst {
    long long off, ld;  // placement of the instance's state (as Seg)
    int N, D;
    int gcoef;          // coefficient block in global memory (as Seg::coef)
    int depth;          // 2; D1Q7: 1 or 2
    int mi;             // batch member index: its boundary values start at phib + mi * stride
};

__host__ __device__ constexpr int span_steps(int B) { return 32 / (2 * wmax(B)); }  // steps whose ends are staged at once
__host__ __device__ constexpr int span_warps(int B, int K) {  // warps an SM: the registers of a lane's nodes
    if (B == 7) return K <= 8 ? 16 : (K <= 16 ? 12 : 8);
    return K <= 8 ? 24 : (K <= 12 ? 16 : (K <= 16 ? 14 : (K <= 20 ? 12 : (K <= 24 ? 10 : 8))));
}

template <int B, int K>
__global__ void __launch_bounds__(32, span_warps(B, K))
    k_span(const float *st_in, float *st_out, const SpanInst *__restrict__ insts, const float *__restrict__ coefs,
           const double *__restrict__ phib, long long stride, long long step0, int nsteps) {
    constexpr int DC = B == 5 ? 5 : 7, W = wmax(B), CS = crow(DC), CH = 4, kSteps = span_steps(B);
    static_assert(K % 4 == 0 && K <= 32, "16-byte loads; the cases of the jump");
    static_assert(W + 2 <= K, "x_f of the left end is a register of lane 0");
    __shared__ __align__(16) float P[(B - 1) * CS], Q[(B - 1) * CS];  // omega f^eq_j, f^eq_j
    __shared__ float E[kSteps * 2 * W * B];                          // phi_b, f^eq_1 .. f^eq_(B-1) of it
    const int lane = threadIdx.x;
    const SpanInst I = insts[blockIdx.x];
    const int crows = (B - 1) * (I.D + 1);
    for (int q = lane; q < (B - 1) * CS; q += 32) {
        const int j = q / CS, p = q % CS;
        P[q] = p <= I.D ? coefs[I.gcoef + j * (I.D + 1) + p] : 0.f;
        Q[q] = p <= I.D ? coefs[I.gcoef + crows + j * (I.D + 1) + p] : 0.f;
    }
    const float omw = coefs[I.gcoef + 2 * crows];
    __syncwarp();
    // this lane's outer value (D1Q7: of all outer nodes of the side; rows 6 and 7 repeat row 5)
    const int row = B == 5 ? lane & 3 : min(lane & 7, B - 2), ol = B == 5 ? lane >> 2 & 1 : 0, side = lane >> 3 & 1;
    float qr[DC + 1];
#pragma unroll
    for (int p = 0; p <= DC; ++p) qr[p] = Q[row * CS + p];
    const int N = I.N, x0 = lane * K;
    const int depth = B == 5 ? 2 : I.depth, xf = N - W - depth;
    const int lf = xf / K, rem = N % K, remf = xf % K;
    int lown[W];  // the lanes of the right outer nodes N - W + l
#pragma unroll
    for (int l = 0; l < W; ++l) lown[l] = (N - W + l) / K;

    float phi[K], v[B - 1][K];
    if (x0 + K <= N) {
#pragma unroll
        for (int j = 0; j < B; ++j) {
            float *d = j ? v[j ? j - 1 : 0] : phi;
#pragma unroll
            for (int q = 0; q < K / 4; ++q) {
                const float4 t = *reinterpret_cast<const float4 *>(st_in + I.off + j * I.ld + x0 + 4 * q);
                d[4 * q] = t.x, d[4 * q + 1] = t.y, d[4 * q + 2] = t.z, d[4 * q + 3] = t.w;
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool ok = x0 + k < N;
            phi[k] = ok ? st_in[I.off + x0 + k] : 0.f;
#pragma unroll
            for (int j = 1; j < B; ++j) v[j - 1][k] = ok ? st_in[I.off + j * I.ld + x0 + k] : 0.f;
        }
    }
    // boundary value of step lane / (2 W) of the next kSteps, outer node lane % (2 W)
    const double *const pb = phib + (long long)I.mi * stride + step0 * (2 * W);
    const long long nval = (long long)nsteps * (2 * W);
    const bool stager = kSteps * 2 * W == 32 || lane < kSteps * 2 * W;
    double ahead = stager && lane < nval ? pb[lane] : 0.0;

#pragma unroll 1
    for (int s = 0; s < nsteps; ++s) {
        const int t = s % kSteps;
        if (t == 0) {
            const float x = (float)ahead;
            const long long nx = (long long)(s + kSteps) * (2 * W) + lane;
            ahead = stager && nx < nval ? pb[nx] : 0.0;
            __syncwarp();
            if (stager) {
                E[lane * B] = x;
#pragma unroll
                for (int j = 1; j < B; ++j) {
                    const float *c = Q + (j - 1) * CS;
                    float acc = c[DC];
#pragma unroll
                    for (int p = DC - 1; p >= 0; --p) acc = __fmaf_rn(acc, x, c[p]);
                    E[lane * B + j] = acc;
                }
            }
            __syncwarp();
        }
        strip_step<B, DC, 0, 0, K, CH>(phi, v, P, omw, 1.f);
        // x_f's state in its lane's u: left x_f is register W - 1 + depth of lane 0, right x_f
        // register remf of lane lf
        float u[B];
        u[0] = depth == 2 ? phi[W + 1] : phi[W];
#pragma unroll
        for (int j = 1; j < B; ++j) u[j] = depth == 2 ? v[j - 1][W + 1] : v[j - 1][W];
        auto take = [&](auto rc) {
            // (at D1Q5's fixed depth from N % K as below: 2.5% faster there than a second variable)
            constexpr int q = B == 5 ? (decltype(rc)::value - W - 2 + 2 * K) % K : decltype(rc)::value;
            const bool right = lane != 0;
            u[0] = right ? phi[q] : u[0];
#pragma unroll
            for (int j = 1; j < B; ++j) u[j] = right ? v[j - 1][q] : u[j];
        };
        float w[W][B];  // the owners' new values
        auto put = [&](auto rc) {
            constexpr int r = decltype(rc)::value;
#pragma unroll
            for (int l = 0; l < W; ++l) {
                const int q = (r - W + l + K) % K;  // node N - W + l
                const bool own = lane == lown[l];
                phi[q] = own ? w[l][0] : phi[q];
#pragma unroll
                for (int j = 1; j < B; ++j) v[j - 1][q] = own ? w[l][j] : v[j - 1][q];
            }
        };
#define LBK_SPAN_CASE(R) \
    case R:              \
        if constexpr (R < K) f(std::integral_constant<int, R>{}); \
        break;
        auto by = [&](int at, auto f) {
            switch (at) {
                LBK_SPAN_CASE(0) LBK_SPAN_CASE(1) LBK_SPAN_CASE(2) LBK_SPAN_CASE(3) LBK_SPAN_CASE(4) LBK_SPAN_CASE(5)
                LBK_SPAN_CASE(6) LBK_SPAN_CASE(7) LBK_SPAN_CASE(8) LBK_SPAN_CASE(9) LBK_SPAN_CASE(10) LBK_SPAN_CASE(11)
                LBK_SPAN_CASE(12) LBK_SPAN_CASE(13) LBK_SPAN_CASE(14) LBK_SPAN_CASE(15) LBK_SPAN_CASE(16) LBK_SPAN_CASE(17)
                LBK_SPAN_CASE(18) LBK_SPAN_CASE(19) LBK_SPAN_CASE(20) LBK_SPAN_CASE(21) LBK_SPAN_CASE(22) LBK_SPAN_CASE(23)
                LBK_SPAN_CASE(24) LBK_SPAN_CASE(25) LBK_SPAN_CASE(26) LBK_SPAN_CASE(27) LBK_SPAN_CASE(28) LBK_SPAN_CASE(29)
                LBK_SPAN_CASE(30) LBK_SPAN_CASE(31)
            }
        };
#undef LBK_SPAN_CASE
        by(B == 5 ? rem : remf, take);
        const int src = side ? lf : 0;
        const float ph = __shfl_sync(0xffffffffu, u[0], src);
        float vf = 0.f;
#pragma unroll
        for (int j = 1; j < B; ++j) {
            const float y = __shfl_sync(0xffffffffu, u[j], src);
            vf = row == j - 1 ? y : vf;
        }
        float f = qr[DC];
#pragma unroll
        for (int p = DC - 1; p >= 0; --p) f = __fmaf_rn(f, ph, qr[p]);
        const float br = vf - f;
        const float val = B == 5 ? E[(t * 2 * W + side * W + ol) * B + 1 + row] + br : br;
        float diff[B];
        const int mine = lane == 0 ? 0 : 1;  // the end whose outer nodes this lane may own
#pragma unroll
        for (int l = 0; l < W; ++l) {
            w[l][0] = E[(t * 2 * W + mine * W + l) * B];
#pragma unroll
            for (int j = 1; j < B; ++j) {
                if (B == 5)
                    w[l][j] = __shfl_sync(0xffffffffu, val, mine * 8 + l * 4 + j - 1);
                else
                    w[l][j] = E[(t * 2 * W + mine * W + l) * B + j] + (l ? diff[j] : (diff[j] = __shfl_sync(0xffffffffu, val, mine * 8 + j - 1)));
            }
        }
#pragma unroll
        for (int l = 0; l < W; ++l) {
            phi[l] = lane == 0 ? w[l][0] : phi[l];
#pragma unroll
            for (int j = 1; j < B; ++j) v[j - 1][l] = lane == 0 ? w[l][j] : v[j - 1][l];
        }
        by(rem, put);
    }
    if (x0 + K <= N) {
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const float *d = j ? v[j ? j - 1 : 0] : phi;
#pragma unroll
            for (int q = 0; q < K / 4; ++q)
                *reinterpret_cast<float4 *>(st_out + I.off + j * I.ld + x0 + 4 * q) =
                    make_float4(d[4 * q], d[4 * q + 1], d[4 * q + 2], d[4 * q + 3]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (x0 + k < N) {
                st_out[I.off + x0 + k] = phi[k];
#pragma unroll
                for (int j = 1; j < B; ++j) st_out[I.off + j * I.ld + x0 + k] = v[j - 1][k];
            }
    }
}

}  // namespace lbk
