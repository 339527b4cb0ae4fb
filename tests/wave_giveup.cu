// A window of k_wave whose neighbour never trades with it (its plan names an unused place of the grid
// as that neighbour, so nothing is written where it waits): every wait runs out, and the launch ends
// with the mark set, the trades' numbers moved on and nothing but NaN in the state.  Then the same
// launch with the plan as it was: the next solve is not affected.  Compiled with few polls a wait.
// Prints "ok" and exits 0, or what is wrong and exits 1.
#include <cmath>
#include <cstdio>
#include <vector>

#include "lbhpde_internal.h"

#define CK(c)                                                                        \
    do {                                                                             \
        const cudaError_t e_ = (c);                                                  \
        if (e_ != cudaSuccess) {                                                     \
            std::printf("%s:%d: %s\n", #c, __LINE__, cudaGetErrorString(e_));        \
            return 1;                                                                \
        }                                                                            \
    } while (0)
#define CHECK(c)                                           \
    do {                                                   \
        if (!(c)) {                                        \
            std::printf("line %d: %s\n", __LINE__, #c);    \
            return 1;                                      \
        }                                                  \
    } while (0)

static int run(int csize) {
    constexpr int b = 5, K = 1, G = 1, T = 2, D = 5, nsteps = 40;
    lbk::Seg s{};
    s.N = 200;
    s.ld = 200;
    s.D = D;
    std::vector<lbk::WaveWin> wins;
    CHECK(lbh::pack_wave({s}, b, K, G, T, csize, wins));
    int nused = 0;
    for (const auto &w : wins) nused += w.N > 0;
    CHECK(nused == 9 && wins[nused].N == 0);  // windows 0 .. 8 of the ring, and unused places after them
    std::vector<float> zero((size_t)b * s.N, 0.f), phi(s.N, 0.25f), got(s.N);
    std::vector<float> coef(2 * (b - 1) * (D + 1) + 1, 0.f);  // omega f^eq = 0, 1 - omega
    coef.back() = 0.5f;
    float *st, *cf;
    lbk::WaveWin *wd;
    unsigned char *box;
    unsigned *ctrl;
    const size_t box_bytes = (size_t)lbk::wave_box_bytes(4, b, K, G) * wins.size();
    CK(cudaMalloc(&st, zero.size() * 4));
    CK(cudaMalloc(&cf, coef.size() * 4));
    CK(cudaMalloc(&wd, wins.size() * sizeof wins[0]));
    CK(cudaMalloc(&box, box_bytes));
    CK(cudaMalloc(&ctrl, 16));
    CK(cudaMemcpy(cf, coef.data(), coef.size() * 4, cudaMemcpyHostToDevice));
    CK(cudaMemset(box, 0, box_bytes));
    CK(cudaMemset(ctrl, 0, 16));
    unsigned c[3];
    for (int round = 0; round < 2; ++round) {
        std::vector<lbk::WaveWin> w = wins;
        if (round == 0) w[4].left = nused;  // 3 waits for 4, and 4 for the unused place
        CK(cudaMemcpy(wd, w.data(), w.size() * sizeof w[0], cudaMemcpyHostToDevice));
        CK(cudaMemcpy(st, zero.data(), zero.size() * 4, cudaMemcpyHostToDevice));
        CK(cudaMemcpy(st, phi.data(), phi.size() * 4, cudaMemcpyHostToDevice));
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        cfg.gridDim = dim3((unsigned)(wins.size() / lbk::kWaveWarps));
        cfg.blockDim = dim3(32 * lbk::kWaveWarps);
        cfg.dynamicSmemBytes = csize > 0 ? (size_t)lbk::wave_box_bytes(4, b, K, G) * lbk::kWaveWarps : 0;
        if (csize > 0) {
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = (unsigned)csize;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        } else {
            at[0].id = cudaLaunchAttributeCooperative;
            at[0].val.cooperative = 1;
        }
        cfg.attrs = at;
        cfg.numAttrs = 1;
        CK(cudaLaunchKernelEx(&cfg, lbk::k_wave<float, b, K, G, D, false>, (const float *)st, st, (const lbk::WaveWin *)wd, nused,
                              (const float *)cf, box, ctrl, nsteps, T, csize, (const float *)nullptr, 0));
        CK(cudaDeviceSynchronize());
        CK(cudaMemcpy(got.data(), st, s.N * 4, cudaMemcpyDeviceToHost));
        CK(cudaMemcpy(c, ctrl, sizeof c, cudaMemcpyDeviceToHost));
        CHECK(c[2] == (round == 0 ? 1u : 0u));
        CHECK(csize > 0 || (c[0] == (round + 1u) * ((nsteps - 1) / T + 1) && c[1] == 0));
        for (float x : got) CHECK(round == 0 ? std::isnan(x) : x == 0.25f);  // (populations of 0: phi stays)
        CK(cudaMemset(ctrl + 2, 0, 4));
    }
    return 0;
}

int main() {
    if (run(0) || run(4)) return 1;
    std::printf("ok\n");
    return 0;
}
