// Host-side pieces shared by the batch API (lbhpde_api.cu) and the request server
// (lbhpde_server.cu): packing of instances onto CTAs for the on-chip kernel and the typed
// kernel launchers.  Implemented in lbhpde_api.cu, so each kernel is compiled once.
#pragma once
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <vector>

#include "lbhpde.h"
#include "lbhpde_bounded.cuh"
#include "lbhpde_kernels.cuh"
#include "lbhpde_ring.cuh"
#include "lbhpde_ring_nee.cuh"
#include "lbhpde_span.cuh"
#include "lbhpde_strip.cuh"
#include "lbhpde_wave.cuh"

namespace lbh {

// A named NVTX range for the scope (tracing: host phases of the API and of the server show in
// Nsight timelines and can filter ncu captures; without a tool attached it costs a branch).
struct TraceRange {
    explicit TraceRange(const char *name) { nvtxRangePushA(name); }
    ~TraceRange() { nvtxRangePop(); }
    TraceRange(const TraceRange &) = delete;
    TraceRange &operator=(const TraceRange &) = delete;
};

constexpr int kChunk = 1024;          // nodes per block of the node-parallel kernels
constexpr int kGenericThreads = 256;  // init / readout / diagnostics threads per block

// The dynamic shared memory a CTA can have (none of the kernels that take any has static one too), and
// a kernel's permission to use it all, whatever a launch takes.  The permission belongs to the kernel
// in the whole process: with each launch asking for its own size, a smaller plan of another handle's
// thread could take it down between a launch's asking and the launch, which then failed.
constexpr size_t kMaxSmem = 227 * 1024;
template <typename F>
bool allow_smem(F fn) {
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem) == cudaSuccess) return true;
    (void)cudaGetLastError();
    return false;
}

// One instance to place on the on-chip kernel.
struct Member {
    lbk::Seg seg;      // placement of the current state (and its coefficient block)
    long long off2;    // where the kernel writes the result (== seg.off for in-place)
    int steps;         // steps this instance takes in the launch
};

// A packed on-chip launch: CTA c holds insts[first[c] .. first[c + 1]).
struct Packed {
    std::vector<lbk::OnchipInst> insts;
    std::vector<int> first;
    int nthreads = 32;  // threads per CTA
    int max_inst = 1;   // instances per CTA (resident mode: rounded up to a multiple of 4)
    size_t smem = 0;    // dynamic shared memory per CTA, bytes
    int stride = 0;     // k_ring: the class's CTA size, the row stride of its exchange buffers
    int ncta() const { return first.empty() ? 0 : (int)first.size() - 1; }
};

// Threads per CTA of the on-chip kernels for (element size, lattice, nodes per thread), 0 when
// no variant exists: resident instances (capacity = threads * K nodes) and temporally blocked
// windows (FP32 D1Q5 with K = 8 uses smaller window CTAs).
constexpr int kHaloThreadsF32Q5 = 128;
// Nodes a thread of the 16-node resident kernel (k_ring, FP32 D1Q5) holds: an instance of up to
// 16 * 512 = 8192 nodes stays in one CTA.  Planned with K == kRingK, resident instances only.
constexpr int kRingK = 16;
// Whether members of (element size, lattice, on-chip degree code) can take k_ring.
bool ring_split_ok(size_t esz, int b, int dc);
int onchip_maxt(size_t esz, int b, int K);
int onchip_maxt_halo(size_t esz, int b, int K);
int default_K(size_t esz, int b);
// Steps per halo window (a power of two up to 64) such that the halo (steps * max|e| on each
// side) leaves at least valid_eighths / 8 of a window of `capacity` nodes valid.  Batches take
// 7/8 (the autotuner's picks on GB300: 32 for FP32 windows, 16 for FP64 D1Q7); the server takes
// 6/8, since each window chunk of a step block is another launch.
int default_tblk(int capacity, int W, int valid_eighths = 7);
// Compile-time degree variant the on-chip kernel uses for a set of members of maximum degree D.
int onchip_dc(int b, int maxD);

// Resident instances (N <= capacity): first fit, largest first, <= 32 per CTA, in CTAs of `threads`
// threads (0: the configuration's resident CTA size).  Runs of threads are warp-aligned for
// k_onchip and thread-granular for k_ring (K == kRingK).
int pack_ring(int b, size_t esz, int K, int dc, const std::vector<Member> &m, Packed &out, int threads = 0);
// Resident size class of an instance of N nodes (0, 1, 2) and the CTA size of a class.
constexpr int kRingClasses = 3;
int ring_class(size_t esz, int b, int K, long long N);
int ring_class_threads(size_t esz, int b, int K, int cls);
// Threads an instance's run is rounded up to (32 for k_onchip, 1 for k_ring).
int ring_granule(int K);
// Instances a CTA holds at most (the tail buffer rows of the on-chip kernels).
constexpr int kRingMaxInstances = 32;
// Wave-aware split of the 16-node resident members (K == kRingK) for a GPU of `sms` SMs: `full`
// packs (first fit, largest first) into whole waves of full-SM CTAs, one CTA per SM at a time;
// `tail` holds the members that do not fit there (or were evicted from a CTA to make room for a
// larger one).  The tail runs afterwards in CTAs of its own size class spread over the SMs, so the
// last, partial wave costs the time of its members' own work instead of a whole wave of full
// CTAs.  False (both empty) when the members do not fill one wave or all fit.
bool split_ring_waves(int b, int K, int sms, const std::vector<Member> &m, std::vector<Member> &full,
                      std::vector<Member> &tail);
// Resident members by the CTA size class they take: their own class, or the largest one where
// they fill a gap left by larger instances.
void split_ring_classes(size_t esz, int b, int K, const std::vector<Member> &m, std::vector<Member> (&out)[kRingClasses]);
// Temporally blocked windows with halo H: one window per CTA.
// wide: windows as large as a resident CTA (fewer, longer windows: the server, whose step
// blocks fix the steps per window) instead of the smaller window CTAs.
// threads > 0: windows of CTAs of at most that many threads, each member cut into equal ones.
int pack_halo(int b, size_t esz, int K, int dc, int H, const std::vector<Member> &m, Packed &out,
              bool wide = false, int threads = 0);
// Whether FP64 periodic members advance faster in windows of a chosen size alone (threads of a CTA,
// steps a launch) than with the short ones resident and the long ones in windows of a CTA's size, with K0
// nodes a thread and T0 steps a launch (0: K and the default).
bool windows_f64(int b, int dc, int K, const std::vector<lbk::Seg> &m, int sms, int *threads, int *steps, int K0 = 0, int T0 = 0);

// K == kRingK launches k_ring (resident plans only).
int launch_onchip(int b, size_t esz, int K, int dc, bool halo, const Packed &p, const lbk::OnchipInst *insts_d,
                  const int *first_d, const void *in, void *out, const void *coefT, int nsteps, cudaStream_t st);
int launch_ring_f32(int dc, const Packed &p, const lbk::OnchipInst *insts_d, const int *first_d, const void *in,
                    void *out, const void *coefT, int nsteps, cudaStream_t st);
// the same for one precision (lbhpde_onchip_f32.cu, lbhpde_onchip_f64.cu)
int launch_onchip_f32(int b, int K, int dc, bool halo, const Packed &p, const lbk::OnchipInst *insts_d,
                      const int *first_d, const void *in, void *out, const void *coefT, int nsteps, cudaStream_t st);
int launch_onchip_f64(int b, int K, int dc, bool halo, const Packed &p, const lbk::OnchipInst *insts_d,
                      const int *first_d, const void *in, void *out, const void *coefT, int nsteps, cudaStream_t st);
// coefT: the coefficient table in the state's type (f^eq rows after the P_j rows, as lbk::Seg::coef).
int launch_init(int b, size_t esz, void *st, const lbk::Seg *segs, const int2 *blocks, int nb, const void *coefT,
                const double *phi0, const long long *blk_off, cudaStream_t stream);

// Bounded grids (lbhpde_bounded.cu): instances of up to kBoundedK * kBoundedMaxT nodes stay
// resident in one CTA each; longer ones take the streaming step plus the outer-node rebuild.
constexpr int kBoundedK = 4;
constexpr int kBoundedMaxT = 512;
constexpr int kBoundedMaxTAny = 256;       // CTA size of the FP64 variants with 3, 5 or 6 nodes a thread
constexpr int kBoundedMaxSteps = 1024;     // steps per resident launch, at most
constexpr int kBoundedStageBytes = 16384;  // shared memory for the launch's boundary data
// Dynamic shared memory of k_bounded for a launch of nsteps steps.
size_t bounded_smem(int b, size_t esz, int nthreads, int D, int nsteps);
// Steps per resident launch: as many as kBoundedStageBytes of staged boundary data hold.
int bounded_launch_steps(int b, size_t esz);
// Smallest position shift that puts each end's outer nodes and extrapolation node in one warp of
// the resident kernel (and keeps the instance within one CTA); -1 if there is none.
int bounded_shift(int b, int N, int depth, int K = kBoundedK);
// The degree k_bounded has compiled; 3, 5 and 6 nodes a thread exist in FP64 for it alone.
constexpr int bounded_degree(int b) { return b == 5 ? 5 : 7; }
// Nodes a thread (4, or 3, 5, 6) with which FP64 bounded members of that degree take the least time.
int bounded_nodes(int b, const std::vector<lbk::Seg> &m, int sms);
// dc: the compiled degree (5 on D1Q5, 7 on D1Q7), 0 for a run-time degree, -1 for the variant
// that also evaluates real-exponent instances (A > 0).
int launch_bounded(int b, size_t esz, int dc, int ninst, int nthreads, size_t smem, const lbk::BoundedInst *insts_d,
                   const void *in, void *out, const void *coefT, const double *phib, long long stride,
                   long long step0, int nsteps, cudaStream_t st, int K = kBoundedK);
int launch_nee_fix(int b, size_t esz, void *st, const lbk::Seg *segs, const int *members, int nmem,
                   const void *coefT, const double *phib, long long stride, long long step, cudaStream_t stream);

// Bounded members on the 16-node resident kernel (k_ring_nee, FP32 D1Q5 polynomial models): the
// interior nodes W..N-W-1 in thread-granular runs of ceil((N - 2W) / 16) threads, first fit,
// largest first, at most 32 instances per CTA of `threads` threads.
struct PackedNee {
    std::vector<lbk::RingNeeInst> insts;
    std::vector<int> first;
    int nthreads = 32, stride = 0;
    bool d2 = false;  // every member of depth 2 with at least 2 interior nodes in its last thread
    size_t smem = 0;
    int ncta() const { return first.empty() ? 0 : (int)first.size() - 1; }
};
struct NeeMember {
    lbk::Seg seg;
    int mi;     // batch member index (its boundary rows)
    int steps;  // steps in the launch
};
// Whether a bounded member can take k_ring_nee: FP32 D1Q5 polynomial, its interior within one
// 512-thread CTA, depth within the first and last 16 interior nodes' reach.
bool ring_nee_ok(size_t esz, int b, const lbk::Seg &s);
int pack_ring_nee(int b, int dc, const std::vector<NeeMember> &m, PackedNee &out, int threads);
// started: an event to record once every CTA has begun (best effort; nullptr: none).
int launch_ring_nee_f32(int dc, const PackedNee &p, const lbk::RingNeeInst *insts_d, const int *first_d,
                        const void *in, void *out, const void *coefT, const double *phib, long long stride,
                        long long step0, int nsteps, cudaStream_t st, cudaEvent_t started = nullptr);

// Small and medium grids in windows of one warp each (k_wave, lbhpde_wave.cu).
struct PackedWave {
    std::vector<lbk::WaveWin> wins;  // whole CTAs (and clusters): unused places have N = 0
    int esz = 0, b = 0, dc = 0;
    int K = 0, G = 0;  // positions a lane, lane groups a window's populations are split over
    bool nee = false;
    int tblk = 0;      // steps between two trades of the windows' borders
    int csize = 0;     // CTAs of a cluster that holds whole instances; 0: boxes in global memory
    int nmem = 0, nused = 0;  // members; windows that hold nodes
    double cost = 0, other = 0;  // modelled clocks of a step, and of a step of the best other kernel
    int wsmem = 0;     // shared-memory elements a window, beside the boxes
    size_t smem = 0, box_bytes = 0;
    int ncta() const { return (int)wins.size() / lbk::kWaveWarps; }
};
// Windows of the members (periodic, or bounded with Seg::pad = depth); false where some member does
// not divide that way.
bool pack_wave(const std::vector<lbk::Seg> &m, int b, int K, int G, int T, int csize, std::vector<lbk::WaveWin> &out);
// The plan of a whole batch, where k_wave is the better kernel for it on a GPU of `sms` SMs.
bool plan_wave(size_t esz, int b, int dc, bool nee, const std::vector<lbk::Seg> &m, int sms, PackedWave &out);
// What a step of its best form costs on that GPU by the model, in SM clocks (as cta_cost, strip_cost).
double wave_cost(size_t esz, int b, int dc, bool nee, const std::vector<lbk::Seg> &m, int sms);
// nsteps steps, in place; ends: the table of launch_wave_ends for the same steps (bounded members).
int launch_wave(const PackedWave &p, const lbk::WaveWin *wins, unsigned char *box, unsigned *ctrl, void *st, const void *coefT,
                int nsteps, const void *ends, cudaStream_t stream);
int launch_wave_ends(const PackedWave &p, void *ends, const lbk::Seg *segs, const int *members, const void *coefT,
                     const double *phib, long long stride, long long step0, int nsteps, cudaStream_t st);

// Strips of one warp each (k_strip, lbhpde_strip.cu): warp w < nmix() holds segs[first[w] .. first[w + 1]),
// warp nmix() + i holds segs[i] alone (i < nfull).
struct PackedStrip {
    std::vector<lbk::StripSeg> segs;
    std::vector<int> first;
    int b = 0, nfull = 0;
    int AA = 0, DG = 0;  // row shape of a real-exponent model (AA = 0: polynomials, of compiled degree DG)
    int nmix() const { return first.empty() ? 0 : (int)first.size() - 1; }
    int nwarps() const { return nfull + nmix(); }
};
// Whether members of (element size, lattice, on-chip degree code) can take k_strip; AA, DG: their row
// shape (AA = 0: polynomials, of compiled degree DG).
bool strip_ok(size_t esz, int b, int dc, const std::vector<lbk::Seg> &m, int *AA, int *DG);
void pack_strip(int b, int AA, int DG, const std::vector<lbk::Seg> &m, PackedStrip &out);
// What a step costs on a GPU of `sms` SMs, in SM clocks: the CTA-wide kernels on a group's members,
// k_strip with a plan.
double cta_cost(size_t esz, int b, int dc, bool nee, bool real, const std::vector<lbk::Seg> &m, int sms);
double strip_cost(const PackedStrip &p, int sms);
// At most lbk::strip_steps(b, AA) steps, from buffer `in` to another one.
int launch_strip(const PackedStrip &p, const lbk::StripSeg *segs, const int *first, const void *in, void *out,
                 const void *coefT, int nsteps, cudaStream_t st);

// Bounded FP32 members of one warp each (k_span, lbhpde_span.cu): whether a member can, and the nodes
// a lane holds then (a multiple of 4).
bool span_ok(size_t esz, int b, const lbk::Seg &s);
int span_nodes(int N);
// The launches of members sorted by their own nodes a lane, falling: (nodes a lane, first member) of
// at most two; a member may run with more than its own.
std::vector<std::pair<int, int>> span_launches(const std::vector<int> &nodes, int sms);
int launch_span(int b, int K, const lbk::SpanInst *insts, int n, const void *in, void *out, const void *coefT, const double *phib,
                long long stride, long long step0, int nsteps, cudaStream_t st);

}  // namespace lbh
