// e2ga_internal.cuh -- device-side layout and helpers shared by the library's
// translation units.  Not part of the public ABI (see include/e2ga.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "e2ga.h"

namespace e2 {

// +inf as a 64-bit key.  Every time in the planner is a non-negative float64
// (or +inf), and non-negative IEEE-754 doubles order exactly like their bit
// patterns read as unsigned integers, so the DP compares 64-bit integer keys.
constexpr uint64_t kInfKey = 0x7FF0000000000000ull;

// Philox stream purposes (counter word 3).
enum Purpose : uint32_t {
    kInitPerm = 0, kInitGroup = 1, kInitRoles = 2, kSelect = 3, kCross = 4, kMutate = 5,
    kMutPerm = 6, kMutGroup = 7, kMutRoles = 8, kCong = 9
};

// Profile arrays in the workspace: kProf* index the 7 arrays of length V.
enum ProfArray { kBlkFlops = 0, kBlkBytes, kBlkMem, kHeadFlops, kHeadBytes, kHeadMem, kAct, kNumProf };

struct DevPop {
    uint16_t *perm;    // [P][M]
    uint16_t *sizes;   // [P][K]
    uint8_t *nclus;    // [P]
    uint64_t *roles;   // [P]
};

// Largest replica (devices) a DP can receive: replicas with more devices than
// blocks are infeasible, and the DP's warps hold up to 8 devices per lane.
constexpr int kMaxReplicaDevices = 256;

// The DP's work list: items in kListBins bins of replica sizes (class 0 before
// class 1, larger first), placed from per-block counts of the slots' items by
// at most kListBlocks blocks.
constexpr int kListBins = 64;
constexpr int kListBlocks = 256;
// Its control words: where each class's items end (class 1's follow class
// 0's) and each class's DP cursor (starting where its items start).
enum CtrlWord { kCtrlEnd = 0, kCtrlNext = 2, kCtrlWords = 4 };

// A slot's info word: the largest decode batch to run (0: none), the largest
// its memory allows, whether the prefill run can matter, which tests were
// made, and the bin of its size in the work list.
constexpr uint32_t kSlotDecMask = 0x7F;
constexpr int kSlotMemShift = 7;
constexpr uint32_t kSlotPrefill = 1u << 14, kSlotDecTested = 1u << 15, kSlotPreTested = 1u << 16;
constexpr int kSlotBinShift = 24;

// The bound of the ABI on the blocks of a fleet, for models of identical blocks:
// inputs are refused for which some replica of m devices and its W = N - m + 1
// block counts come to more bytes, as counted here, than a CTA may have of shared
// memory (up to 16 devices any N, 32 devices 752 blocks, 64 462, 128 337, 256
// 328).  No kernel lays this out; the bound is kept so that the sizes accepted stay
// the same.
__host__ __forceinline__ size_t dp_table_bytes(int m, int N, bool spill)
{
    const size_t W = (size_t)(N - m + 1), mm = (size_t)m;
    const size_t keys = 2 * mm * W + (spill ? 2 : mm) * W + (spill ? 14 : 10) * W + 2 * mm;
    return (mm * 12 + keys * 4 + mm * 2 + 15) & ~(size_t)15;
}
__host__ __forceinline__ size_t dp_size_limit_bytes(int M, int N)
{
    const int mmax = M < N ? M : N;
    size_t best[2] = {0, 0};
    for (int m = 1; m <= mmax; ++m)
        for (int s = 0; s < 2; ++s) {
            const size_t b = dp_table_bytes(m, N, s != 0);
            if (b > best[s]) best[s] = b;
        }
    return best[0] > 40u * 1024u ? best[1] : best[0];
}
// Slots of the duplicate test's fingerprint table: the power of two >= 2P.
__host__ __device__ __forceinline__ unsigned dup_table_size(int P)
{
    unsigned t = 2;
    while (t < 2u * (unsigned)P) t <<= 1;
    return t;
}
// Stats slots (unsigned long long, atomically accumulated).
enum StatSlot { kStGenomes = 0, kStReplicas, kStDpRuns, kStCells, kStProbes, kStPaper, kStPrecheck,
                kStServed, kStTpsPruned, kStDpRunsSmall, kStRoleCapped, kStDeviceErrors, kNumStats };

// Everything a kernel needs, passed by value.
struct Dims {
    int M, N, V, b_max, P, Q, K;
    int LS;              // leaf row stride (>= N, even)
    int tournament;
    uint64_t NP, ND;
    double min_tps, t_a;
    double lam_max;      // largest latency Lambda with 1.0 / Lambda >= min_tps (see e2_create)
    int role_search;     // 1: both roles per replica, best assignment per genome (Alg. 2);
                         // 2: both roles per replica, the adapted-SplitWise rule picks the roles
    float lam_max_up;    // lam_max rounded up to float (the float latency bound is compared with it)
    int dp_mmax;         // min(M, N): the largest replica's devices
    int dp_split;        // DP class 0: the replicas of at most this many devices (0: all of them)
    float lam_fx;        // 2^22 / lam_max for the fixed-point latency test (0: not used)
    int grows;           // 1: block memory, head memory, block flops and bytes and activation bytes never
                         // shrink from one decode batch to the next (the pre-pass tests are then monotone)
    int objective;       // 0: waiting time w (Eq. 3-5); 1: per-request finishing time FT
    int offload;         // 1: some device has host memory for offloaded blocks
    int layered;         // 1: blocks of several types (per-layer prefix sums): the per-layer DP path
};

// A link of a variant: its time, its order key against the stage times
// (ranks.cu) and the time rounded down.
struct __align__(16) LinkRec {
    double t;
    uint32_t key;
    float lb;
};

struct Tables {
    // The fleet and the profile as given.  No kernel of an evaluation reads these
    // seven; they keep the parameters after the tables where they are: without them
    // class 1 of the DP took 139.7 us instead of 137.8 at 512 devices and a whole
    // evaluation 0.2 to 0.6% longer, in every order of the parameters tried, and with
    // seven words of padding in their place it did not.
    const double *rate, *bw;
    const uint64_t *mem;
    const double *rate_cpu, *bw_cpu;   // [M] host side of offloaded blocks (offload only)
    const uint64_t *mem_cpu;           // [M] host memory for blocks, bytes (offload only)
    const uint64_t *prof;      // [kNumProf][V]
    const double *leaf;        // [V][M][2][LS]: leaf[((v*M+d)*2+mf)*LS + n-1] = l_d(n blocks, master mf)
    const LinkRec *tau;        // [V][M][M]
    const int32_t *capg;       // [V][M][2]: most blocks in device memory, without / with the head (-1: the head
                               // does not fit)
    const uint32_t *leaf_rank; // [V][M][2][LS]: order key of leaf within its variant's value set
    const double *lcost;       // [V][M][2][N][N] (per-layer profiles only): lcost[((v*M+d)*2+mf)*N*N + j*N + n-1]
                               // = time of blocks j..j+n-1 on device d (+inf beyond the model or memory)
    const uint4 *drec;         // [V][M] the DP's view of a device: {cap | cap with head << 16, and as floats
                               // 1 / block time, the head in blocks, host block rate / device block rate}
    const float *fxs;          // [V] 2^22 / the largest 1 / block time: its fixed-point scale
    const uint4 *prec;         // [M] the pre-pass's view of a device: 1 / rate and 1 / bandwidth rounded down
                               // (float bits), its capacities (| with the head << 16) at batch 1 and b_max
    const float2 *prech;       // [M] 1 / rate and 1 / bandwidth of its host, rounded down (0: no host memory)
    const uint32_t *capv;      // [M][V] its capacities (| with the head << 16)
    const float *ibw;          // [M][M] 1 / effective link bandwidth, rounded down
    const float4 *fpr;         // [V] block flops, block bytes, activation bytes, rounded down
};

// Per (genome, replica slot) results of the evaluation pre-pass.
struct SlotInfo {
    int32_t *off;              // [P*K] offset of the replica in the ordering chromosome
    uint32_t *info;            // [P*K] its verdicts (kSlot*)
};

// Work items of the DP: (slot << 8) | role << 7 | variant bit.
struct WorkList {
    uint64_t *items;           // [2*P*K] (per-layer profiles: [V*P*K])
    unsigned *ctrl;            // [kCtrlWords]
};

// Results per (slot, role) where both roles are evaluated (role_search); with
// roles in the genome the DP writes the replica's outputs directly.
struct SplitOut {
    double *T, *L;             // [P*K][2]
    int16_t *mu;               // [P*K][2]
    int16_t *code;             // [P*K][2] the accepted variant's bit (prefill: 0), -1: none
    int16_t *layers;           // [P][2][M]
};

// Results per (slot, variant) of per-layer profiles, whose batches run as
// separate items (prefill: variant 0, decode batch b: variant b).
struct VariantOut {
    double *T, *L;             // [P*K][V]
    int16_t *mu;               // [P*K][V]
    int16_t *layers;           // [P][V][M]
    int32_t *best;             // [P*K] largest batch accepted so far - 1 (-1: none)
};

struct EvalOut {
    double *fit;               // [P][4]
    int16_t *layers;           // [P][M]
    int16_t *master, *bsel;    // [P][K]
    double *T, *L;             // [P][K]
    uint64_t *hash;            // [P]
    unsigned long long *stats; // [kNumStats]
    int16_t *gpu_layers;       // [P][M] blocks in device memory (offload only)
};

// ---------------------------------------------------------------------------
// Philox-4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 32x32->64 multiplies of counter words 0 and 2, the high halves xored with
// the other words and the key, the key advanced by the Weyl increments
// between rounds.
// ---------------------------------------------------------------------------
// First call of a kernel launched early: waits for the end of the kernel before
// it in the stream (its writes are visible then) and lets the kernel after it
// be placed.  Both do nothing in an ordinary launch.
__device__ __forceinline__ void after_previous()
{
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
}

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

// A stream (seed, generation, slot, purpose) of 32-bit words; word t is
// component t%4 of the block with counter (t/4, slot, generation, purpose).
struct Stream {
    uint32_t k0, k1, gen, slot, purpose;
    uint32_t blk;
    uint4 cache;
    __device__ Stream(uint64_t seed, uint32_t g, uint32_t s, uint32_t p)
        : k0((uint32_t)seed), k1((uint32_t)(seed >> 32)), gen(g), slot(s), purpose(p), blk(0xFFFFFFFFu) {}
    __device__ __forceinline__ uint32_t word(uint32_t t)
    {
        const uint32_t b = t >> 2;
        if (b != blk) {
            cache = philox4x32_10(make_uint4(b, slot, gen, purpose), k0, k1);
            blk = b;
        }
        const uint32_t q = t & 3u;
        return q == 0 ? cache.x : q == 1 ? cache.y : q == 2 ? cache.z : cache.w;
    }
};

// Integer in [0, n): multiply-shift of one word (Lemire, no rejection).
__device__ __forceinline__ uint32_t below(uint32_t x, uint32_t n)
{
    return (uint32_t)(((uint64_t)x * n) >> 32);
}

// Entries of the ascending list a[0, n) below x.
__device__ __forceinline__ size_t count_below(const uint64_t *a, size_t n, uint64_t x)
{
    size_t lo = 0, hi = n;
    while (lo < hi) {
        const size_t mid = (lo + hi) >> 1;
        if (a[mid] < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ uint64_t dkey(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ double keyd(uint64_t k) { return __longlong_as_double((long long)k); }
__device__ __forceinline__ uint64_t umin64(uint64_t a, uint64_t b) { return a < b ? a : b; }
__device__ __forceinline__ uint64_t umax64(uint64_t a, uint64_t b) { return a > b ? a : b; }

}  // namespace e2

// Host-side context (opaque to callers).
struct e2_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    cudaStream_t side = nullptr;                 // children of the generation step run here
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    e2::Dims dm{};
    double cong_lo = 0, cong_hi = 0;
    uint64_t thr_cx = 0, thr_half = 0, thr_mut = 0, thr_k1 = 0, thr_k2 = 0, thr_k3 = 0;
    // device pointers (all inside the caller's workspace)
    double *rate = nullptr, *bw = nullptr;
    uint64_t *mem = nullptr;
    double *rate_cpu = nullptr, *bw_cpu = nullptr;   // host side of offload (zeros without it)
    uint64_t *mem_cpu = nullptr;
    int32_t *capg = nullptr;                          // [V][M][2] blocks in device memory
    uint64_t *psum = nullptr;                         // [3][V][N+1] per-layer prefix sums PF, PB, PM (layered)
    double *lcost = nullptr;                          // [V][M][2][N][N] per-layer stage times (layered)
    int16_t *gpu_layers = nullptr;                    // [P][M] G of the G--C split (offload only)
    double *link_bw = nullptr, *cong = nullptr;
    uint64_t *prof = nullptr;
    double *leaf = nullptr;
    e2::LinkRec *tau = nullptr;
    uint4 *prec = nullptr;            // [M]
    float2 *prech = nullptr;          // [M]
    uint32_t *capv = nullptr;         // [M][V]
    float *ibw = nullptr;             // [M][M]
    float4 *fpr = nullptr;            // [V]
    uint64_t *leaf_sorted = nullptr;  // [V][pow2(2 M N)] sorted stage-time keys
    uint32_t *leaf_rank = nullptr;    // [V][M][2][LS]
    e2::DevPop pop[2]{};
    int cur = 0;
    double *fit = nullptr;
    int16_t *layers = nullptr, *master = nullptr, *bsel = nullptr;
    double *T = nullptr, *L = nullptr;
    uint64_t *hash = nullptr;
    int32_t *dup = nullptr, *elite = nullptr;
    unsigned long long *dup_tab = nullptr;   // [dup_table_size(P)] fingerprint table of the duplicate test
    double *elite_fit = nullptr;
    unsigned long long *elite_ctl = nullptr;   // [8]: threshold key of the elite selection, counts, path flag
    int32_t *elite_cand = nullptr;             // [P] its candidates
    unsigned long long *stats = nullptr;
    int32_t *err = nullptr;
    unsigned *list_ctrl = nullptr;    // [kCtrlWords]
    unsigned *list_hist = nullptr;    // [kListBlocks][kListBins]
    uint64_t *items = nullptr;        // [2*P*K] DP work items, largest replicas first
    int32_t *slot_off = nullptr;      // [P*K]
    uint32_t *slot_info = nullptr;    // [P*K]
    uint4 *drec = nullptr;            // [V][M]
    float *fxs = nullptr;             // [V]
    double *split_T = nullptr, *split_L = nullptr;   // [P*K][2]
    int16_t *split_mu = nullptr, *split_code = nullptr;   // [P*K][2]
    int16_t *split_layers = nullptr;                 // [P][2][M]
    double *var_T = nullptr, *var_L = nullptr;       // [P*K][V] (layered)
    int16_t *var_mu = nullptr, *var_layers = nullptr;   // [P*K][V], [P][V][M] (layered)
    int32_t *var_best = nullptr;                     // [P*K] (layered)
    mutable unsigned long long launches = 0;   // kernels launched (a graph replay adds its kernel nodes)
    unsigned long long gen_kernels[2] = {0, 0}; // kernel nodes of each recorded generation
    int dp_grid = 0;                  // persistent DP CTAs of class 0
    int dp_grid1 = 0;                 // persistent DP CTAs of class 1 (0: one class)
    size_t dp_smem1 = 0;              // their shared memory
    cudaEvent_t ev_dp_start = nullptr, ev_dp_stop = nullptr;   // optional timing hook
    // recorded generation (e2_run_generation), one per population buffer
    cudaStream_t cap_stream = nullptr;                          // private stream the graphs are recorded on
    cudaGraph_t gen_graph[2] = {nullptr, nullptr};
    cudaGraphExec_t gen_exec[2] = {nullptr, nullptr};
    cudaGraphNode_t gen_ga_node[2] = {nullptr, nullptr};        // the generation kernel's node
    cudaEvent_t gen_ev[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};   // timing events recorded in it
    bool gen_eager = false;                                     // recording failed: eager launches
    size_t dp_smem = 0;               // shared memory of class 0's CTAs
    bool evaluated = false;
    bool have_elites = false;
    bool have_results = false;           // an evaluation has filled the result buffers
    std::string last_error;
};

namespace e2 {
// A launch that may start while the kernel before it in the stream still runs
// (programmatic dependent launch): its blocks are placed as that kernel's run
// out and wait in after_previous() for its end, which hides launch latency (an
// eager evaluation of 512 offloading genomes of 32 devices: 104 -> 83 us; ten
// recorded generations of 1,024: 728 -> 710).  Every kernel launched so calls after_previous() first,
// in all its threads: its end then implies the end of all before it.
// early = false: an ordinary launch.
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool early, A... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Arrays of one device copied by one kernel (copy_kernel): blocks
// first[i]..first[i+1]-1 copy piece i, kCopyChunk bytes each.
constexpr int kCopyPieces = 7;
constexpr size_t kCopyChunk = 16 * 1024;
struct CopyList {
    const unsigned char *src[kCopyPieces];
    unsigned char *dst[kCopyPieces];
    unsigned long long bytes[kCopyPieces];
    unsigned first[kCopyPieces + 1];
    int n;
    int32_t *word;           // a word to set to kNoBadGenome besides (nullptr: none)
};

// The error word of an upload without an invalid genome (above every index).
constexpr int32_t kNoBadGenome = 0x7F7F7F7F;

// launchers (defined in the .cu files); return cudaGetLastError()
cudaError_t launch_copies(const CopyList &l, cudaStream_t st);
cudaError_t launch_tables(const e2_ctx *c);   // stage times and device tables (and lcost for per-layer profiles)
cudaError_t launch_tau(const e2_ctx *c);
cudaError_t launch_redraw(const e2_ctx *c, uint64_t seed, uint32_t gen);
cudaError_t launch_validate(const e2_ctx *c, const DevPop &p, bool early);
cudaError_t launch_eval(const e2_ctx *c, const DevPop &p);
cudaError_t launch_init(const e2_ctx *c, const DevPop &p, uint64_t seed);
cudaError_t launch_elites(const e2_ctx *c, const DevPop &p, const DevPop &dst, bool early);
cudaError_t launch_ga(const e2_ctx *c, const DevPop &src, const DevPop &dst, uint64_t seed, uint32_t gen,
                      cudaStream_t st);
// elites and children of the next population (children on the side stream);
// after_eval: right behind the evaluation's kernels
cudaError_t launch_step(const e2_ctx *c, const DevPop &src, const DevPop &dst, uint64_t seed, uint32_t gen,
                        bool after_eval);
// the generation kernel's node of a recorded graph, and new (seed, generation) for it
cudaError_t find_ga_node(cudaGraph_t graph, cudaGraphNode_t *node);
cudaError_t set_ga_node(const e2_ctx *c, cudaGraphExec_t exec, cudaGraphNode_t node, const DevPop &src,
                        const DevPop &dst, uint64_t seed, uint32_t gen);
// The DP of identical blocks (dp_order.cu) over class cls of the work list,
// for replicas of up to mmax devices, a run per warp: warps per CTA, shared
// memory per CTA, CTAs per SM and the launch.
__host__ __device__ constexpr int dp_order_warps(int cls) { return cls ? 4 : 12; }
size_t dp_order_smem(int mmax, int cls);
cudaError_t dp_order_occupancy(int mmax, int cls, bool off, int *per_sm);
cudaError_t dp_order_launch(int grid, int mmax, int cls, cudaStream_t stream, const Dims &dm, const Tables &tb,
                            const DevPop &pop, const EvalOut &out, const WorkList &wl, const int32_t *slot_off,
                            const SplitOut &so, bool early);
size_t dp_layered_smem_bytes(int M, int N);   // the per-layer DP's shared memory for the largest replica
cudaError_t configure_eval(e2_ctx *c);   // shared memory limit and persistent grid size
size_t rank_pow2(size_t n);
cudaError_t build_stage_keys(const e2_ctx *c);    // once per context, before launch_tau
}  // namespace e2
