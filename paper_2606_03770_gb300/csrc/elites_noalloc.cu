// elites_noalloc.cu -- elite selection for callers that cannot allocate
// device memory.
//
// The regular path (e2_ga_step) keeps its scratch (genome fingerprints and
// duplicate flags) in the workspace the caller allocated for a context.  Some
// callers cannot allocate at all: code running while a CUDA graph is being
// captured (cudaMalloc is not capturable), plug-ins inside a host framework
// whose allocator already owns the device memory and hands none out, or
// latency-critical loops that must never hit cudaMalloc's implicit device
// synchronisation.  e2_select_elites_noalloc serves them: the caller passes
// only its inputs (population and fitness) and its output (elite indices);
// the scratch lives in the file-scope array below, sized for at most
// E2_NOALLOC_MAX_POP genomes.  The array is part of the library's device image:
// every GPU that loads the library holds it (1.6 MiB) until the process exits.
//
// Every call shares that one array and leaves its contents behind.  Nothing in
// it has to start at zero (each call writes every entry it reads), but two
// calls that overlap on the GPU -- on different streams, or from different
// host threads -- race on it and must be serialised by the caller.
//
// The duplicate test and the selection are e2_ga_step's (elites.cuh), in the
// same order: fitness keys compared as the bit patterns of w and phase (the
// order of the values for the non-negative and +inf results an evaluation
// produces, and a total order for any other input).
//
// Bound by the read of the population for the fingerprints and by the
// selection's passes on one SM: 62 us for 16,384 genomes of 512 devices (two
// O(P^2) passes over the keys and a thread per genome for its fingerprint took
// 562).
#include <mutex>

#include "e2ga_internal.cuh"
#include "elites.cuh"

namespace {

constexpr int kNoallocMaxPop = E2_NOALLOC_MAX_POP;
constexpr int kMaxDeviceIds = 64;
constexpr int kWarps = 8;
// Populations up to this size skip the selection (dup_small_noalloc).  At 4,096
// genomes the quadratic ranking loses (53 us with Q = P against 31 for a
// selection), and the table no longer fits the 48 KB that any block may use.
constexpr int kSmallPop = 2048;

// Scratch: the fingerprints, the fingerprint table (reused for the candidate
// list once the duplicates are known), the duplicate flags and the selection's
// control words.
struct Scratch {
    uint64_t hash[kNoallocMaxPop];
    unsigned long long table[2 * kNoallocMaxPop];
    uint8_t dup[kNoallocMaxPop];
    unsigned long long ctl[8];
};
static __device__ __align__(256) Scratch g_noalloc_scratch;

// Device address of g_noalloc_scratch per device id, with the CUDA context
// that was current when it was looked up (a reset device gets a new context,
// and the address is looked up again).
struct ScratchSlot {
    void *ctx = nullptr;
    Scratch *addr = nullptr;
};
ScratchSlot g_scratch[kMaxDeviceIds];
std::mutex g_scratch_mutex;

// cuCtxGetCurrent, reached through the runtime's entry-point table (no link
// against the driver library).
typedef int (*CtxGetCurrentFn)(void **);

void *current_context()
{
    static CtxGetCurrentFn fn = nullptr;
    static bool looked = false;
    if (!looked) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<CtxGetCurrentFn>(p);
        else
            cudaGetLastError();
        looked = true;
    }
    void *ctx = nullptr;
    if (!fn || fn(&ctx) != 0) return nullptr;
    return ctx;
}

// A warp per genome; the blocks also clear the fingerprint table.  The
// fitness here is the caller's, so w and phase are part of what makes a
// duplicate (an evaluation gives equal genomes equal ones).
__global__ void __launch_bounds__(32 * kWarps) fingerprint_noalloc(e2::DevPop p, const uint64_t *fk, int P, int M, int K,
                                                                   Scratch *sc, unsigned slots)
{
    const int lane = threadIdx.x & 31, g = blockIdx.x * kWarps + (threadIdx.x >> 5);
    for (unsigned s = blockIdx.x * blockDim.x + threadIdx.x; s < slots; s += gridDim.x * blockDim.x)
        sc->table[s] = e2::kFreeSlot;
    if (g >= P) return;
    const int R = min((int)p.nclus[g], K);
    const int lo = lane < R ? p.sizes[(size_t)g * K + lane] : 0, hi = lane + 32 < R ? p.sizes[(size_t)g * K + lane + 32] : 0;
    const uint64_t h = e2::fingerprint(p.perm + (size_t)g * M, M, lo, hi, R, p.roles[g], lane,
                                       0x9E3779B97F4A7C15ull ^ fk[(size_t)g * 4] ^ (fk[(size_t)g * 4 + 1] << 1));
    if (lane == 0) sc->hash[g] = h;
}

__global__ void __launch_bounds__(256) insert_noalloc(int P, Scratch *sc, unsigned mask)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < P) e2::table_insert(sc->table, mask, sc->hash[g], g);
}

__global__ void __launch_bounds__(32 * kWarps) dup_noalloc(e2::DevPop p, const uint64_t *fk, int P, int M, int K, Scratch *sc,
                                                           unsigned mask)
{
    const int lane = threadIdx.x & 31, g = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (g >= P) return;
    const bool d = e2::is_duplicate(p, sc->table, mask, sc->hash, g, M, K, lane, fk);
    if (lane == 0) sc->dup[g] = d;
}

// Small populations: the duplicates through a table per block, and the ranks of
// all genomes without a selection.  Three short kernels, the last two placed
// early: 8 us for 64 genomes of 32 devices, 14 for 1,024, 25 for 2,048; the five
// kernels below, bound by their chain, take 25, 28 and 29.
__global__ void __launch_bounds__(e2::kDupThreads) dup_small_noalloc(e2::DevPop p, const uint64_t *fk, int P, int M, int K,
                                                                     Scratch *sc, unsigned mask)
{
    e2::after_previous();
    extern __shared__ unsigned long long tab[];
    e2::flag_duplicates(tab, mask, p, sc->hash, sc->dup, P, M, K, fk);
}

__global__ void __launch_bounds__(32 * kWarps) rank_small_noalloc(int P, int Q, const double *fit, const Scratch *sc,
                                                                  int32_t *elite)
{
    e2::after_previous();
    __shared__ e2::EliteTile tile;
    e2::rank_all(tile, P, Q, fit, sc->dup, [&](int rank, int g, int lane) {
        if (lane == 0) elite[rank] = g;
    });
}

// The listed genomes' ranks; with fewer than Q distinct genomes, the ranks of
// all of them.  Bound by the comparisons of every pair: 312 us for 16,384
// genomes of 32 devices and 3.9 ms for 65,536; by strided reads of the caller's
// rows instead of tiles 594 us and 8.0 ms, on half the blocks 349 us and 4.5 ms.
__global__ void __launch_bounds__(32 * kWarps) rank_noalloc(int P, int Q, const double *fit, const Scratch *sc, int32_t *elite)
{
    __shared__ e2::EliteTile tile;
    auto take = [&](int rank, int g, int lane) {
        if (lane == 0) elite[rank] = g;
    };
    if (sc->ctl[2] != 0) e2::rank_listed(tile, Q, fit, sc->ctl, reinterpret_cast<const int32_t *>(sc->table), take);
    else e2::rank_all(tile, P, Q, fit, sc->dup, take);
}

// Device memory of device `dev` (or managed memory).
bool on_device(const void *p, int dev)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type == cudaMemoryTypeManaged) return true;
    return a.type == cudaMemoryTypeDevice && a.device == dev;
}

// Statuses only: this entry point keeps no error text.
int reject(int code, const char *) { return code; }

}  // namespace

extern "C" int e2_select_elites_noalloc(const e2_genomes *pop, const double *fitness, int32_t P, int32_t M,
                                        int32_t K_max, int32_t Q, int32_t *elite_idx, void *stream)
{
    if (!pop || !pop->perm || !pop->sizes || !pop->nclus || !pop->roles || !fitness)
        return reject(E2_EINVAL, "null input");
    if (P < 1 || P > kNoallocMaxPop) return reject(E2_EINVAL, "P must lie in [1, E2_NOALLOC_MAX_POP]");
    if (M < 1 || M > E2_MAX_DEVICES || K_max < 1 || K_max > E2_MAX_CLUSTERS || Q < 0 || Q > P)
        return reject(E2_EINVAL, "M, K_max or Q out of range");
    if (Q > 0 && !elite_idx) return reject(E2_EINVAL, "null output");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return reject(E2_ECUDA, "cudaGetDevice failed");
    if (dev < 0 || dev >= kMaxDeviceIds) return reject(E2_EINVAL, "device id beyond the supported range");
    if (!on_device(pop->perm, dev) || !on_device(pop->sizes, dev) || !on_device(pop->nclus, dev) ||
        !on_device(pop->roles, dev) || !on_device(fitness, dev) || (Q > 0 && !on_device(elite_idx, dev)))
        return reject(E2_EINVAL, "inputs and output must be device memory of the current device");
    Scratch *sc = nullptr;
    {
        // set-up, once per device and context: the scratch array's device
        // address, looked up with that device current
        std::lock_guard<std::mutex> lock(g_scratch_mutex);
        void *ctx = current_context();
        ScratchSlot &sl = g_scratch[dev];
        if (!sl.addr || sl.ctx != ctx) {
            void *addr = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&addr, g_noalloc_scratch);
            if (e != cudaSuccess || !addr) {
                cudaGetLastError();
                return reject(E2_ECUDA, "cudaGetSymbolAddress of the scratch array failed");
            }
            sl.addr = static_cast<Scratch *>(addr);
            sl.ctx = ctx;
        }
        sc = sl.addr;
    }
    const e2::DevPop p{pop->perm, pop->sizes, pop->nclus, pop->roles};
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const uint64_t *fk = reinterpret_cast<const uint64_t *>(fitness);
    const unsigned slots = e2::dup_table_size(P);
    const unsigned wblocks = (unsigned)((P + kWarps - 1) / kWarps);
    if (P <= kSmallPop) {
        fingerprint_noalloc<<<wblocks, 32 * kWarps, 0, s>>>(p, fk, P, M, K_max, sc, 0);
        // (a genome per warp: the blocks are one wave whatever P)
        const unsigned per = e2::kDupThreads / 32;
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess)
            e = e2::launch_kernel(dup_small_noalloc, ((unsigned)P + per - 1) / per, e2::kDupThreads,
                                  sizeof(unsigned long long) * slots, s, true, p, fk, P, M, K_max, sc, slots - 1);
        if (e == cudaSuccess && Q > 0)
            // (early only up to a block per SM: placed while the kernel before it runs, more of
            // them crowd on the SMs that it leaves free, 31 us instead of 24 at 2,048 genomes)
            e = e2::launch_kernel(rank_small_noalloc, wblocks, 32 * kWarps, 0, s, wblocks <= 152, P, Q, fitness, sc,
                                  elite_idx);
        return e == cudaSuccess ? E2_OK : reject(E2_ECUDA, cudaGetErrorString(e));
    }
    fingerprint_noalloc<<<wblocks, 32 * kWarps, 0, s>>>(p, fk, P, M, K_max, sc, slots);
    insert_noalloc<<<(unsigned)((P + 255) / 256), 256, 0, s>>>(P, sc, slots - 1);
    dup_noalloc<<<wblocks, 32 * kWarps, 0, s>>>(p, fk, P, M, K_max, sc, slots - 1);
    if (Q > 0) {
        e2::elite_select_kernel<<<1, e2::kSelThreads, 0, s>>>(P, Q, fitness, sc->dup, sc->ctl,
                                                                reinterpret_cast<int32_t *>(sc->table));
        // (at most eight blocks per SM)
        rank_noalloc<<<wblocks < 1216 ? wblocks : 1216, 32 * kWarps, 0, s>>>(P, Q, fitness, sc, elite_idx);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return reject(E2_ECUDA, cudaGetErrorString(e));
    return E2_OK;
}
