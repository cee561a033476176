// dp_eval.cu -- population fitness around the DP: the pre-pass, the work list,
// the DP of models with several block types, the objective (Eq. 3-5) and the
// launch sequence of an evaluation.
//
// An evaluation is a pre-pass that decides, per (genome, replica slot) and
// role, which decode batches (or whether the prefill run) can matter (memory
// and latency bounds); a count and a scatter that put the surviving work into
// one list, by replica size; the DP (dp_order.cu for identical blocks,
// dp_layered_kernel here for blocks of several types), persistent warps or
// CTAs over the list; and a warp per genome (a block per genome for a wide
// role search) that scores the genome.
#include "e2ga_internal.cuh"
#include "elites.cuh"

namespace e2 {

namespace {

// Candidates (mu, k, i, j) the plain recurrence examines for one DP run:
// m * (N + sum_{k=2..m} (N-k+1)(N-k+2)/2).
__device__ __forceinline__ unsigned long long paper_candidates(int m, int N)
{
    const unsigned long long a = (unsigned long long)(N - m + 1), b = (unsigned long long)(N - 1);
    unsigned long long s = 0;
    if (m >= 2) s = (b * (b + 1) * (b + 2) - (a - 1) * a * (a + 1)) / 6;
    return (unsigned long long)m * ((unsigned long long)N + s);
}

// A warp's sum, in every lane.
__device__ __forceinline__ int warp_sum(int x) { return __reduce_add_sync(0xFFFFFFFFu, x); }

}  // namespace

// Bin of a replica of m devices in the work list: with two DP classes, the
// sizes up to dp_split (class 0) take bins 0..31 and the larger ones bins
// 32..63; larger first within a class.
__device__ __forceinline__ uint32_t size_bin(const Dims &dm, int m)
{
    constexpr int half = kListBins / 2;
    if (!dm.dp_split) return (uint32_t)(kListBins - 1 - (m - 1) * kListBins / dm.dp_mmax);
    if (m <= dm.dp_split) return (uint32_t)(half - 1 - (m - 1) * half / dm.dp_split);
    return (uint32_t)(kListBins - 1 - (m - dm.dp_split - 1) * half / (dm.dp_mmax - dm.dp_split));
}

// Pre-pass, one block per genome, a warp per replica at a time.  For each
// variant of the replica (prefill: v = 0; decode: v = 1..b_max, bit v-1) the
// warp decides whether a DP run can matter:
//  * memory: with identical blocks a partition with master mu exists iff every
//    device holds >= 1 block and the capacities, capped at W = N - m + 1, add
//    up to N (exact);
//  * decode latency: Lambda >= sum of link times + sum_k n_k c_k (c_k the
//    per-block time; the head only adds), at least, for any price x >= 0,
//        x (N - m) + sum_k c_k + sum_{c_k < x} (cap_k - 1) (c_k - x)
//    (the linear program's dual: one block on each device, the other N - m
//    bought at x, less what devices cheaper than x save).  The block time of
//    the marginal device, up to which the cheaper devices just hold N - m more
//    blocks, gives the program's own optimum; it is found by bisection at the
//    smallest and the largest batch and kept for those between.  All in float
//    from times rounded down, every operation rounded toward -inf, so the bound
//    never exceeds the exact value; a variant whose bound is above Lambda_max
//    (rounded up to float) fails whatever partition the DP returns.
// With blocks of several types the capacities are the longest run of blocks each
// device holds and c_k comes from the least block's flops and bytes, so both
// tests stay necessary conditions: at 32 devices they drop 5,400 of 9,900 runs
// (evaluation 552 -> 432 us).
// Both tests are monotone in the batch: the capacities shrink as b grows (more
// KV memory per block), and the program's optimum is the least of a linear
// cost whose coefficients (per-block and link times) grow with b over a
// feasible set that shrinks with b, when the profile's costs grow with the
// batch (physical profiles do; checked at e2_create).  So each is tried on the
// smallest batch first; if that passes, the largest batch the memory allows is
// found by a search (the largest batch first, then bisection), and the largest
// the bound keeps by a second search below it; every smaller batch is kept.  A
// failed test is exact (memory, identical blocks) or a proof (the bound never
// exceeds the optimum, and the optimum of every larger batch is no smaller), so
// every batch above it fails too;
// rounding and the price can only keep a variant the optimum would drop,
// which costs a DP run and changes no result.  Other profiles test every
// batch from the largest down, and the first that passes keeps the smaller
// ones.
// The verdicts go into the slot's info word (kSlot*), with the bin of its
// size in the work list's order.  A replica with nothing to run (more devices
// than blocks, no variant left) gets its outputs here, and so do the empty
// slots.
//
// Bound by the chain of dependent reads per replica (device, its record and
// link, the verdicts).  Per device one 16-byte record serves every variant
// (1 / rate, 1 / bandwidth, the capacities of the smallest and the largest
// batch), and one 1 / bandwidth per link every batch's link time, so a second
// variant reads nothing.
constexpr int kPreWarps = 8;

// A replica's devices for the pre-pass: lane k holds device k (SMALL: at most
// 32 devices) or visits devices k, k + 32, ...
template <bool SMALL, typename F>
__device__ __forceinline__ void each_device(int m, int lane, F f)
{
    if (SMALL) {
        if (lane < m) f(lane);
    } else {
#pragma unroll 1
        for (int k = lane; k < m; k += 32) f(k);
    }
}

// Whether the capacities (without | with the head << 16 of each device) admit
// a partition of N blocks.
template <bool SMALL, typename Caps>
__device__ __forceinline__ bool memory_ok(int m, int N, int lane, Caps caps)
{
    const int W = N - m + 1;
    int s = 0;
    uint32_t own = 0;
    each_device<SMALL>(m, lane, [&](int k) {
        const uint32_t x = caps(k);
        own = x;
        const int c0 = min((int)(x & 0xFFFFu), W);
        s += c0 + (c0 == 0 ? 1 << 20 : 0);
    });
    s = warp_sum(s);
    const int zero = s >> 20, S = s & 0xFFFFF;
    bool ok = false;
    each_device<SMALL>(m, lane, [&](int k) {
        const uint32_t x = SMALL ? own : caps(k);
        const int c0 = min((int)(x & 0xFFFFu), W), c1 = min((int)(x >> 16), W);
        ok |= zero - (c0 == 0) == 0 && c1 >= 1 && S - c0 + c1 >= N;
    });
    return __any_sync(0xFFFFFFFFu, ok);
}

__device__ __forceinline__ float warp_sum_rd(float x)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) x = __fadd_rd(x, __shfl_xor_sync(0xFFFFFFFFu, x, o));
    return x;
}

// The decode verdicts of a replica on devices dev[0..m-1]: the largest batch
// its memory allows and, of those, the largest the latency bound keeps.
template <bool SMALL>
__device__ __forceinline__ uint32_t decode_verdict(const Dims &dm, const Tables &tb, const uint16_t *dev, int m, int lane)
{
    const int M = dm.M, N = dm.N, W = N - m + 1, need = N - m;
    const bool timed = dm.min_tps > 0.0;                   // the latency bound applies
    // lane k's device and its link, kept; the devices beyond 32 are read again
    const uint4 mine = lane < m ? tb.prec[dev[lane]] : make_uint4(0, 0, 0, 0);
    float X = 0.0f;                                        // sum of the links' 1 / bandwidth
    if (timed) each_device<SMALL>(m, lane, [&](int k) {
        if (k >= 1) X = __fadd_rd(X, tb.ibw[(size_t)dev[k - 1] * M + dev[k]]);
    });
    auto rec = [&](int k) -> uint4 { return SMALL || k == lane ? mine : tb.prec[dev[k]]; };
    auto caps = [&](int k, int v) -> uint32_t {
        if (v == 1) return rec(k).z;
        if (v == dm.b_max) return rec(k).w;
        return tb.capv[(size_t)dev[k] * dm.V + v];
    };
    if (timed) X = warp_sum_rd(X);
    auto mem_of = [&](int v) { return memory_ok<SMALL>(m, N, lane, [&](int k) { return caps(k, v); }); };
    // the marginal device: the price is its block time (found at the smallest batch
    // and again at the largest, and kept: which devices are cheap hardly depends on
    // the batch, but how much they hold does)
    int marginal = -1;
    auto fast_enough = [&](int v) -> bool {
        const float4 q = tb.fpr[v];                        // block flops and bytes, activation bytes, rounded down
        auto cost = [&](int k) -> float {                  // a block's time, rounded down
            const uint4 r = rec(k);
            float t = fmaxf(__fmul_rd(q.x, __uint_as_float(r.x)), __fmul_rd(q.y, __uint_as_float(r.y)));
            if (dm.offload) {
                const float2 h = tb.prech[dev[k]];
                if (h.x > 0.0f) t = fminf(t, fmaxf(__fmul_rd(q.x, h.x), __fmul_rd(q.y, h.y)));
            }
            return t;
        };
        float c_own = 0.0f;
        int e_own = 0;
        if (lane < m) {
            c_own = cost(lane);
            e_own = min((int)(caps(lane, v) & 0xFFFFu), W) - 1;
        }
        auto c_of = [&](int k) -> float { return SMALL || k == lane ? c_own : cost(k); };
        auto e_of = [&](int k) -> int { return SMALL || k == lane ? e_own : min((int)(caps(k, v) & 0xFFFFu), W) - 1; };
        float price = 0.0f;
        if (need > 0) {
            if (marginal < 0) {
                uint32_t lo = 0x7F800000u, hi = 0;         // (bits order as the non-negative values)
                each_device<SMALL>(m, lane, [&](int k) {
                    const uint32_t x = __float_as_uint(c_of(k));
                    lo = min(lo, x);
                    hi = max(hi, x);
                });
                lo = __reduce_min_sync(0xFFFFFFFFu, lo);
                hi = __reduce_max_sync(0xFFFFFFFFu, hi);
#pragma unroll 1
                for (int it = 0; it < 7 && lo < hi; ++it) {
                    const uint32_t mid = lo + ((hi - lo) >> 1);
                    int s = 0;
                    each_device<SMALL>(m, lane, [&](int k) { if (__float_as_uint(c_of(k)) <= mid) s += e_of(k); });
                    if (warp_sum(s) >= need) hi = mid;
                    else lo = mid + 1;
                }
                // the dearest device at or below the price found (there is one: the cheapest)
                unsigned best = 0;
                int at = 0;
                each_device<SMALL>(m, lane, [&](int k) {
                    const uint32_t x = __float_as_uint(c_of(k));
                    if (x <= hi && x >= best) { best = x; at = k; }
                });
                const unsigned top = __reduce_max_sync(0xFFFFFFFFu, best);
                marginal = (int)__reduce_max_sync(0xFFFFFFFFu, best == top && lane < m ? (unsigned)at : 0u);
            }
            price = SMALL ? __shfl_sync(0xFFFFFFFFu, c_own, marginal) : cost(marginal);
        }
        float sum = 0.0f;
        each_device<SMALL>(m, lane, [&](int k) {
            const float ck = c_of(k);
            sum = __fadd_rd(sum, ck);
            if (ck < price) sum = __fadd_rd(sum, __fmul_rd((float)e_of(k), __fsub_rd(ck, price)));
        });
        sum = warp_sum_rd(sum);
        sum = __fadd_rd(sum, __fmul_rd(price, (float)need));
        sum = __fadd_rd(sum, __fmul_rd(q.z, X));
        return !(sum > dm.lam_max_up);                     // 1.0 / Lambda >= Min_TPS possible
    };
    // the largest batch above lo, from top down, that a test passes (lo: none does)
    auto search = [&](int lo, int top, auto pass) -> int {
        int hi = top + 1, next = top;
#pragma unroll 1
        while (hi - lo > 1) {
            if (pass(next)) lo = next;
            else hi = next;
            next = dm.grows ? (lo + hi) >> 1 : hi - 1;
        }
        return lo;
    };
    int bm = 0, bs = 0;
    if (dm.grows) {
        // the smallest batch first: its capacities are at hand, and a replica that
        // cannot hold it (72% of a 512-device population), or is too slow with it,
        // fails at every other (512 devices: 273-320 us with the largest batch first,
        // 260 so; 256 devices, where most serve the largest: 125-130 and 147, and the
        // price found here saves DP runs, so the evaluation is no slower)
        if (mem_of(1)) {
            bm = search(1, dm.b_max, mem_of);
            if (!timed) {
                bs = bm;
            } else if (fast_enough(1)) {
                marginal = -1;                             // (found again at the largest batch's capacities)
                bs = search(1, bm, fast_enough);
            }
        }
    } else {
        bm = search(0, dm.b_max, mem_of);
        bs = timed ? search(0, bm, [&](int v) { return mem_of(v) && fast_enough(v); }) : bm;
    }
    return kSlotDecTested | (uint32_t)bs | (uint32_t)bm << kSlotMemShift;
}

__global__ void __launch_bounds__(32 * kPreWarps, 5) slot_kernel(Dims dm, Tables tb, DevPop pop, SlotInfo si, EvalOut out,
                                                              SplitOut so, VariantOut vo)
{
    after_previous();
    extern __shared__ uint16_t s_perm[];                   // the genome's ordering
    __shared__ int s_off[E2_MAX_CLUSTERS], s_size[E2_MAX_CLUSTERS];
    const int g = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, NW = blockDim.x >> 5;
    const int K = dm.K, M = dm.M, N = dm.N;
    const int R = pop.nclus[g];
    const uint64_t roles = pop.roles[g];
    const size_t base = (size_t)g * K;
    if (wid == 0) {                                        // replica offsets: a scan of the sizes
        const int lo = lane < R ? pop.sizes[base + lane] : 0;
        const int hi = lane + 32 < R ? pop.sizes[base + lane + 32] : 0;
        int a = lo, b = hi;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xFFFFFFFFu, a, o), y = __shfl_up_sync(0xFFFFFFFFu, b, o);
            if (lane >= o) { a += x; b += y; }
        }
        b += __shfl_sync(0xFFFFFFFFu, a, 31);
        if (lane < R) { s_off[lane] = a - lo; s_size[lane] = lo; si.off[base + lane] = a - lo; }
        if (lane + 32 < R) { s_off[lane + 32] = b - hi; s_size[lane + 32] = hi; si.off[base + lane + 32] = b - hi; }
    }
    for (int i = tid; i < M; i += blockDim.x) s_perm[i] = pop.perm[(size_t)g * M + i];
    for (int c = R + tid; c < K; c += blockDim.x) {        // the empty slots
        si.info[base + c] = 0;
        out.master[base + c] = -1; out.bsel[base + c] = -1;
        out.T[base + c] = keyd(kInfKey); out.L[base + c] = keyd(kInfKey);
    }
    __syncthreads();
    for (int c = wid; c < R; c += NW) {
        const int off = s_off[c], m = s_size[c], role = (int)((roles >> c) & 1ull);
        const size_t slot = base + c;
        uint32_t info = 0;
        if (m <= N) {
            const uint16_t *dev = s_perm + off;
            if (dm.role_search || !role) {
                auto caps = [&](int k) { return tb.drec[dev[k]].x; };
                const bool ok = m <= 32 ? memory_ok<true>(m, N, lane, caps) : memory_ok<false>(m, N, lane, caps);
                info |= kSlotPreTested | (ok ? kSlotPrefill : 0u);
            }
            if (dm.role_search || role)
                info |= m <= 32 ? decode_verdict<true>(dm, tb, dev, m, lane) : decode_verdict<false>(dm, tb, dev, m, lane);
            info |= size_bin(dm, m) << kSlotBinShift;
        }
        // ---- the slot's verdicts, and the outputs of a replica that cannot serve
        const bool dec = (info & kSlotDecMask) != 0, pre = (info & kSlotPrefill) != 0;
        if (lane == 0) {
            si.info[slot] = info;
            if (dm.layered) vo.best[slot] = -1;
        }
        if (dm.role_search) {
            if (lane == 0) {
                if (!pre) so.code[slot * 2] = -1;
                if (!dec) so.code[slot * 2 + 1] = -1;
            }
        } else if (!dec && !pre) {
            for (int k = lane; k < m; k += 32) out.layers[(size_t)g * M + off + k] = -1;
            if (lane == 0) {
                out.master[slot] = -1; out.bsel[slot] = -1;
                out.T[slot] = keyd(kInfKey); out.L[slot] = keyd(kInfKey);
            }
        }
    }
}

// The work list's order: class 0 (the first DP launch) before class 1, larger
// replicas first within a class, in kListBins bins of equal size ranges.  The
// count (bins_kernel) and the scatter split the slots into the same chunks,
// one per block; a block of the scatter gets its place in each bin from the
// counts of the blocks before it, so neither takes a global atomic.
// With per-layer profiles (long runs, few of them) each batch of a decode sweep
// is an item of its own, all replicas' largest batches first: by the time the
// smaller ones come up the larger one has usually been decided.
__device__ __forceinline__ int items_of(uint32_t info)
{
    return ((info & kSlotDecMask) != 0) + ((info & kSlotPrefill) != 0);
}

__device__ __forceinline__ uint32_t layered_bin(uint32_t info, int level)
{
    return (uint32_t)min(level, 7) * 8u + (info >> kSlotBinShift) / (kListBins / 8);
}

__global__ void __launch_bounds__(256) bins_kernel(Dims dm, SlotInfo si, unsigned *hist, unsigned long long *stats)
{
    after_previous();
    __shared__ unsigned s_bin[kListBins];
    const int total = dm.P * dm.K, chunk = (total + gridDim.x - 1) / gridDim.x;
    const int lo = blockIdx.x * chunk, hi = min(total, lo + chunk);
    for (int b = threadIdx.x; b < kListBins; b += blockDim.x) s_bin[b] = 0;
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < kNumStats; i += blockDim.x) stats[i] = 0;
    __syncthreads();
    for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        const uint32_t info = si.info[i];
        const int n = items_of(info);
        if (dm.layered) {
            for (int lv = 0; lv < (int)(info & kSlotDecMask); ++lv) atomicAdd(&s_bin[layered_bin(info, lv)], 1u);
            if (info & kSlotPrefill) atomicAdd(&s_bin[layered_bin(info, 0)], 1u);
        } else if (n) {
            atomicAdd(&s_bin[info >> kSlotBinShift], (unsigned)n);
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kListBins; b += blockDim.x) hist[(size_t)blockIdx.x * kListBins + b] = s_bin[b];
}

// Items are (slot << 8) | role << 7 | top: the decode sweep (role 1) from batch
// top + 1 down (per-layer profiles: that batch), or the prefill run (role 0).  Block 0 also sets the classes'
// ends and cursors.
__global__ void __launch_bounds__(256) order_scatter_kernel(Dims dm, SlotInfo si, WorkList wl, const unsigned *hist)
{
    after_previous();
    __shared__ unsigned s_all[4][kListBins], s_before[4][kListBins], s_at[kListBins];
    const int total = dm.P * dm.K, chunk = (total + gridDim.x - 1) / gridDim.x;
    const int lo = blockIdx.x * chunk, hi = min(total, lo + chunk);
    {
        const int b = threadIdx.x & (kListBins - 1), part = threadIdx.x / kListBins;
        unsigned all = 0, before = 0;
        for (int q = part; q < (int)gridDim.x; q += 4) {
            const unsigned x = hist[(size_t)q * kListBins + b];
            all += x;
            if (q < (int)blockIdx.x) before += x;
        }
        s_all[part][b] = all;
        s_before[part][b] = before;
    }
    __syncthreads();
    if (threadIdx.x < kListBins) {
        const int b = threadIdx.x;
        unsigned start = 0;                                  // all items of the bins before b
        for (int q = 0; q < b; ++q) start += s_all[0][q] + s_all[1][q] + s_all[2][q] + s_all[3][q];
        s_at[b] = start + s_before[0][b] + s_before[1][b] + s_before[2][b] + s_before[3][b];
        if (blockIdx.x == 0) {
            const unsigned end = start + s_all[0][b] + s_all[1][b] + s_all[2][b] + s_all[3][b];
            if (b == 0) wl.ctrl[kCtrlNext] = 0;
            if (b == kListBins - 1) wl.ctrl[kCtrlEnd + 1] = end;
            if (b == (dm.dp_split ? kListBins / 2 : kListBins) - 1) wl.ctrl[kCtrlEnd] = wl.ctrl[kCtrlNext + 1] = end;
        }
    }
    __syncthreads();
    for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        const uint32_t info = si.info[i];
        const int n = items_of(info);
        if (!n) continue;
        const uint64_t slot = (uint64_t)i << 8;
        if (dm.layered) {
            const int top = (int)(info & kSlotDecMask) - 1;
            for (int bit = top; bit >= 0; --bit)
                wl.items[atomicAdd(&s_at[layered_bin(info, top - bit)], 1u)] = slot | 0x80u | (unsigned)bit;
            if (info & kSlotPrefill) wl.items[atomicAdd(&s_at[layered_bin(info, 0)], 1u)] = slot;
            continue;
        }
        unsigned at = atomicAdd(&s_at[info >> kSlotBinShift], (unsigned)n);
        if (info & kSlotDecMask) wl.items[at++] = slot | 0x80u | ((info & kSlotDecMask) - 1u);
        if (info & kSlotPrefill) wl.items[at] = slot;
    }
}

// ---------------------------------------------------------------------------
// Blocks of several types (per-layer prefix sums).
//
// A stage's cost now depends on where it starts, and the best bottleneck of a
// prefix is no longer monotone in its length (a heavy block can make fewer
// blocks cost more).  The columns are Eq. 1's, on the float64 times themselves
// (their bit patterns, which order like the values), read from the per-layer
// cost table:
//   F_k[r] = min_s max(F_{k-1}[s], l_k(s+k-1 .. r+k-1), tau_k)     devices 1..k, no master
//   G_k[b] = min_u max(G_{k+1}[u], l_k(the b-u+1 blocks before them), tau_{k+1})   devices k..m
//   V_mu   = min_{a,b} max(F_{mu-1}[a], l^head_mu(the W-a-b blocks between), G_{mu+1}[b], tau_mu, tau_mu+1)
// The stage time falls as the split s rises (fewer blocks), so a split may be
// charged the least F over all splits from s on without changing the minimum:
// that range minimum rises with s, the stage time falls, and the cell is at
// their crossover, found by bisection instead of a scan over the splits.
// Range minima come from a sparse table of the previous column (minima over
// 2^l entries), rebuilt per column.  A master's (a, b) search bisects over a
// for each b in the same way.
// mu* = the smallest mu with the least V_mu; masters are tried four at a time
// until one reaches the master-free optimum F_m (the head only adds).  mu*'s
// prefix columns are recomputed from column mu* on, and the traceback takes
// the smallest split attaining each cell's value.  Every value and tie is the
// oracle's.
//
// Bound by latency: about log2(W) dependent table reads (L2) per column.  The
// scan it replaces made W / 2 reads per cell.
// ---------------------------------------------------------------------------
constexpr int kLayeredWarps = 4;

// Levels above the column itself in the sparse table of W entries.
__host__ __device__ __forceinline__ unsigned sparse_levels(unsigned W)
{
    unsigned l = 0;
    while ((2u << l) <= W) ++l;
    return l;
}

__host__ __device__ __forceinline__ unsigned dp_layered_item_bytes(int m, int N)
{
    const unsigned W = (unsigned)(N - m + 1);
    const unsigned keys = 2u * (unsigned)m * W + kLayeredWarps * sparse_levels(W) * W + 2u * (unsigned)m;
    return (8u * keys + 4u * (unsigned)m + 2u * (unsigned)m + 15u) & ~15u;
}

size_t dp_layered_smem_bytes(int M, int N)
{
    size_t best = 0;
    const int mmax = M < N ? M : N;
    for (int m = 1; m <= mmax; ++m) {
        const size_t b = dp_layered_item_bytes(m, N);
        if (b > best) best = b;
    }
    return best;
}

// The sparse table of a column by n threads (id 0..n-1), which `sync` joins:
// sp[(l-1) W + i] = min col[i .. i + 2^l - 1].
template <typename Sync>
__device__ __forceinline__ void sparse_build(const uint64_t *col, uint64_t *sp, int W, int id, int n, Sync sync)
{
    const uint64_t *below = col;
    for (int half = 1; 2 * half <= W; half *= 2) {
        for (int i = id; i + 2 * half <= W; i += n) sp[i] = umin64(below[i], below[i + half]);
        below = sp;
        sp += W;
        sync();
    }
}

// min col[s .. r] (s <= r)
__device__ __forceinline__ uint64_t range_min(const uint64_t *col, const uint64_t *sp, int W, int s, int r)
{
    const int l = 31 - __clz(r - s + 1);
    const uint64_t *t = l ? sp + (size_t)(l - 1) * W : col;
    return umin64(t[s], t[r - (1 << l) + 1]);
}

// min over s in [0, r] of max(col[s], cost(s)), cost non-increasing in s.
template <typename Cost>
__device__ __forceinline__ uint64_t crossover(const uint64_t *col, const uint64_t *sp, int W, int r, Cost cost)
{
    int lo = 0, hi = r + 1;
    uint64_t left = kInfKey, right = kInfKey;     // cost just before the crossover, range minimum at it
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const uint64_t c = cost(mid), q = range_min(col, sp, W, mid, r);
        if (q >= c) { hi = mid; right = q; }
        else { lo = mid + 1; left = c; }
    }
    return umin64(left, right);
}

__device__ __forceinline__ void bar_named(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

__global__ void __launch_bounds__(32 * kLayeredWarps) dp_layered_kernel(Dims dm, Tables tb, DevPop pop, EvalOut out,
                                                                        WorkList wl, SlotInfo si, VariantOut vo)
{
    after_previous();
    extern __shared__ __align__(16) unsigned char lsm[];
    __shared__ unsigned s_item;
    __shared__ int s_done, s_mu;
    __shared__ unsigned long long s_V0, s_V;
    __shared__ double s_T, s_L;
    const int K = dm.K, M = dm.M, N = dm.N;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint64_t INF = kInfKey;
    const unsigned n_items = wl.ctrl[kCtrlEnd];
    const size_t NN = (size_t)N * N;
    for (;;) {
        if (tid == 0) s_item = atomicAdd(&wl.ctrl[kCtrlNext], 1u);
        __syncthreads();
        const unsigned idx = s_item;
        __syncthreads();
        if (idx >= n_items) break;
        const uint64_t item = wl.items[idx];
        const int slot = (int)(item >> 8), code = (int)(item & 0x3Fu);
        if (tid == 0) s_done = (item >> 7 & 1u) && *(volatile const int32_t *)&vo.best[slot] > code;
        __syncthreads();
        if (s_done) continue;                                     // a larger batch won
        const int g = slot / K;
        const int off = si.off[slot], m = pop.sizes[slot];
        const int role = (int)((item >> 7) & 1u);
        const int v = role ? code + 1 : 0;
        const size_t sv = (size_t)slot * dm.V + v;
        const int W = N - m + 1;
        const size_t levels = sparse_levels((unsigned)W);
        uint64_t *F = reinterpret_cast<uint64_t *>(lsm);          // [m][W] prefix (then mu*'s) columns
        uint64_t *G = F + (size_t)m * W;                          // [m][W] suffix columns
        uint64_t *sp = G + (size_t)m * W;                         // [warps][levels][W] sparse tables
        uint64_t *Vmu = sp + kLayeredWarps * levels * W;          // [m]
        uint64_t *tk = Vmu + m;                                   // [m] tk[k] = link k-1 -> k (0-based)
        int *nk = reinterpret_cast<int *>(tk + m);                // [m]
        uint16_t *devs = reinterpret_cast<uint16_t *>(nk + m);    // [m]
        uint64_t *spw = sp + (size_t)wid * levels * W;            // this warp's table
        const double *lc = tb.lcost + (size_t)v * M * 2 * NN;
        for (int k = tid; k < m; k += blockDim.x) devs[k] = pop.perm[(size_t)g * M + off + k];
        __syncthreads();
        for (int k = tid; k < m; k += blockDim.x)
            tk[k] = k ? dkey(tb.tau[((size_t)v * M + devs[k - 1]) * M + devs[k]].t) : 0ull;
        // device k's (0-based) times: entry [j][n - 1] of blocks j .. j+n-1, with the head when mf
        auto rows = [&](int k, int mf) -> const double * { return lc + ((size_t)devs[k] * 2 + mf) * NN; };
        unsigned long long probes = 0;
        for (int r = tid; r < W; r += blockDim.x) {
            F[r] = dkey(rows(0, 0)[r]);
            G[(size_t)(m - 1) * W + r] = dkey(rows(m - 1, 0)[(size_t)(N - 1 - r) * N + r]);
        }
        __syncthreads();
        // cell r of device k's prefix column (0-based k >= 1), from column k - 1
        auto prefix_cell = [&](const uint64_t *prev, const uint64_t *s_prev, int k, int mf, int r) -> uint64_t {
            const double *t = rows(k, mf);
            return umax64(crossover(prev, s_prev, W, r, [&](int s) {
                              ++probes;
                              return dkey(t[(size_t)(s + k) * N + (r - s)]);
                          }), tk[k]);
        };
        // ---- prefix columns 1..m-2 on warps 0-1, suffix columns m-2..1 on warps 2-3
        if (wid < 2) {
            auto join = [] { bar_named(1, 64); };
            for (int k = 1; k <= m - 2; ++k) {
                const uint64_t *prev = F + (size_t)(k - 1) * W;
                sparse_build(prev, sp, W, tid, 64, join);
                for (int r = tid; r < W; r += 64) F[(size_t)k * W + r] = prefix_cell(prev, sp, k, 0, r);
                join();
            }
        } else {
            auto join = [] { bar_named(2, 64); };
            uint64_t *s2 = sp + 2 * levels * W;
            for (int k = m - 2; k >= 1; --k) {
                const uint64_t *next = G + (size_t)(k + 1) * W;
                sparse_build(next, s2, W, tid - 64, 64, join);
                const double *t = rows(k, 0);
                for (int b = tid - 64; b < W; b += 64) {
                    const double *row = t + (size_t)(N - (b + m - k)) * N;   // its first block
                    G[(size_t)k * W + b] = umax64(crossover(next, s2, W, b, [&](int u) {
                                                      ++probes;
                                                      return dkey(row[b - u]);
                                                  }), tk[k + 1]);
                }
                join();
            }
        }
        __syncthreads();
        // ---- the master-free optimum F_m[W-1], over every split
        if (wid == 0) {
            uint64_t x = m == 1 ? dkey(rows(0, 0)[N - 1]) : INF;
            if (m >= 2) {
                const uint64_t *prev = F + (size_t)(m - 2) * W;
                const double *t = rows(m - 1, 0);
                for (int s = lane; s < W; s += 32) {
                    x = umin64(x, umax64(prev[s], dkey(t[(size_t)(s + m - 1) * N + (W - 1 - s)])));
                    ++probes;
                }
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) x = umin64(x, __shfl_xor_sync(0xFFFFFFFFu, x, o));
            if (lane == 0) {
                s_V0 = umax64(x, tk[m - 1]);
                s_V = INF;
                s_mu = 0;
            }
        }
        __syncthreads();
        // ---- masters, four at a time in index order, a warp each, lanes over b
        for (int mu0 = 1; mu0 <= m && s_V > s_V0; mu0 += kLayeredWarps) {   // (uniform: s_V changes below only)
            const int mu = mu0 + wid;
            uint64_t best = INF;
            if (mu <= m) {
                const uint64_t *Fp = F + (size_t)(mu >= 2 ? mu - 2 : 0) * W;
                const uint64_t *Gs = G + (size_t)(mu <= m - 1 ? mu : m - 1) * W;
                const double *h = rows(mu - 1, 1);
                uint64_t lk = 0;
                if (mu >= 2) lk = umax64(lk, tk[mu - 1]);
                if (mu <= m - 1) lk = umax64(lk, tk[mu]);
                if (mu >= 2) sparse_build(Fp, spw, W, lane, 32, [] { __syncwarp(); });
                for (int b = lane; b < (mu <= m - 1 ? W : 1); b += 32) {
                    const uint64_t gb = mu <= m - 1 ? Gs[b] : 0ull;
                    if (gb >= best) continue;                     // cannot lower the minimum
                    uint64_t x;
                    if (mu == 1) {
                        x = dkey(h[W - b - 1]);
                        ++probes;
                    } else {
                        x = crossover(Fp, spw, W, W - 1 - b, [&](int a) {
                            ++probes;
                            return dkey(h[(size_t)(mu - 1 + a) * N + (W - a - b - 1)]);
                        });
                    }
                    best = umin64(best, umax64(x, gb));
                }
#pragma unroll
                for (int o = 16; o; o >>= 1) best = umin64(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
                if (lane == 0) Vmu[mu - 1] = umax64(best, lk);
            }
            __syncthreads();
            if (tid == 0)                                         // the smallest master with the least value
                for (int q = mu0; q < mu0 + kLayeredWarps && q <= m; ++q)
                    if (Vmu[q - 1] < s_V) { s_V = Vmu[q - 1]; s_mu = q; }
            __syncthreads();
        }
        const int mus = s_mu;
        const uint64_t V = s_V;
        __syncthreads();                                          // (s_mu and s_V are the next run's)
        if (V == INF) {                                           // no partition (memory)
            if (tid == 0 && !role) {                              // a prefill result that does not exist
                vo.T[sv] = keyd(kInfKey);
                vo.L[sv] = keyd(kInfKey);
            }
            {                                                         // every thread's probes
                unsigned p = (unsigned)probes;
                p = __reduce_add_sync(0xFFFFFFFFu, p);
                if (lane == 0) atomicAdd(&out.stats[kStProbes], (unsigned long long)p);
            }
            if (tid == 0) atomicAdd(&out.stats[kStDpRuns], 1ull);
            __syncthreads();
            continue;
        }
        // ---- mu*'s prefix columns from column mu* on (the head at mu*)
        for (int k = mus - 1; k <= m - 2; ++k) {
            uint64_t *cur = F + (size_t)k * W;
            const int mf = k == mus - 1;
            if (k == 0) {
                for (int r = tid; r < W; r += blockDim.x) cur[r] = dkey(rows(0, 1)[r]);
            } else {
                const uint64_t *prev = F + (size_t)(k - 1) * W;
                sparse_build(prev, sp, W, tid, blockDim.x, [] { __syncthreads(); });
                for (int r = tid; r < W; r += blockDim.x) cur[r] = prefix_cell(prev, sp, k, mf, r);
            }
            __syncthreads();
        }
        // ---- traceback (warp 0): the smallest split attaining each cell's value
        if (wid == 0) {
            int r = W - 1;
            uint64_t D = V;
            for (int k = m - 1; k >= 1; --k) {
                const uint64_t *prev = F + (size_t)(k - 1) * W;
                const double *t = rows(k, k == mus - 1);
                int split = -1;
                for (int base = 0; base <= r && split < 0; base += 32) {
                    const int s = base + lane;
                    const bool hit = s <= r && umax64(umax64(prev[s], dkey(t[(size_t)(s + k) * N + (r - s)])), tk[k]) == D;
                    const unsigned bal = __ballot_sync(0xFFFFFFFFu, hit);
                    if (bal) split = base + __ffs(bal) - 1;
                }
                if (split < 0) {                                  // cannot happen: D is attained
                    split = 0;
                    if (lane == 0) atomicAdd(&out.stats[kStDeviceErrors], 1ull);
                }
                if (lane == 0) nk[k] = r - split + 1;
                r = split;
                D = prev[r];
            }
            if (lane == 0) nk[0] = r + 1;
            __syncwarp();
            // stage and link times of the partition, lane k holds device k; Lambda in pipeline order
            double lam = 0.0;
            uint64_t tmax = 0;
            int first = 0;                                        // first block of device `base`
            for (int base = 0; base < m; base += 32) {
                const int k = base + lane;
                const int n = k < m ? nk[k] : 0;
                int incl = n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= o) incl += y;
                }
                double l = 0.0, t = 0.0;
                if (k < m) {
                    l = rows(k, k == mus - 1)[(size_t)(first + incl - n) * N + n - 1];
                    if (k) t = keyd(tk[k]);
                    tmax = umax64(tmax, umax64(dkey(l), dkey(t)));
                }
                for (int q = 0; q < 32 && base + q < m; ++q) {
                    const double lq = __shfl_sync(0xFFFFFFFFu, l, q), tq = __shfl_sync(0xFFFFFFFFu, t, q);
                    if (base + q == 0) lam = lq;
                    else { lam = lam + tq; lam = lam + lq; }
                }
                first += __shfl_sync(0xFFFFFFFFu, incl, 31);
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) tmax = umax64(tmax, __shfl_xor_sync(0xFFFFFFFFu, tmax, o));
            if (lane == 0) {
                s_L = lam;
                s_T = keyd(tmax);
                s_done = (!role) || lam <= dm.lam_max;            // 1.0 / lam >= Min_TPS
            }
        }
        __syncthreads();
        if (s_done) {
            int16_t *lay_out = vo.layers + ((size_t)g * dm.V + v) * M + off;
            for (int k = tid; k < m; k += blockDim.x) lay_out[k] = (int16_t)nk[k];
            if (tid == 0) {
                vo.mu[sv] = (int16_t)(mus - 1);
                vo.T[sv] = s_T;
                vo.L[sv] = s_L;
                __threadfence();
                if (role) atomicMax(&vo.best[slot], code);
            }
        } else if (tid == 0 && !role) {
            vo.T[sv] = keyd(kInfKey);
        }
        {                                                         // every thread's probes
            unsigned p = (unsigned)probes;
            p = __reduce_add_sync(0xFFFFFFFFu, p);
            if (lane == 0) atomicAdd(&out.stats[kStProbes], (unsigned long long)p);
        }
        if (tid == 0) {
            atomicAdd(&out.stats[kStDpRuns], 1ull);
            atomicAdd(&out.stats[kStCells], (unsigned long long)(2 * m + (m - mus + 1)) * W + m);
        }
        __syncthreads();
    }
}

// The accepted runs' results become the replicas' outputs, a warp per slot: the
// largest accepted batch of a decode sweep, and the prefill run unless it found
// no partition.
__global__ void __launch_bounds__(128) layered_pick_kernel(Dims dm, DevPop pop, SlotInfo si, VariantOut vo, EvalOut out,
                                                           SplitOut so)
{
    after_previous();
    const int lane = threadIdx.x & 31;
    const long long slot = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (slot >= (long long)dm.P * dm.K) return;
    const uint32_t info = si.info[slot];
    const int M = dm.M, g = (int)(slot / dm.K), off = si.off[slot];
    for (int role = 0; role < 2; ++role) {
        if (!(role ? info & kSlotDecMask : info & kSlotPrefill)) continue;
        const int m = pop.sizes[slot];
        const int best = role ? vo.best[slot] : 0;
        const size_t sv = (size_t)slot * dm.V + (role ? best + 1 : 0);
        const bool ok = role ? best >= 0 : vo.T[sv] < keyd(kInfKey);
        const int16_t *lay = vo.layers + ((size_t)g * dm.V + (role ? best + 1 : 0)) * M + off;
        int16_t *to = dm.role_search ? so.layers + ((size_t)g * 2 + role) * M + off : out.layers + (size_t)g * M + off;
        for (int k = lane; k < m; k += 32) to[k] = ok ? lay[k] : (int16_t)-1;
        if (lane != 0) continue;
        if (dm.role_search) {
            const size_t s2 = (size_t)slot * 2 + role;
            so.code[s2] = (int16_t)(ok ? best : -1);
            if (ok) { so.mu[s2] = vo.mu[sv]; so.T[s2] = vo.T[sv]; so.L[s2] = vo.L[sv]; }
        } else {
            out.master[slot] = ok ? vo.mu[sv] : (int16_t)-1;
            out.bsel[slot] = (int16_t)(ok ? (role ? best + 1 : 0) : -1);
            out.T[slot] = ok ? vo.T[sv] : keyd(kInfKey);
            out.L[slot] = ok ? vo.L[sv] : keyd(kInfKey);
        }
    }
}

// The genome's objective from the role sums (PS, DS; PL, DL the rate-weighted
// latencies sum_P PS_c Lambda_c and sum_D DS_c Lambda_c, all summed in
// ascending replica order).  Objective 0: Eq. 3 bottleneck phase, Eq. 4
// backlog, Eq. 5 waiting time.  Objective 1: the per-request finishing time of
// the FT comparison, a request's prefill pass plus ND decode passes, each
// averaged over its role's replicas in proportion to their rates.  Either way
// the second key is Eq. 3's phase; no prefill or no decode capacity: +inf.
__device__ __forceinline__ void objective(const Dims &dm, double PS, double DS, double PL, double DL, double &w,
                                          double &phase)
{
    w = keyd(kInfKey);
    phase = keyd(kInfKey);
    if (PS != 0.0 && DS != 0.0) {
        const double tp = (double)dm.NP / PS, td = (double)dm.ND / DS;
        phase = tp >= td ? tp : td;                 // Eq. 3
        if (dm.objective == 1) {
            w = PL / PS + (double)dm.ND * (DL / DS);
        } else {
            const double x = phase - dm.t_a;
            const double bn = x > 0.0 ? x : 0.0;    // Eq. 4
            w = bn > 0.0 ? tp + bn : 0.0;           // Eq. 5
        }
    }
}

// A replica's pre-pass verdicts as counts: variants that its memory (n_pre)
// and the latency bound (n_tps) rejected.
__device__ __forceinline__ void slot_tallies(const Dims &dm, uint32_t info, unsigned &n_pre, unsigned &n_tps)
{
    if (info & kSlotDecTested) {
        const unsigned mem = (info >> kSlotMemShift) & kSlotDecMask;
        n_pre += (unsigned)dm.b_max - mem;
        n_tps += mem - (info & kSlotDecMask);
    }
    if ((info & (kSlotPreTested | kSlotPrefill)) == kSlotPreTested) ++n_pre;
}

// A genome's counts, summed over its warp's lanes into `sum` (genomes,
// replicas, served, memory rejections, latency rejections, paper candidates).
constexpr int kTallies = 6;
__device__ __forceinline__ void genome_tallies(unsigned long long *sum, int R, unsigned n_served, unsigned n_pre,
                                               unsigned n_tps, unsigned long long n_paper, int lane)
{
    n_served = __reduce_add_sync(0xFFFFFFFFu, n_served);
    n_pre = __reduce_add_sync(0xFFFFFFFFu, n_pre);
    n_tps = __reduce_add_sync(0xFFFFFFFFu, n_tps);
#pragma unroll
    for (int o = 16; o; o >>= 1) n_paper += __shfl_xor_sync(0xFFFFFFFFu, n_paper, o);
    const unsigned long long x = lane == 0 ? 1ull : lane == 1 ? (unsigned long long)R : lane == 2 ? n_served
                               : lane == 3 ? n_pre : lane == 4 ? n_tps : n_paper;
    if (lane < kTallies && x) atomicAdd(&sum[lane], x);
}

// ... and into the evaluation's counters (threads 0..kTallies-1).
__device__ __forceinline__ void add_tallies(const EvalOut &out, const unsigned long long *sum, int i)
{
    constexpr int to[kTallies] = {kStGenomes, kStReplicas, kStServed, kStPrecheck, kStTpsPruned, kStPaper};
    if (i < kTallies && sum[i]) atomicAdd(&out.stats[to[i]], sum[i]);
}

// Scores the genomes after the DP has written every replica's outputs, eight
// per block, a warp each: the lanes take their replicas' rates (NP / T for
// prefill, b / T for decode) into shared memory, and one warp then sums PS and
// DS of all eight in ascending replica order, a lane per sum (a replica of the
// other role adds 0.0, which changes no sum), and applies Eq. 3 (bottleneck
// phase), Eq. 4 (backlog) and Eq. 5 (waiting time).
//
// Bound by the float64 pipe (two lanes per SM: a warp instruction takes 16
// cycles whatever its lanes) when a warp per genome summed alone: 70 us for
// 16,384 genomes of 32 replicas on average, 32 with eight genomes' sums per
// instruction, the latency sums only where the objective needs them and the
// counters added once per block.
constexpr int kScoreGenomes = 8;

template <bool FT>
__global__ void __launch_bounds__(32 * kScoreGenomes) finalize_score_kernel(Dims dm, DevPop pop, SlotInfo si, EvalOut out)
{
    after_previous();
    constexpr int S = FT ? 4 : 2;                          // PS, DS (and the rate-weighted latencies PL, DL)
    __shared__ double s_x[S][kScoreGenomes][E2_MAX_CLUSTERS + 1];
    __shared__ int s_R[kScoreGenomes];
    __shared__ unsigned long long s_tally[kTallies];
    const int wl = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g0 = blockIdx.x * kScoreGenomes, g = g0 + wl;
    if (threadIdx.x < kTallies) s_tally[threadIdx.x] = 0;
    __syncthreads();
    int R = 0;
    if (g < dm.P) {
        const int K = dm.K, M = dm.M;
        R = pop.nclus[g];
        const uint64_t roles = pop.roles[g];
        const int sz_lo = lane < R ? pop.sizes[(size_t)g * K + lane] : 0;
        const int sz_hi = lane + 32 < R ? pop.sizes[(size_t)g * K + lane + 32] : 0;
        unsigned n_served = 0, n_pre = 0, n_tps = 0;
        unsigned long long n_paper = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = lane + 32 * h;
            if (c >= R) continue;
            const int slot = g * K + c, b = out.bsel[slot], role = (int)((roles >> c) & 1ull);
            const int m = h ? sz_hi : sz_lo;
            slot_tallies(dm, si.info[slot], n_pre, n_tps);
            unsigned long long nrun = role ? (unsigned long long)dm.b_max : 1ull;
            double rate = 0.0, weighted = 0.0;
            if (b >= 0) {
                rate = (role ? (double)b : (double)dm.NP) / out.T[slot];
                if (FT) weighted = rate * out.L[slot];
                if (role) nrun = (unsigned long long)(dm.b_max - b + 1);   // variants b_max .. b
                ++n_served;
            }
            s_x[0][wl][c] = role ? 0.0 : rate;
            s_x[1][wl][c] = role ? rate : 0.0;
            if (FT) {
                s_x[S - 2][wl][c] = role ? 0.0 : weighted;
                s_x[S - 1][wl][c] = role ? weighted : 0.0;
            }
            if (m <= dm.N) n_paper += nrun * paper_candidates(m, dm.N);
        }
        genome_tallies(s_tally, R, n_served, n_pre, n_tps, n_paper, lane);
        const uint64_t h = fingerprint(pop.perm + (size_t)g * M, M, sz_lo, sz_hi, R, roles, lane);
        if (lane == 0) out.hash[g] = h;
    }
    if (lane == 0) s_R[wl] = R;
    __syncthreads();
    if (wl == 1) add_tallies(out, s_tally, lane);
    if (wl != 0) return;
    // lane: sum lane / 8 (PS, DS, PL, DL) of genome lane % 8
    const int q = lane & (kScoreGenomes - 1), which = lane / kScoreGenomes;
    double x = 0.0;
    if (which < S)
        for (int c = 0; c < s_R[q]; ++c) x = x + s_x[which < S ? which : 0][q][c];
    const double DS = __shfl_sync(0xFFFFFFFFu, x, q + kScoreGenomes);
    const double PL = FT ? __shfl_sync(0xFFFFFFFFu, x, q + 2 * kScoreGenomes) : 0.0;
    const double DL = FT ? __shfl_sync(0xFFFFFFFFu, x, q + 3 * kScoreGenomes) : 0.0;
    if (lane >= kScoreGenomes || g0 + q >= dm.P) return;
    double w, phase;
    objective(dm, x, DS, PL, DL, w, phase);
    double *f = out.fit + (size_t)(g0 + q) * 4;
    f[0] = w; f[1] = phase; f[2] = x; f[3] = DS;
}

// Alg. 2's role search, one warp per genome (or a block, below).  The lead
// warp reads every replica's two results (lane l: replicas l and l + 32): the
// prefill run (variant bit b_max, run when the memory allows) and the decode
// sweep's answer (the largest accepted batch).  Every role assignment r (bit
// c = 1: replica c decodes) is scored with the objective (PS and DS summed in
// ascending replica order over the replicas that serve their role); the least
// (objective, phase, r) wins.  Some replicas' roles are fixed in the winner:
// one that serves neither role has its bit clear (it adds nothing either way,
// and the smaller mask wins); under the waiting time, one that cannot decode
// prefills (clearing its bit keeps DS and can only raise PS, since
// round-to-nearest addition is monotone, so w and the phase do not grow and
// the mask shrinks; under the finishing time a slow prefill replica can raise
// the rate-weighted mean latency, so only the first rule applies).  The
// search therefore walks the F other ("free") replicas' roles, free replica j
// being replica fr(j): compact assignments r' over j, in the order of the
// full masks they stand for.  With more than E2_MAX_ROLE_SEARCH free replicas
// the search is not run: the genome keeps its own role bits for them (the
// fixed replicas' bits clear) and is counted in the stats.  The replicas'
// outputs are those of their chosen roles, the chosen roles are written into
// the genome, and the genome is scored.
template <int WPG, bool FT>
__global__ void __launch_bounds__(128) finalize_roles_kernel(Dims dm, DevPop pop, SlotInfo si, SplitOut so,
                                                             EvalOut out)
{
    after_previous();
    constexpr int KC = E2_MAX_CLUSTERS, KF = E2_MAX_ROLE_SEARCH;
    __shared__ double s_ps[4][KC], s_ds[4][KC];
    __shared__ double s_pl[4][KC], s_dl[4][KC];        // rate x Lambda (finishing time)
    __shared__ int s_pv[4][KC], s_dv[4][KC];
    __shared__ int s_off[4][KC + 1], s_code[4][KC];
    __shared__ long long s_qp[4][KC], s_qd[4][KC];
    __shared__ int s_fr[4][KF];                        // full index of free replica j
    __shared__ uint64_t s_free[4];                     // mask of the free replicas
    __shared__ double s_bw[4], s_bph[4];
    __shared__ unsigned long long s_wmin[4];           // the least w a warp of the genome has scored (bits)
    __shared__ uint64_t s_br[4];
    __shared__ unsigned long long s_tally[4][kTallies];    // (a row per warp)
    const int wl = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // WPG warps per genome: 1 (four genomes per block), or 4 (one genome per
    // block, its assignments split over the block's 128 threads)
    const int g = WPG == 1 ? (int)blockIdx.x * 4 + wl : (int)blockIdx.x;
    const int gw = WPG == 1 ? wl : 0;                  // the genome's shared-memory row
    const int id = WPG == 1 ? lane : (int)threadIdx.x; // the thread's place in its genome's search
    const bool lead = WPG == 1 || wl == 0;              // the warp that reads and writes the genome
    if (g >= dm.P) return;
    const int K = dm.K, M = dm.M, bp = dm.b_max;
    const int R = pop.nclus[g];
    const uint64_t roles0 = pop.roles[g];
    // the objective of full assignment r, PS and DS (and, for the finishing
    // time, the rate-weighted latencies) summed in ascending replica order from
    // replica c0 on, the sums over replicas 0..c0-1 given
    constexpr bool ft = FT;                            // objective 1: the finishing time
    auto score_from = [&](uint64_t r, int c0, const double *pre, double &PS, double &DS, double &w,
                          double &phase) {
        PS = pre[0]; DS = pre[1];
        double PL = pre[2], DL = pre[3];
        for (int c = c0; c < R; ++c) {
            if ((r >> c) & 1ull) {
                if (s_dv[gw][c]) { DS = DS + s_ds[gw][c]; if (ft) DL = DL + s_dl[gw][c]; }
            } else if (s_pv[gw][c]) {
                PS = PS + s_ps[gw][c];
                if (ft) PL = PL + s_pl[gw][c];
            }
        }
        objective(dm, PS, DS, PL, DL, w, phase);
    };
    const double zero4[4] = {0.0, 0.0, 0.0, 0.0};
    auto score = [&](uint64_t r, double &PS, double &DS, double &w, double &phase) {
        score_from(r, 0, zero4, PS, DS, w, phase);
    };
    // ---- each replica's two results (lane l: replicas l and l + 32)
    int best[2] = {-1, -1}, pok[2] = {0, 0}, m[2] = {0, 0};
    if (lead) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = lane + 32 * h;
            if (c >= R) continue;
            const int slot = g * K + c;
            const size_t sp = (size_t)slot * 2, sd = sp + 1;      // its prefill run and its decode sweep
            m[h] = pop.sizes[slot];
            pok[h] = so.code[sp] >= 0;
            best[h] = so.code[sd];
            s_off[gw][c] = si.off[slot];
            s_pv[gw][c] = pok[h];
            s_dv[gw][c] = best[h] >= 0;
            s_ps[gw][c] = pok[h] ? (double)dm.NP / so.T[sp] : 0.0;
            s_ds[gw][c] = best[h] >= 0 ? (double)(best[h] + 1) / so.T[sd] : 0.0;
            s_pl[gw][c] = pok[h] ? s_ps[gw][c] * so.L[sp] : 0.0;
            s_dl[gw][c] = best[h] >= 0 ? s_ds[gw][c] * so.L[sd] : 0.0;
        }
        // the free replicas: those that can decode, and under the finishing
        // time also those that can only prefill
        const bool f0 = lane < R && (best[0] >= 0 || (ft && pok[0]));
        const bool f1 = lane + 32 < R && (best[1] >= 0 || (ft && pok[1]));
        const unsigned b0 = __ballot_sync(0xFFFFFFFFu, f0), b1 = __ballot_sync(0xFFFFFFFFu, f1);
        const uint64_t fm = (uint64_t)b0 | ((uint64_t)b1 << 32);
        const uint64_t below = (1ull << lane) - 1ull;
        if (f0) { const int j = __popcll(fm & below); if (j < KF) s_fr[gw][j] = lane; }
        if (f1) { const int j = __popcll(fm & (below << 32 | 0xFFFFFFFFull)); if (j < KF) s_fr[gw][j] = lane + 32; }
        if (lane == 0) { s_off[gw][R] = M; s_free[gw] = fm; }
    }
    if (WPG == 1) __syncwarp();
    else __syncthreads();
    const uint64_t freem = s_free[gw];
    const int F = __popcll(freem);
    // a compact assignment over the free replicas -> its full mask
    auto expand = [&](uint64_t r) -> uint64_t {
        uint64_t full = 0;
        for (int j = 0; j < F; ++j)
            if ((r >> j) & 1ull) full |= 1ull << s_fr[gw][j];
        return full;
    };
    double bw = keyd(kInfKey), bph = keyd(kInfKey);
    uint64_t br = ~0ull;                                // compact
    bool capped = F > KF;
    if (!capped) {
    // ---- the best assignment.  Thread id owns the compact assignments whose
    //      first low = min(F, 5) free replicas' roles (7 with a block per
    //      genome) are the bits of id, and walks the other H = F - low free
    //      replicas' roles in Gray-code order (one role flips per step).  Along
    //      the walk PS and DS are kept as exact fixed-point sums (each rate
    //      rounded to an integer multiple of 2^-s, s per genome so that the
    //      total stays below 2^62), with the counts of replicas serving each
    //      role; the fixed replicas add constant terms.  Two screens skip
    //      assignments that can only lose (waiting time only).  (1) Integer
    //      compares: a w no larger than the best w needs NP/PS <= max(w, T_a)
    //      and ND/DS <= T_a + w (the phase exceeds T_a by at most w, and
    //      w >= NP/PS once it does), i.e. PS and DS above thresholds derived
    //      from the best, with margins for the fixed-point rounding; with a
    //      best w of 0, both must stay within the best phase.  (2) A lower
    //      bound on w and the phase from the float values of the sums, without
    //      a division (relative error below 1e-6, against a 1e-5 margin),
    //      against the best.  The others are scored exactly: PS and DS summed
    //      in float64 in ascending replica order, then the objective, as the
    //      oracle does.  The best key is shared over the warp whenever a lane
    //      improves it, so that few steps of the warp take the exact path.
    //      With at most 8 free replicas every assignment is scored exactly.
    constexpr int kFixed = WPG == 1 ? 5 : 7;            // free replicas whose roles are the bits of id
    const int low = F < kFixed ? F : kFixed, H = F - low;
    // fixed-point scales: totals below 2^62; the screen needs every serving
    // rate to be at least 2^24 units (else every assignment is scored exactly)
    double totp = 0.0, totd = 0.0;
    for (int c = 0; c < R; ++c) { totp = totp + s_ps[gw][c]; totd = totd + s_ds[gw][c]; }
    const int sp_ = totp > 0.0 ? 61 - ilogb(totp) : 0, sd_ = totd > 0.0 ? 61 - ilogb(totd) : 0;
    // the screens bound the waiting time; the finishing time is scored exactly
    bool in_range = !ft && isfinite(totp) && isfinite(totd) && sp_ > -126 + 64 && sp_ < 126 && sd_ > -126 + 64 &&
                    sd_ < 126;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c >= R) continue;
        const long long qp = in_range && s_pv[gw][c] ? __double2ll_rn(ldexp(s_ps[gw][c], sp_)) : 0ll;
        const long long qd = in_range && s_dv[gw][c] ? __double2ll_rn(ldexp(s_ds[gw][c], sd_)) : 0ll;
        if (lead) {
            s_qp[gw][c] = qp;
            s_qd[gw][c] = qd;
        }
        if ((s_pv[gw][c] && qp < (1ll << 24)) || (s_dv[gw][c] && qd < (1ll << 24))) in_range = false;
    }
    in_range = __all_sync(0xFFFFFFFFu, in_range);
    if (lead && lane == 0) s_wmin[gw] = dkey(keyd(kInfKey));
    if (WPG == 1) __syncwarp();
    else __syncthreads();
    if (F <= 8) {                                               // at most 256 assignments: score them all
        for (uint64_t r = id; r < (1ull << F); r += 32 * WPG) {
            double PS, DS, w, ph;
            score(expand(r), PS, DS, w, ph);
            if (w < bw || (w == bw && (ph < bph || (ph == bph && r < br)))) { bw = w; bph = ph; br = r; }
        }
    } else {
        auto fr = [&](int j) { return s_fr[gw][j]; };
        long long P = 0, D = 0;                                 // fixed-point PS and DS
        int np = 0, nd = 0;                                     // replicas serving prefill / decode
        for (int c = 0; c < R; ++c)                             // the fixed replicas prefill
            if (!((freem >> c) & 1ull) && s_pv[gw][c]) { P += s_qp[gw][c]; ++np; }
        for (int j = 0; j < F; ++j) {                           // free replicas above low start as prefill
            const int c = fr(j);
            const bool dec = j < low && ((id >> j) & 1);
            if (dec) { if (s_dv[gw][c]) { D += s_qd[gw][c]; ++nd; } }
            else if (s_pv[gw][c]) { P += s_qp[gw][c]; ++np; }
        }
        // float value of a fixed-point sum (truncated to 24 bits, then scaled)
        auto to_float = [](long long x, int s) -> float {
            const int lz = __clzll(x), sh = lz < 40 ? 40 - lz : 0;
            return __uint2float_rn((unsigned)(x >> sh)) * __int_as_float((127 + sh - s) << 23);
        };
        const float npf = (float)dm.NP, ndf = (float)dm.ND;
        const float ta_up = (float)dm.t_a * (1.0f + 1e-6f);
        bool finite = false, zero = false;                      // the screen's w: finite / own best w of 0
        bool improved = false;                                  // this lane found a better one
        float bw_up = 0.0f, bph_up = 0.0f;                      // the screen's w and phase, rounded up to float
        long long pthr = 0, dthr = 0;                           // screen (1): P, D below these lose
        // the screens compare with we = min(own best w, the least w any warp of
        // the genome has scored); the phase screen only with the own best
        double wsh = keyd(kInfKey);                             // the shared least w last taken
        // start from the genome's own roles over the free replicas: a real
        // assignment, scored exactly
        bool own_fin;                                           // the lane's own best w is finite
        {
            uint64_t r0 = 0;
            for (int j = 0; j < F; ++j) r0 |= ((roles0 >> fr(j)) & 1ull) << j;
            double PS, DS, w, ph;
            score(expand(r0), PS, DS, w, ph);
            bw = w; bph = ph; br = r0;
            own_fin = w < keyd(kInfKey);
            improved = true;
        }
        // one assignment: the screens, then the exact score where they cannot
        // decide.  With a block per genome the roles of free replicas
        // 0..low+1 are fixed per thread and combination: the exact sums over
        // full replicas 0..fr(low+1) are taken once (prefix)
        double pre[4][4] = {{0.0, 0.0, 0.0, 0.0}, {0.0, 0.0, 0.0, 0.0}, {0.0, 0.0, 0.0, 0.0},
                            {0.0, 0.0, 0.0, 0.0}};     // [combination][PS, DS, PL, DL]
        const int c_pre = WPG > 1 ? fr(low + 1) + 1 : 0;       // first replica after the prefix
        auto consider = [&](long long P, long long D, int np, int nd, uint64_t r, int j) {
            if (np == 0 || nd == 0) {                              // PS or DS is 0: w = phase = +inf
                if (!own_fin && r < br) br = r;                    // ties the own best only while it is +inf
                return;
            }
            if (finite && in_range) {
                if (P < pthr || D < dthr) return;
                const float tp = npf * __frcp_rn(to_float(P, sp_)), td = ndf * __frcp_rn(to_float(D, sd_));
                const float ph_lo = fmaxf(tp, td) * (1.0f - 1e-5f);
                const float w_lo = ph_lo > ta_up ? (tp * (1.0f - 1e-5f) + ph_lo) - ta_up : 0.0f;
                if (w_lo > bw_up || (zero && ph_lo > bph_up)) return;
            }
            double PS, DS, w, ph;
            if (WPG > 1) score_from(expand(r), c_pre, pre[j], PS, DS, w, ph);
            else score(expand(r), PS, DS, w, ph);
            if (w < bw || (w == bw && (ph < bph || (ph == bph && r < br)))) {
                bw = w; bph = ph; br = r;
                own_fin = true;                                    // PS, DS > 0: w is finite
                improved = true;
            }
        };
        // the first U = min(H, 2) walked free replicas are taken in all 2^U
        // combinations at every step (independent work for the lane); the
        // Gray code walks the other H - U
        const int U = H < 2 ? H : 2;                            // 2 with a block per genome (F >= 9)
        if (WPG > 1)
            for (int j = 0; j < 4; ++j)
                for (int c = 0; c < c_pre; ++c) {
                    bool dec = false;                               // fixed replicas prefill
                    if ((freem >> c) & 1ull) {
                        const int jj = __popcll(freem & ((1ull << c) - 1ull));   // its free index (< low + 2)
                        dec = jj < low ? ((id >> jj) & 1) : ((j >> (jj - low)) & 1);
                    }
                    if (dec) {
                        if (s_dv[gw][c]) {
                            pre[j][1] = pre[j][1] + s_ds[gw][c];
                            if (ft) pre[j][3] = pre[j][3] + s_dl[gw][c];
                        }
                    } else if (s_pv[gw][c]) {
                        pre[j][0] = pre[j][0] + s_ps[gw][c];
                        if (ft) pre[j][2] = pre[j][2] + s_pl[gw][c];
                    }
                }
        long long dP[2] = {0, 0}, dD[2] = {0, 0};
        int dn[2] = {0, 0}, dm_[2] = {0, 0};
        for (int j = 0; j < U; ++j) {                           // free replica low + j: prefill -> decode
            const int c = fr(low + j);
            dP[j] = -s_qp[gw][c]; dD[j] = s_qd[gw][c];
            dn[j] = -s_pv[gw][c]; dm_[j] = s_dv[gw][c];
        }
        uint64_t gq = 0;                                        // Gray code of the outer step
        const uint64_t nq = 1ull << (H - U);
        for (uint64_t q = 0;; ) {
            const uint64_t rb = (uint64_t)id | (gq << (low + U));
            consider(P, D, np, nd, rb, 0);
            if (U >= 1) consider(P + dP[0], D + dD[0], np + dn[0], nd + dm_[0], rb | (1ull << low), 1);
            if (U >= 2) {
                consider(P + dP[1], D + dD[1], np + dn[1], nd + dm_[1], rb | (2ull << low), 2);
                consider(P + dP[0] + dP[1], D + dD[0] + dD[1], np + dn[0] + dn[1], nd + dm_[0] + dm_[1],
                         rb | (3ull << low), 3);
            }
            // every lane screens against the warp's best: when a lane improved
            // on its own, the best key (w, phase, r) is shared (all 32 lanes
            // run the same number of steps once F >= 5)
            if (H > 0 && __any_sync(0xFFFFFFFFu, improved)) {
#pragma unroll
                for (int o = 16; o; o >>= 1) {
                    const double ow = __shfl_xor_sync(0xFFFFFFFFu, bw, o), op = __shfl_xor_sync(0xFFFFFFFFu, bph, o);
                    const uint64_t orr = __shfl_xor_sync(0xFFFFFFFFu, br, o);
                    if (ow < bw || (ow == bw && (op < bph || (op == bph && orr < br)))) { bw = ow; bph = op; br = orr; }
                }
                improved = true;                                    // every lane's best may have changed
                own_fin = bw < keyd(kInfKey);
                if (lane == 0 && own_fin) atomicMin(&s_wmin[gw], (unsigned long long)dkey(bw));
            }
            {                                                       // another warp's better w
                const double ws = keyd(*reinterpret_cast<volatile unsigned long long *>(&s_wmin[gw]));
                if (ws < wsh) { wsh = ws; improved = true; }
            }
            if (improved) {                                         // the float copies of the screen's state
                improved = false;
                const double we = bw < wsh ? bw : wsh;
                if (we < keyd(kInfKey)) {
                    finite = true;
                    zero = bw == 0.0;
                    bw_up = (float)we;
                    if ((double)bw_up < we) bw_up = nextafterf(bw_up, HUGE_VALF);
                    bph_up = (float)bph;
                    if ((double)bph_up < bph) bph_up = nextafterf(bph_up, HUGE_VALF);
                    if (in_range) {
                        // PS >= NP / max(w, T_a) and DS >= ND / (T_a + w) for a w no larger than
                        // we (with an own best w of 0: both phases within its phase), less
                        // 1e-9 relative and R units
                        const double ptp = zero ? bph : (we > dm.t_a ? we : dm.t_a);
                        const double ptd = zero ? bph : dm.t_a + we;
                        const double pmin = ldexp((double)dm.NP / ptp, sp_) * (1.0 - 1e-9);
                        const double dmin = ldexp((double)dm.ND / ptd, sd_) * (1.0 - 1e-9);
                        pthr = pmin < 4e18 ? (long long)pmin - R : (long long)4e18;
                        dthr = dmin < 4e18 ? (long long)dmin - R : (long long)4e18;
                    }
                }
            }
            if (++q == nq) break;
            // the next Gray code flips bit t: free replica low + U + t changes role
            const int t = __ffsll((long long)q) - 1, c = fr(low + U + t);
            gq ^= 1ull << t;
            const long long qp = s_qp[gw][c], qd = s_qd[gw][c];     // 0 where the role is not served
            const int pv = s_pv[gw][c], dv = s_dv[gw][c];
            if ((gq >> t) & 1ull) { P -= qp; D += qd; np -= pv; nd += dv; }   // prefill -> decode
            else { P += qp; D -= qd; np += pv; nd -= dv; }                     // decode -> prefill
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const double ow = __shfl_xor_sync(0xFFFFFFFFu, bw, o), op = __shfl_xor_sync(0xFFFFFFFFu, bph, o);
        const uint64_t orr = __shfl_xor_sync(0xFFFFFFFFu, br, o);
        if (ow < bw || (ow == bw && (op < bph || (op == bph && orr < br)))) { bw = ow; bph = op; br = orr; }
    }
    if (WPG > 1) {                                      // the best of the genome's warps
        if (lane == 0) { s_bw[wl] = bw; s_bph[wl] = bph; s_br[wl] = br; }
        __syncthreads();
        if (wl != 0) return;
        for (int o = 1; o < WPG; ++o) {
            const double ow = s_bw[o], op = s_bph[o];
            const uint64_t orr = s_br[o];
            if (ow < bw || (ow == bw && (op < bph || (op == bph && orr < br)))) { bw = ow; bph = op; br = orr; }
        }
    }
    }  // !capped
    else if (!lead) {
        return;
    }
    // ---- outputs of the chosen roles (the genome's first warp)
    const uint64_t brf = capped ? (roles0 & freem) : expand(br);
    unsigned n_served = 0, n_pre = 0, n_tps = 0;
    unsigned long long n_paper = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c >= R) continue;
        const int slot = g * K + c;
        const int role = (int)((brf >> c) & 1ull);
        const size_t sv = (size_t)slot * 2 + role;
        const int code = role ? best[h] : (pok[h] ? 0 : -1);
        s_code[gw][c] = code < 0 ? -1 : role;
        if (code < 0) {
            out.master[slot] = -1; out.bsel[slot] = -1;
            out.T[slot] = keyd(kInfKey); out.L[slot] = keyd(kInfKey);
        } else {
            const double T = so.T[sv], L = so.L[sv];
            out.master[slot] = so.mu[sv];
            out.bsel[slot] = (int16_t)(role ? code + 1 : 0);
            out.T[slot] = T;
            out.L[slot] = L;
            ++n_served;
        }
        slot_tallies(dm, si.info[slot], n_pre, n_tps);
        const unsigned long long ndec = (unsigned long long)(best[h] >= 0 ? bp - best[h] : bp);
        if (m[h] <= dm.N) n_paper += (1 + ndec) * paper_candidates(m[h], dm.N);
    }
    __syncwarp();
    const int16_t *split = so.layers + (size_t)g * 2 * M;
    for (int i = lane; i < M; i += 32) {
        int lo = 0, hi = R - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_off[gw][mid] <= i) lo = mid;
            else hi = mid - 1;
        }
        const int code = s_code[gw][lo];
        out.layers[(size_t)g * M + i] = code >= 0 ? split[(size_t)code * M + i] : (int16_t)-1;
    }
    if (lane < kTallies) s_tally[wl][lane] = 0;
    __syncwarp();
    genome_tallies(s_tally[wl], R, n_served, n_pre, n_tps, n_paper, lane);
    __syncwarp();
    add_tallies(out, s_tally[wl], lane);
    const uint64_t h = fingerprint(pop.perm + (size_t)g * M, M, m[0], m[1], R, brf, lane);
    if (lane != 0) return;
    if (capped) atomicAdd(&out.stats[kStRoleCapped], 1ull);
    double PS, DS, w, phase;
    score(brf, PS, DS, w, phase);
    double *f = out.fit + (size_t)g * 4;
    f[0] = w; f[1] = phase; f[2] = PS; f[3] = DS;
    pop.roles[g] = brf;
    out.hash[g] = h;
}

// The adapted-SplitWise rule of the paper's comparison (Sec. 4.2, "Baseline
// chosen"), one warp per genome; lane l holds replicas l and l + 32.  Every
// replica was evaluated in both roles (as for the role search): its prefill
// run (variant bit b_max, present when the memory allows) and its decode
// sweep's answer (the largest accepted batch).  A replica's strength is its
// prefill throughput NP/T (-1 when it cannot prefill); the n_P strongest
// replicas prefill (ties to the lower index), the rest decode, with
// n_P = R NP / (NP + ND) rounded half up and clamped to [1, R-1] (R = 1: 1).
// The replicas' outputs are those of their roles, the roles are written into
// the genome, and the genome is scored.
__global__ void __launch_bounds__(128) finalize_splitwise_kernel(Dims dm, DevPop pop, SlotInfo si, SplitOut so,
                                                                 EvalOut out)
{
    after_previous();
    __shared__ int s_off[4][E2_MAX_CLUSTERS + 1];     // replica start in the ordering
    __shared__ int s_code[4][E2_MAX_CLUSTERS];        // the role whose result is taken, -1 none
    __shared__ unsigned long long s_tally[4][kTallies];   // (a row per warp)
    const int wl = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.x * 4 + wl;
    if (g >= dm.P) return;
    const int K = dm.K, M = dm.M, bp = dm.b_max;
    const int R = pop.nclus[g];
    double strength[2];
    int pok[2], best[2], m[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        strength[h] = -1.0;
        pok[h] = 0;
        best[h] = -1;
        m[h] = 0;
        if (c < R) {
            const int slot = g * K + c;
            const size_t sp = (size_t)slot * 2;
            m[h] = pop.sizes[slot];
            pok[h] = so.code[sp] >= 0;
            best[h] = so.code[sp + 1];
            s_off[wl][c] = si.off[slot];
            if (pok[h]) strength[h] = (double)dm.NP / so.T[sp];
        }
    }
    if (lane == 0) s_off[wl][R] = M;
    // prefill count from the token ratio, in integers
    int nP = R;
    if (R > 1) {
        const uint64_t den = dm.NP + dm.ND;
        nP = (int)((2ull * (uint64_t)R * dm.NP + den) / (2ull * den));
        nP = nP < 1 ? 1 : (nP > R - 1 ? R - 1 : nP);
    }
    // rank of each replica by strength (stronger first, ties to the lower index)
    int rank[2] = {0, 0};
    for (int o = 0; o < R; ++o) {
        const double so_ = __shfl_sync(0xFFFFFFFFu, o < 32 ? strength[0] : strength[1], o & 31);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = lane + 32 * h;
            if (c < R && o != c && (so_ > strength[h] || (so_ == strength[h] && o < c))) ++rank[h];
        }
    }
    const unsigned dec_lo = __ballot_sync(0xFFFFFFFFu, lane < R && rank[0] >= nP);
    const unsigned dec_hi = __ballot_sync(0xFFFFFFFFu, lane + 32 < R && rank[1] >= nP);
    const uint64_t roles = (uint64_t)dec_lo | ((uint64_t)dec_hi << 32);
    // outputs of the chosen roles
    double rate[2] = {0.0, 0.0}, lat[2] = {0.0, 0.0};
    int kind[2] = {-1, -1};
    unsigned n_served = 0, n_pre = 0, n_tps = 0;
    unsigned long long n_paper = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c >= R) continue;
        const int slot = g * K + c;
        const int role = (int)((roles >> c) & 1ull);
        const size_t sv = (size_t)slot * 2 + role;
        const int code = role ? best[h] : (pok[h] ? 0 : -1);
        s_code[wl][c] = code < 0 ? -1 : role;
        if (code < 0) {
            out.master[slot] = -1; out.bsel[slot] = -1;
            out.T[slot] = keyd(kInfKey); out.L[slot] = keyd(kInfKey);
        } else {
            const double T = so.T[sv], L = so.L[sv];
            out.master[slot] = so.mu[sv];
            out.bsel[slot] = (int16_t)(role ? code + 1 : 0);
            out.T[slot] = T;
            out.L[slot] = L;
            lat[h] = L;
            kind[h] = role;
            rate[h] = role ? (double)(code + 1) / T : (double)dm.NP / T;
            ++n_served;
        }
        slot_tallies(dm, si.info[slot], n_pre, n_tps);
        const unsigned long long ndec = (unsigned long long)(best[h] >= 0 ? bp - best[h] : bp);
        if (m[h] <= dm.N) n_paper += (1 + ndec) * paper_candidates(m[h], dm.N);
    }
    __syncwarp();
    const int16_t *split = so.layers + (size_t)g * 2 * M;
    for (int i = lane; i < M; i += 32) {
        int lo = 0, hi = R - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_off[wl][mid] <= i) lo = mid;
            else hi = mid - 1;
        }
        const int code = s_code[wl][lo];
        out.layers[(size_t)g * M + i] = code >= 0 ? split[(size_t)code * M + i] : (int16_t)-1;
    }
    if (lane < kTallies) s_tally[wl][lane] = 0;
    __syncwarp();
    genome_tallies(s_tally[wl], R, n_served, n_pre, n_tps, n_paper, lane);
    __syncwarp();
    add_tallies(out, s_tally[wl], lane);
    double PS = 0.0, DS = 0.0, PL = 0.0, DL = 0.0;
    for (int c = 0; c < R; ++c) {
        const int h = c >> 5;
        const double x = __shfl_sync(0xFFFFFFFFu, h ? rate[1] : rate[0], c & 31);
        const double l = __shfl_sync(0xFFFFFFFFu, h ? lat[1] : lat[0], c & 31);
        const int k = __shfl_sync(0xFFFFFFFFu, h ? kind[1] : kind[0], c & 31);
        if (k == 0) { PS = PS + x; PL = PL + x * l; }
        else if (k == 1) { DS = DS + x; DL = DL + x * l; }
    }
    const uint64_t h = fingerprint(pop.perm + (size_t)g * M, M, m[0], m[1], R, roles, lane);
    if (lane != 0) return;
    double w, phase;
    objective(dm, PS, DS, PL, DL, w, phase);
    double *f = out.fit + (size_t)g * 4;
    f[0] = w; f[1] = phase; f[2] = PS; f[3] = DS;
    pop.roles[g] = roles;
    out.hash[g] = h;
}

// The G--C split of the plans (Sec. 4.3) under GPU-CPU offload, one warp per
// genome: of the n blocks at ordering position i, the ones in the device's own
// memory, min(n, capg), for the variant its replica serves (bsel: 0 prefill,
// b decode) and whether the device is the replica's master; -1 where the
// replica cannot serve.  Runs after the replicas' outputs are final.
__global__ void __launch_bounds__(128) gc_split_kernel(Dims dm, DevPop pop, const int32_t *capg, EvalOut out)
{
    after_previous();
    __shared__ int s_off[4][E2_MAX_CLUSTERS + 1];
    const int wl = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.x * 4 + wl;
    if (g >= dm.P) return;
    const int K = dm.K, M = dm.M;
    const int R = pop.nclus[g];
    // replica offsets: an exclusive scan of the sizes (lane l: replicas l and l + 32)
    const int s_lo = lane < R ? pop.sizes[(size_t)g * K + lane] : 0;
    const int s_hi = lane + 32 < R ? pop.sizes[(size_t)g * K + lane + 32] : 0;
    int in_lo = s_lo, in_hi = s_hi;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xFFFFFFFFu, in_lo, o), b = __shfl_up_sync(0xFFFFFFFFu, in_hi, o);
        if (lane >= o) { in_lo += a; in_hi += b; }
    }
    const int total_lo = __shfl_sync(0xFFFFFFFFu, in_lo, 31);
    if (lane < R) s_off[wl][lane] = in_lo - s_lo;
    if (lane + 32 < R) s_off[wl][lane + 32] = total_lo + in_hi - s_hi;
    if (lane == 0) s_off[wl][R] = M;
    __syncwarp();
    for (int i = lane; i < M; i += 32) {
        int lo = 0, hi = R - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_off[wl][mid] <= i) lo = mid;
            else hi = mid - 1;
        }
        const size_t slot = (size_t)g * K + lo;
        const int n = out.layers[(size_t)g * M + i];
        int16_t gb = -1;
        if (n >= 0) {
            const int v = out.bsel[slot];
            const int mf = (i - s_off[wl][lo]) == out.master[slot];
            const int d = pop.perm[(size_t)g * M + i];
            const int c = capg[((size_t)v * M + d) * 2 + mf];
            gb = (int16_t)(n < c ? n : c);
        }
        out.gpu_layers[(size_t)g * M + i] = gb;
    }
}

// Persistent grids of the DP.  Replicas of up to 32 devices (a device per
// lane) and larger ones (several per lane, more registers) form two launches
// where both sizes can occur.  (A second launch for the replicas of more than 8
// devices on smaller fleets with 32,768 slots or more was slower at every size
// measured: 8,192 genomes of 32 devices 172 us a generation against 167, 16,384
// 280 against 262, 65,536 891 against 870.)
cudaError_t configure_eval(e2_ctx *c)
{
    cudaError_t e = cudaSuccess;
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    if (e != cudaSuccess) return e;
    if (sms < 1) sms = 1;
    const int mmax = c->dm.M < c->dm.N ? c->dm.M : c->dm.N;
    c->dm.dp_mmax = mmax;
    c->dm.dp_split = 0;
    c->dp_grid1 = 0;
    c->dp_smem1 = 0;
    if (c->dm.layered) {                         // the per-layer DP: one launch, one class
        // the limit on its shared memory belongs to the kernel on this device, not to a
        // context: every context sets the same one, all that a CTA may have beside the
        // kernel's own arrays, so none lowers what another one launches with
        const void *lk = reinterpret_cast<const void *>(dp_layered_kernel);
        cudaFuncAttributes own;
        int optin = 0;
        if ((e = cudaFuncGetAttributes(&own, lk)) != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(lk, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)own.sharedSizeBytes);
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lk, 32 * kLayeredWarps, c->dp_smem);
        if (e != cudaSuccess) return e;
        c->dp_grid = (per_sm > 0 ? per_sm : 1) * sms;
        return cudaSuccess;
    }
    const bool off = c->dm.offload != 0;
    if (mmax > 32) c->dm.dp_split = 32;
    const int m0 = c->dm.dp_split ? c->dm.dp_split : mmax;   // class 0's largest replica
    int per_sm = 0;
    e = dp_order_occupancy(m0, 0, off, &per_sm);
    if (e != cudaSuccess) return e;
    c->dp_grid = (per_sm > 0 ? per_sm : 1) * sms;
    c->dp_smem = dp_order_smem(m0, 0);
    if (c->dm.dp_split) {
        e = dp_order_occupancy(mmax, 1, off, &per_sm);
        if (e != cudaSuccess) return e;
        c->dp_grid1 = (per_sm > 0 ? per_sm : 1) * sms;
        c->dp_smem1 = dp_order_smem(mmax, 1);
    }
    return cudaSuccess;
}

cudaError_t launch_eval(const e2_ctx *c, const DevPop &p)
{
    Tables tb{c->rate, c->bw, c->mem, c->rate_cpu, c->bw_cpu, c->mem_cpu, c->prof, c->leaf, c->tau,
              c->capg, c->leaf_rank, c->lcost, c->drec, c->fxs, c->prec, c->prech, c->capv,
              c->ibw, c->fpr};
    EvalOut out{c->fit, c->layers, c->master, c->bsel, c->T, c->L, c->hash, c->stats, c->gpu_layers};
    SlotInfo si{c->slot_off, c->slot_info};
    WorkList wl{c->items, c->list_ctrl};
    SplitOut so{c->split_T, c->split_L, c->split_mu, c->split_code, c->split_layers};
    VariantOut vo{c->var_T, c->var_L, c->var_mu, c->var_layers, c->var_best};
    const long long slots = (long long)c->dm.P * c->dm.K;
    cudaError_t e = cudaSuccess;
    slot_kernel<<<(unsigned)c->dm.P, 32 * (c->dm.K < kPreWarps ? c->dm.K : kPreWarps), 2 * (size_t)c->dm.M, c->stream>>>(
        c->dm, tb, p, si, out, so, vo);
    // (1,024 slots per block of the count and the scatter, more on large populations:
    // 8.7 us a generation for both at 32,768 slots, 14 with 4,096 per block)
    const long long nb = (slots + 1023) / 1024;
    const unsigned lb = (unsigned)(nb < kListBlocks ? nb : kListBlocks);
    if ((e = launch_kernel(bins_kernel, lb, 256, 0, c->stream, true, c->dm, si, c->list_hist, c->stats)) != cudaSuccess) return e;
    if ((e = launch_kernel(order_scatter_kernel, lb, 256, 0, c->stream, true, c->dm, si, wl, c->list_hist)) != cudaSuccess)
        return e;
    // while a launch sequence is being recorded, the timing events become
    // event-record nodes of the graph (an ordinary record would only mark a
    // dependency)
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (c->ev_dp_start && (e = cudaStreamIsCapturing(c->stream, &cs)) != cudaSuccess) return e;
    const unsigned rec = cs == cudaStreamCaptureStatusActive ? cudaEventRecordExternal : cudaEventRecordDefault;
    if (c->ev_dp_start && (e = cudaEventRecordWithFlags(c->ev_dp_start, c->stream, rec)) != cudaSuccess) return e;
    if (c->dm.layered) {
        e = launch_kernel(dp_layered_kernel, (unsigned)c->dp_grid, 32 * kLayeredWarps, c->dp_smem, c->stream, !c->ev_dp_start,
                          c->dm, tb, p, out, wl, si, vo);
        if (e == cudaSuccess)
            e = launch_kernel(layered_pick_kernel, (unsigned)((slots + 3) / 4), 128, 0, c->stream, true, c->dm, p, si, vo, out, so);
        if (e != cudaSuccess) return e;
        ++c->launches;
    } else {
        // the larger replicas run beside the others on the side stream (few runs,
        // each a longer chain)
        if (c->dp_grid1 > 0) {
            if ((e = cudaEventRecord(c->ev_fork, c->stream)) != cudaSuccess) return e;
            if ((e = cudaStreamWaitEvent(c->side, c->ev_fork, 0)) != cudaSuccess) return e;
            e = dp_order_launch(c->dp_grid1, c->dm.dp_mmax, 1, c->side, c->dm, tb, p, out, wl, c->slot_off, so, false);
            if (e != cudaSuccess) return e;
            if ((e = cudaEventRecord(c->ev_join, c->side)) != cudaSuccess) return e;
        }
        // (an early class 0 would fill the SMs before class 1, which has the longer chains:
        // 1,057 us instead of 978 for four generations of 4,096 genomes of 128 devices)
        e = dp_order_launch(c->dp_grid, c->dm.dp_split ? c->dm.dp_split : c->dm.dp_mmax, 0, c->stream, c->dm, tb, p, out,
                            wl, c->slot_off, so, !c->ev_dp_start && c->dp_grid1 == 0);
        if (e == cudaSuccess && c->dp_grid1 > 0) e = cudaStreamWaitEvent(c->stream, c->ev_join, 0);
        if (e != cudaSuccess) return e;
    }
    if (c->ev_dp_stop && (e = cudaEventRecordWithFlags(c->ev_dp_stop, c->stream, rec)) != cudaSuccess) return e;
    const unsigned fb = (unsigned)(((size_t)c->dm.P * 32 + 127) / 128), fg = (unsigned)c->dm.P;
    const bool early = !c->ev_dp_stop && (c->dm.layered || c->dp_grid1 == 0);   // (a kernel comes right before)
    const bool ft = c->dm.objective == 1;
    if (c->dm.role_search == 2)
        e = launch_kernel(finalize_splitwise_kernel, fb, 128, 0, c->stream, early, c->dm, p, si, so, out);
    else if (c->dm.role_search && c->dm.K >= 12)      // up to 2^K_max assignments: a block per genome
        e = launch_kernel(ft ? finalize_roles_kernel<4, true> : finalize_roles_kernel<4, false>, fg, 128, 0, c->stream, early,
                          c->dm, p, si, so, out);
    else if (c->dm.role_search)
        e = launch_kernel(ft ? finalize_roles_kernel<1, true> : finalize_roles_kernel<1, false>, fb, 128, 0, c->stream, early,
                          c->dm, p, si, so, out);
    else
        e = launch_kernel(ft ? finalize_score_kernel<true> : finalize_score_kernel<false>,
                          (unsigned)((c->dm.P + kScoreGenomes - 1) / kScoreGenomes), 32 * kScoreGenomes, 0, c->stream, early,
                          c->dm, p, si, out);
    if (e != cudaSuccess) return e;
    c->launches += c->dp_grid1 > 0 ? 6 : 5;
    if (c->dm.offload) {
        if ((e = launch_kernel(gc_split_kernel, fb, 128, 0, c->stream, true, c->dm, p, c->capg, out)) != cudaSuccess) return e;
        ++c->launches;
    }
    return cudaGetLastError();
}

}  // namespace e2
