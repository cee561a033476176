// elites.cuh -- the elites' device code, shared by the generation step (ga.cu)
// and the allocation-free selection (elites_noalloc.cu): the duplicate test
// through a fingerprint table, and the selection of the Q first distinct
// genomes in the order (w, phase, index).  w and phase are compared as their
// bit patterns (the order of the values for the non-negative and +inf results
// of an evaluation, and a total order for anything else).
#pragma once
#include "e2ga_internal.cuh"

namespace e2 {

namespace {

// 64-bit fingerprint of a genome (ordering, replica sizes and count, roles) for
// the duplicate test, by a warp: the lanes mix interleaved slices, then fold as
// a tree.  Valid in lane 0.  (Orderings are read two positions at a time where
// the row starts on 4 bytes; which is the same for every genome of a call.)
__device__ __forceinline__ uint64_t fingerprint(const uint16_t *perm, int M, int sz_lo, int sz_hi, int R, uint64_t roles,
                                                int lane, uint64_t seed = 0x9E3779B97F4A7C15ull)
{
    auto mix = [](uint64_t h, uint64_t x) { h = (h ^ x) * 0xBF58476D1CE4E5B9ull; return h ^ (h >> 31); };
    uint64_t h = seed ^ (uint64_t)lane;
    if ((M & 1) == 0 && (reinterpret_cast<uintptr_t>(perm) & 3) == 0) {
        const uint32_t *p2 = reinterpret_cast<const uint32_t *>(perm);
        for (int i = lane; i < M / 2; i += 32) h = mix(h, p2[i]);
    } else {
        for (int i = lane; i < M; i += 32) h = mix(h, perm[i]);
    }
    if (lane < R) h = mix(h, (uint64_t)sz_lo << 16);
    if (lane + 32 < R) h = mix(h, (uint64_t)sz_hi << 16);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const uint64_t other = __shfl_down_sync(0xFFFFFFFFu, h, o);
        if (lane < o) h = mix(h, other);
    }
    return mix(mix(h, (uint64_t)R << 40), roles);
}

// The fingerprint table: open addressing with linear probing over a power of
// two of at least 2 P slots (so a free one is always found).  A slot holds the
// high half of a fingerprint, which never changes once the slot is taken, over
// the smallest index of the genomes that came to it with that half, so a probe
// is one read.
constexpr unsigned long long kFreeSlot = 0x7F7F7F7F7F7F7F7Full;   // (bytes 0x7F)

__device__ __forceinline__ unsigned table_start(uint64_t h, unsigned mask) { return (unsigned)(h ^ (h >> 32)) & mask; }
// (a half equal to a free slot's is taken for its neighbour's)
__device__ __forceinline__ uint32_t table_tag(uint64_t h)
{
    const uint32_t t = (uint32_t)(h >> 32);
    return t == 0x7F7F7F7Fu ? t + 1 : t;
}

__device__ __forceinline__ void table_insert(unsigned long long *tab, unsigned mask, uint64_t h, int g)
{
    const uint32_t tag = table_tag(h);
    const unsigned long long mine = (unsigned long long)tag << 32 | (unsigned)g;
    unsigned s = table_start(h, mask);
    for (unsigned i = 0; i <= mask; ++i, s = (s + 1) & mask) {
        unsigned long long o = *(volatile unsigned long long *)&tab[s];
        if (o == kFreeSlot) {
            o = atomicCAS(&tab[s], kFreeSlot, mine);
            if (o == kFreeSlot) return;
        }
        if ((uint32_t)(o >> 32) == tag) {
            atomicMin(&tab[s], mine);
            return;
        }
    }
}

// The smallest index in g's slot: no larger than that of any genome with g's
// fingerprint (they probe alike, so they share a slot).
__device__ __forceinline__ int table_first(const unsigned long long *tab, unsigned mask, uint64_t h, int g)
{
    const uint32_t tag = table_tag(h);
    unsigned s = table_start(h, mask);
    for (unsigned i = 0; i <= mask; ++i, s = (s + 1) & mask) {
        const unsigned long long o = tab[s];
        if (o == kFreeSlot) break;
        if ((uint32_t)(o >> 32) == tag) return (int)(uint32_t)o;
    }
    return g;
}

// Whether genomes a and b are equal (ordering, sizes, replica count, roles); a warp.
__device__ __forceinline__ bool same_genome(const DevPop &p, int a, int b, int M, int K, int lane)
{
    bool diff = p.nclus[a] != p.nclus[b] || p.roles[a] != p.roles[b];
    for (int i = lane; i < M && !diff; i += 32) diff = p.perm[(size_t)a * M + i] != p.perm[(size_t)b * M + i];
    for (int i = lane; i < K && !diff; i += 32) diff = p.sizes[(size_t)a * K + i] != p.sizes[(size_t)b * K + i];
    return __ballot_sync(0xFFFFFFFFu, diff) == 0u;
}

// Whether genome g equals a lower-indexed one; a warp.  It is compared in full
// with the lowest-indexed genome of its slot; if the two differ -- fingerprints
// with equal halves, a 64-bit collision, or genomes that differ only in sizes
// or role bits past their replica count, which the fingerprint does not cover
// -- with every later one below g that has its fingerprint.  With fk (fitness rows of four
// words) a duplicate has the same w and phase too.
__device__ __forceinline__ bool is_duplicate(const DevPop &p, const unsigned long long *tab, unsigned mask, const uint64_t *hash, int g,
                                             int M, int K, int lane, const uint64_t *fk = nullptr)
{
    auto same = [&](int o) {
        if (fk && (fk[(size_t)o * 4] != fk[(size_t)g * 4] || fk[(size_t)o * 4 + 1] != fk[(size_t)g * 4 + 1])) return false;
        return same_genome(p, o, g, M, K, lane);
    };
    const uint64_t h = hash[g];
    int first = g;
    if (lane == 0) first = table_first(tab, mask, h, g);
    first = __shfl_sync(0xFFFFFFFFu, first, 0);
    if (first >= g) return false;
    bool d = same(first);
    for (int base = first + 1; base < g && !d; base += 32) {
        const int o = base + lane;
        unsigned b = __ballot_sync(0xFFFFFFFFu, o < g && hash[o] == h);
        while (b && !d) {
            const int oo = base + __ffs(b) - 1;
            b &= b - 1;
            d = same(oo);
        }
    }
    return d;
}

// Duplicate flags of small populations, by every block of a grid: each fills a
// table of its own in shared memory (mask + 1 slots) and looks up its share of
// the genomes, which saves a fill in global memory, a launch and its atomics.
constexpr int kDupThreads = 512;

template <typename Dup>
__device__ __forceinline__ void flag_duplicates(unsigned long long *tab, unsigned mask, const DevPop &p, const uint64_t *hash,
                                                Dup *dup, int P, int M, int K, const uint64_t *fk = nullptr)
{
    const int lane = threadIdx.x & 31;
    for (unsigned s = threadIdx.x; s <= mask; s += kDupThreads) tab[s] = kFreeSlot;
    __syncthreads();
    for (int g = threadIdx.x; g < P; g += kDupThreads) table_insert(tab, mask, hash[g], g);
    __syncthreads();
    for (int g = blockIdx.x * (kDupThreads / 32) + (threadIdx.x >> 5); g < P; g += gridDim.x * (kDupThreads / 32)) {
        const bool d = is_duplicate(p, tab, mask, hash, g, M, K, lane, fk);
        if (lane == 0) dup[g] = d;
    }
}

// A list that holds the Q first distinct genomes in the order (w, phase,
// index), made by one CTA without ranking every genome.  Each thread takes the
// least key of its share of the genomes; the Q-th least of these minima has at
// least Q keys at or before it, so the genomes at or before it are the list:
// little more than Q of them, since a share of 8 to 32 keys seldom holds two of
// the first 1/32.  (Where there are fewer minima than Q, or Q is most of them,
// the selection takes all keys.)  The Q-th least comes from a radix select over
// the bit patterns of w, 8 bits a pass from the highest bit in which any two
// differ, which stops as soon as a bucket is needed whole; where more keys
// share that w than are needed, from a second select over their phases; and
// where more share both, the first by index are taken.
//
// Genomes strictly before the threshold go to cand[0, ctl[1]) in any order
// (rank_listed orders them), and those tied at it follow in index order,
// ctl[3] of them, as far as Q needs them.  With fewer than Q distinct genomes
// (duplicates then fill the elite slots) ctl[2] is 0 and the full ranking runs
// instead.
//
// Bound by the passes' latency on one SM: two sweeps over the keys, and three
// barriers and one shared-memory atomic per thread for each of three to eight
// passes: 12 us for 8,192 genomes most of which wait 0 s (a select over every
// key took 24, and listed thousands of ties for the ranking: 88 us, now 9).
constexpr int kSelThreads = 1024;

template <typename Dup>
__global__ void __launch_bounds__(kSelThreads) elite_select_kernel(int P, int Q, const double *fit, const Dup *dup,
                                                                   unsigned long long *ctl, int32_t *cand)
{
    after_previous();
    __shared__ unsigned hist[256];
    __shared__ unsigned long long s_prefix, s_and, s_or;
    __shared__ unsigned s_need, s_count, s_minima, s_n, s_run, s_wsum[kSelThreads / 32];
    __shared__ int s_shift;
    struct Key { uint64_t x, y; };                        // w, phase
    auto key_of = [&](int g) {                            // (the caller's rows may start on any 8 bytes)
        const uint64_t *fk = reinterpret_cast<const uint64_t *>(fit) + (size_t)g * 4;
        return Key{fk[0], fk[1]};
    };
    const int tid = threadIdx.x, lane = tid & 31, wl = tid >> 5;
    constexpr uint64_t kAll = ~0ull;
    if (tid == 0) { s_count = 0; s_minima = 0; }
    __syncthreads();
    // this thread's share, genomes tid, tid + 1024, ...: its distinct ones and their least key
    unsigned nd = 0;
    uint64_t mw = kAll, mp = kAll;
#pragma unroll 8
    for (int g = tid; g < P; g += kSelThreads) {
        const Key k = key_of(g);
        if (dup[g] == 0) {
            if (k.x < mw || (k.x == mw && k.y < mp) || nd == 0) { mw = k.x; mp = k.y; }
            ++nd;
        }
    }
    {
        const unsigned all = __reduce_add_sync(0xFFFFFFFFu, nd), some = __popc(__ballot_sync(0xFFFFFFFFu, nd != 0));
        if (lane == 0) { atomicAdd(&s_count, all); atomicAdd(&s_minima, some); }
    }
    __syncthreads();
    const unsigned distinct = s_count, need0 = (unsigned)Q;
    if (Q <= 0 || distinct < need0) {                     // (uniform)
        if (tid < 4) ctl[tid] = 0;
        return;
    }
    const bool minima = s_minima >= need0 && 4u * need0 <= 3u * kSelThreads;
    // f(w, phase) for every key the threshold is chosen among
    auto each = [&](auto f) {
        if (minima) {
            if (nd) f(mw, mp);
        } else {
#pragma unroll 4
            for (int g = tid; g < P; g += kSelThreads) {
                const Key k = key_of(g);
                if (dup[g] == 0) f(k.x, k.y);
            }
        }
    };
    // The need-th smallest of the keys x that key(w, phase, x) accepts: s_prefix
    // becomes the largest key of the last bucket examined, s_need how many of
    // the keys in that bucket are needed and s_n how many there are.
    auto select = [&](unsigned need, auto key) {
        if (tid == 0) { s_and = kAll; s_or = 0; s_need = need; }
        __syncthreads();
        uint64_t a = kAll, o = 0;
        each([&](uint64_t w, uint64_t p) {
            uint64_t x;
            if (key(w, p, x)) { a &= x; o |= x; }
        });
        const uint32_t al = __reduce_and_sync(0xFFFFFFFFu, (uint32_t)a), ah = __reduce_and_sync(0xFFFFFFFFu, (uint32_t)(a >> 32));
        const uint32_t ol = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)o), oh = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)(o >> 32));
        if (lane == 0) {
            atomicAnd(&s_and, (unsigned long long)((uint64_t)ah << 32 | al));
            atomicOr(&s_or, (unsigned long long)((uint64_t)oh << 32 | ol));
        }
        __syncthreads();
        const uint64_t diff = s_and ^ s_or;
        int shift = diff ? max(63 - __clzll((long long)diff) - 7, 0) : 0;
        uint64_t mask = shift < 56 ? ~0ull << (shift + 8) : 0ull, prefix = s_and & mask;
        for (;;) {
            if (tid < 256) hist[tid] = 0;
            __syncthreads();
            each([&](uint64_t w, uint64_t p) {
                uint64_t x;
                if (key(w, p, x) && (x & mask) == prefix) atomicAdd(&hist[(x >> shift) & 0xFFu], 1u);
            });
            __syncthreads();
            if (tid < 32) {                               // the bucket holding the need-th smallest
                const unsigned want = s_need;
                unsigned c = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) c += hist[tid * 8 + j];
                unsigned incl = c;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const unsigned y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                    if (tid >= d) incl += y;
                }
                const unsigned crossed = __ballot_sync(0xFFFFFFFFu, incl >= want);
                if (tid == __ffs(crossed) - 1) {
                    unsigned left = want - (incl - c), b = (unsigned)tid * 8;
                    while (hist[b] < left) { left -= hist[b]; ++b; }
                    const bool done = hist[b] == left || shift == 0;   // (whole bucket needed)
                    s_need = left;
                    s_n = hist[b];
                    s_prefix = prefix | (uint64_t)b << shift;
                    s_shift = done ? -1 : max(shift - 8, 0);
                }
            }
            __syncthreads();
            mask |= 0xFFull << shift;
            prefix = s_prefix;
            const int next = s_shift;
            __syncthreads();                              // (s_prefix and s_shift are written again)
            if (next < 0) {
                if (tid == 0) s_prefix = prefix | ~mask;
                __syncthreads();
                return;
            }
            shift = next;
        }
    };
    select(need0, [](uint64_t w, uint64_t, uint64_t &x) { x = w; return true; });
    const uint64_t wq = s_prefix;
    unsigned need = s_need;
    bool ties = s_n > need;                               // more keys at w = wq than needed
    uint64_t pq = kAll;
    const bool phases = ties;                             // the phases decide among them
    __syncthreads();
    if (ties) {
        select(need, [&](uint64_t w, uint64_t p, uint64_t &x) { x = p; return w == wq; });
        pq = s_prefix;
        ties = s_n > s_need;
        __syncthreads();
    }
    // list the genomes before the threshold (with ties: strictly before it)
    if (tid == 0) { s_count = 0; s_run = 0; }
    __syncthreads();
#pragma unroll 8
    for (int g = tid; g < P; g += kSelThreads) {
        const Key k = key_of(g);
        const bool in = k.x < wq || (k.x == wq && (!phases || (ties ? k.y < pq : k.y <= pq)));
        if (in && dup[g] == 0) cand[atomicAdd(&s_count, 1u)] = g;
    }
    __syncthreads();
    const unsigned before = s_count;
    need = ties && before < need0 ? need0 - before : 0;   // of those tied at it
    for (int base = 0; need && base < P && s_run < need; base += kSelThreads) {   // (uniform)
        const int g = base + tid;
        bool f = false;
        if (g < P) {
            const Key k = key_of(g);
            f = dup[g] == 0 && k.x == wq && k.y == pq;
        }
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, f);
        if (lane == 0) s_wsum[wl] = __popc(bal);
        __syncthreads();
        const unsigned mine = s_wsum[lane];               // (a scan of the warps' counts, by every warp)
        unsigned incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
            if (lane >= d) incl += y;
        }
        const unsigned run = s_run, ahead = __shfl_sync(0xFFFFFFFFu, incl - mine, wl);
        const unsigned ord = run + ahead + __popc(bal & ((1u << lane) - 1u));
        if (f && ord < need) cand[before + ord] = g;
        __syncthreads();
        if (tid == 31) s_run = run + incl;
        __syncthreads();
    }
    if (tid == 0) {
        ctl[0] = wq;
        ctl[1] = before;
        ctl[2] = 1ull;
        ctl[3] = need;
    }
}

// Keys staged in shared memory for the ranks, shared by the block's warps.
constexpr int kEliteTile = 1024;
struct EliteTile {
    uint64_t w[kEliteTile], p[kEliteTile];
    int x[kEliteTile];                             // the genome's index, or its duplicate flag
};

// Ranks of the listed genomes, a warp each: every genome before a listed one
// in the elite order is distinct and listed too, so its rank is its count of
// listed genomes before it, taken over tiles of the list staged in shared
// memory; entries from ctl[1] on have their place in the list as rank.
// elite(rank, g, lane) takes a genome of rank < Q (by the whole warp).
template <typename Take>
__device__ __forceinline__ void rank_listed(EliteTile &t, int Q, const double *fit, const unsigned long long *ctl,
                                            const int32_t *cand, Take elite)
{
    const unsigned ncand = (unsigned)ctl[1], total = ncand + (unsigned)ctl[3];
    const int lane = threadIdx.x & 31, NWB = blockDim.x >> 5;
    const uint64_t *fk = reinterpret_cast<const uint64_t *>(fit);
    for (unsigned i0 = blockIdx.x * NWB; i0 < total; i0 += gridDim.x * NWB) {   // uniform over the block
        const unsigned i = i0 + (threadIdx.x >> 5);
        const bool live = i < total, ranked = i < ncand;
        const int g = live ? cand[i] : 0;
        const uint64_t w = ranked ? fk[(size_t)g * 4] : 0, ph = ranked ? fk[(size_t)g * 4 + 1] : 0;
        int rank = (int)i;
        if (i0 < ncand) {
            unsigned cnt = 0;
            for (unsigned base = 0; base < ncand; base += kEliteTile) {
                __syncthreads();
                for (unsigned j = threadIdx.x; j < kEliteTile && base + j < ncand; j += blockDim.x) {
                    const int h = cand[base + j];
                    t.x[j] = h;
                    t.w[j] = fk[(size_t)h * 4];
                    t.p[j] = fk[(size_t)h * 4 + 1];
                }
                __syncthreads();
                if (ranked) {
                    const unsigned lim = min((unsigned)kEliteTile, ncand - base);
                    for (unsigned j = lane; j < lim; j += 32)
                        cnt += t.w[j] != w ? t.w[j] < w : t.p[j] != ph ? t.p[j] < ph : t.x[j] < g;
                }
            }
            cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
            if (ranked) rank = (int)cnt;
        }
        if (live && rank < Q) elite(rank, g, lane);
    }
}

// Ranks of all genomes, a warp each, in the order (duplicate, w, phase, index),
// over tiles of the keys: where fewer than Q are distinct, so that duplicates
// fill elite slots.
template <typename Dup, typename Take>
__device__ __forceinline__ void rank_all(EliteTile &t, int P, int Q, const double *fit, const Dup *dup, Take elite)
{
    const int lane = threadIdx.x & 31, NWB = blockDim.x >> 5;
    const uint64_t *fk = reinterpret_cast<const uint64_t *>(fit);
    for (int g0 = blockIdx.x * NWB; g0 < P; g0 += gridDim.x * NWB) {            // uniform over the block
        const int g = g0 + (threadIdx.x >> 5);
        const bool live = g < P;
        const uint64_t w = live ? fk[(size_t)g * 4] : 0, ph = live ? fk[(size_t)g * 4 + 1] : 0;
        const int dg = live ? dup[g] : 0;
        unsigned rank = 0;
        for (int base = 0; base < P; base += kEliteTile) {
            __syncthreads();
            for (int j = threadIdx.x; j < kEliteTile && base + j < P; j += blockDim.x) {
                t.w[j] = fk[(size_t)(base + j) * 4];
                t.p[j] = fk[(size_t)(base + j) * 4 + 1];
                t.x[j] = dup[base + j];
            }
            __syncthreads();
            const int lim = live ? min(kEliteTile, P - base) : 0;
            for (int j = lane; j < lim; j += 32)
                rank += t.x[j] != dg ? t.x[j] < dg : t.w[j] != w ? t.w[j] < w : t.p[j] != ph ? t.p[j] < ph : base + j < g;
        }
        rank = __reduce_add_sync(0xFFFFFFFFu, rank);
        if (live && rank < (unsigned)Q) elite((int)rank, g, lane);
    }
}

}  // namespace

}  // namespace e2
