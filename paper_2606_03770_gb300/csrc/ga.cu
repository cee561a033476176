// ga.cu -- cost tables, congestion redraw, population validation, the random
// initial population, elites and the generation step (Sec. 3.2 cost model,
// Sec. 3.4 and App. A genetic algorithm).  All randomness comes from
// Philox-4x32-10 streams keyed by (seed, generation, slot, purpose), so a
// generation replays bit for bit whatever the thread mapping.
#include "e2ga_internal.cuh"
#include "elites.cuh"

namespace e2 {

namespace {

constexpr int kBitmapWords = E2_MAX_DEVICES / 32;

// Blocks of a stage that sit in device memory: as many as fit beside the LM
// head and output layer on the master (which never leave device memory); -1
// when the head alone does not fit.
__device__ __forceinline__ long long device_blocks(uint64_t nb, uint64_t bm, uint64_t hm, uint64_t mem)
{
    if (hm > mem) return -1;
    const uint64_t cap = bm ? (mem - hm) / bm : nb;
    return (long long)(nb < cap ? nb : cap);
}

// l_d(n, master): the larger of compute time and streaming time of n identical
// blocks (plus the LM head and output layer on the master), +inf when they do
// not fit in memory (Sec. 3.2).  With GPU-CPU offload (a device with host
// memory) the blocks beyond device memory sit in host memory, if they fit,
// and run there at the host's rate and bandwidth after the device's part:
// the two times add (the plans' G--C split, Sec. 4.3).
__global__ void tables_kernel(Dims dm, const double *rate, const double *bw, const uint64_t *mem,
                              const double *rate_cpu, const double *bw_cpu, const uint64_t *mem_cpu,
                              const uint64_t *prof, double *leaf)
{
    const size_t total = (size_t)dm.V * dm.M * 2 * dm.LS;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int n = (int)(idx % dm.LS);
        size_t rest = idx / dm.LS;
        const int mf = (int)(rest & 1);
        rest >>= 1;
        const int d = (int)(rest % dm.M);
        const int v = (int)(rest / dm.M);
        double out = keyd(kInfKey);
        if (n < dm.N) {
            const uint64_t nb = (uint64_t)n + 1;
            const int V = dm.V;
            const uint64_t bm = prof[kBlkMem * V + v];
            const long long g = device_blocks(nb, bm, mf ? prof[kHeadMem * V + v] : 0ull, mem[d]);
            const uint64_t c = g < 0 ? 0ull : nb - (uint64_t)g;        // offloaded blocks
            if (g >= 0 && (c == 0 || c * bm <= mem_cpu[d])) {
                const uint64_t gb = (uint64_t)g;
                const uint64_t fl = gb * prof[kBlkFlops * V + v] + (mf ? prof[kHeadFlops * V + v] : 0ull);
                const uint64_t by = gb * prof[kBlkBytes * V + v] + (mf ? prof[kHeadBytes * V + v] : 0ull);
                const double tc = __ull2double_rn(fl) / rate[d];
                const double tm = __ull2double_rn(by) / bw[d];
                out = tc >= tm ? tc : tm;
                if (c > 0) {
                    const double hc = __ull2double_rn(c * prof[kBlkFlops * V + v]) / rate_cpu[d];
                    const double hb = __ull2double_rn(c * prof[kBlkBytes * V + v]) / bw_cpu[d];
                    out = out + (hc >= hb ? hc : hb);
                }
            }
        }
        leaf[idx] = out;
    }
}

// Per-layer profiles (blocks of several types): the time of blocks j..j+n-1 on
// device d, with and without the head, from the prefix sums PF, PB, PM
// (psum[a][v][N+1]): the larger of compute and streaming time, +inf beyond
// device memory or past the last block.
__global__ void layered_tables_kernel(Dims dm, const double *rate, const double *bw, const uint64_t *mem,
                                      const uint64_t *prof, const uint64_t *psum, double *lcost)
{
    const size_t NN = (size_t)dm.N * dm.N, total = (size_t)dm.V * dm.M * 2 * NN;
    const size_t row = (size_t)dm.N + 1, plane = (size_t)dm.V * row;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int n = (int)(idx % dm.N) + 1;
        const int j = (int)((idx / dm.N) % dm.N);
        size_t rest = idx / NN;
        const int mf = (int)(rest & 1);
        rest >>= 1;
        const int d = (int)(rest % dm.M);
        const int v = (int)(rest / dm.M);
        double out = keyd(kInfKey);
        if (j + n <= dm.N) {
            const int V = dm.V;
            const uint64_t *pf = psum + (size_t)v * row, *pb = psum + plane + (size_t)v * row,
                           *pm = psum + 2 * plane + (size_t)v * row;
            const uint64_t need = pm[j + n] - pm[j] + (mf ? prof[kHeadMem * V + v] : 0ull);
            if (need <= mem[d]) {
                const uint64_t fl = pf[j + n] - pf[j] + (mf ? prof[kHeadFlops * V + v] : 0ull);
                const uint64_t by = pb[j + n] - pb[j] + (mf ? prof[kHeadBytes * V + v] : 0ull);
                const double tc = __ull2double_rn(fl) / rate[d];
                const double tm = __ull2double_rn(by) / bw[d];
                out = tc >= tm ? tc : tm;
            }
        }
        lcost[idx] = out;
    }
}

// Per (variant, device): the most blocks the device can hold in device and
// host memory together, without and with the LM head (the number of finite
// entries of its two cost rows), and the most of them in device memory (the G
// of the G--C split; -1 where the head does not fit).  drec gathers what the
// DP's estimate needs of a device in 16 bytes (Tables); the head in blocks is
// how much later its row reaches a count of a few blocks.  prec, prech, capv
// and fpr are the pre-pass's view (Tables).
__global__ void captab_kernel(Dims dm, const double *rate, const double *bw, const uint64_t *mem,
                              const double *rate_cpu, const double *bw_cpu, const uint64_t *mem_cpu,
                              const uint64_t *prof, const uint64_t *psum, const double *leaf, int32_t *capg,
                              uint4 *drec, uint4 *prec, float2 *prech, uint32_t *capv, float4 *fpr)
{
    const size_t total = (size_t)dm.V * dm.M;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int v = (int)(idx / dm.M), d = (int)(idx - (size_t)v * dm.M);
        const int V = dm.V;
        const uint64_t N = (uint64_t)dm.N;
        const uint64_t bm = prof[kBlkMem * V + v], hm = prof[kHeadMem * V + v], mm = mem[d];
        // (each count is capped at the model's blocks before the two are added: an unlimited
        // memory, 2^64 - 1 bytes, holds 2^64 - 1 blocks of a byte)
        auto holds = [&](uint64_t bytes) { return bm && bytes / bm < N ? bytes / bm : N; };
        const uint64_t hc = holds(mem_cpu[d]);                        // blocks host memory holds
        const uint64_t g0 = holds(mm);
        const uint64_t c0 = g0 + hc;
        const uint64_t g1 = mm < hm ? 0ull : holds(mm - hm);
        const uint64_t c1 = mm < hm ? 0ull : g1 + hc;
        capg[idx * 2] = (int32_t)g0;
        capg[idx * 2 + 1] = mm < hm ? -1 : (int32_t)g1;
        const double tc = __ull2double_rn(prof[kBlkFlops * V + v]) / rate[d];
        const double tm = __ull2double_rn(prof[kBlkBytes * V + v]) / bw[d];
        const double tdev = tc >= tm ? tc : tm;
        float ratio = 0.0f;                                          // host block rate / device block rate
        if (dm.offload && hc > 0) {
            const double hf = __ull2double_rn(prof[kBlkFlops * V + v]) / rate_cpu[d];
            const double hb = __ull2double_rn(prof[kBlkBytes * V + v]) / bw_cpu[d];
            const double th = hf >= hb ? hf : hb;
            ratio = th > 0.0 ? (float)fmin(tdev / th, 1e6) : 1e6f;
        }
        uint32_t caps = (uint32_t)(c0 < N ? c0 : N) | (uint32_t)(c1 < N ? c1 : N) << 16;
        uint64_t bf = prof[kBlkFlops * V + v], bb = prof[kBlkBytes * V + v];
        if (dm.layered) {
            // per-layer profiles: the longest run of blocks the device holds, without and
            // with the head, and the least block's flops and bytes, so that the pre-pass's
            // tests stay necessary conditions
            const size_t row = (size_t)dm.N + 1, plane = (size_t)V * row;
            const uint64_t *pf = psum + (size_t)v * row, *pb = pf + plane, *pm = pb + plane;
            int n0 = 0, n1 = 0;
            for (int j = 0; j < dm.N; ++j) {
                while (j + n0 < dm.N && pm[j + n0 + 1] - pm[j] <= mm) ++n0;
                while (mm >= hm && j + n1 < dm.N && pm[j + n1 + 1] - pm[j] <= mm - hm) ++n1;
            }
            caps = (uint32_t)n0 | (uint32_t)n1 << 16;
            if (d == 0) {
                bf = pf[1] - pf[0];
                bb = pb[1] - pb[0];
                for (int j = 1; j < dm.N; ++j) {
                    const uint64_t f = pf[j + 1] - pf[j], b = pb[j + 1] - pb[j];
                    bf = f < bf ? f : bf;
                    bb = b < bb ? b : bb;
                }
            }
        }
        capv[(size_t)d * V + v] = caps;
        if (d == 0)
            fpr[v] = make_float4(__ull2float_rd(bf), __ull2float_rd(bb), __ull2float_rd(prof[kAct * V + v]), 0.0f);
        if (v == 1) prec[d].z = caps;
        if (v == dm.b_max) prec[d].w = caps;
        if (v == 0) {
            prec[d].x = __float_as_uint(__double2float_rd(__ddiv_rd(1.0, rate[d])));
            prec[d].y = __float_as_uint(__double2float_rd(__ddiv_rd(1.0, bw[d])));
            const bool host = dm.offload && mem_cpu[d] > 0;
            prech[d] = host ? make_float2(__double2float_rd(__ddiv_rd(1.0, rate_cpu[d])),
                                          __double2float_rd(__ddiv_rd(1.0, bw_cpu[d])))
                            : make_float2(0.0f, 0.0f);
        }
        const float cinv = tdev > 1e-30 ? (float)(1.0 / tdev) : 1e30f;
        float head = 1e6f;
        const int nr = c1 < 4 ? (int)c1 : N < 4 ? (int)N : 4;
        if (nr >= 1 && tdev > 0.0) {
            const double *row = leaf + (size_t)idx * 2 * dm.LS;
            const double x = (row[dm.LS + nr - 1] - row[nr - 1]) / tdev;
            if (x >= 0.0 && x < 1e6) head = (float)x;
        } else if (nr >= 1) {
            head = 0.0f;
        }
        drec[idx] = make_uint4(caps, __float_as_uint(cinv), __float_as_uint(head), __float_as_uint(ratio));
    }
}

// tau_v(a, b) = A_v / (B(a,b) * congestion(a,b)) (Sec. 3.2), its order key (the
// stage times of the variant that are no larger, ranks.cu) and itself rounded
// down to float for the DP's estimate, one 16-byte record per link and variant;
// and 1 / (B * congestion) rounded down for the latency bound.
__global__ void tau_kernel(Dims dm, const double *link_bw, const double *cong, const uint64_t *prof,
                           const uint64_t *sorted, size_t cap, LinkRec *tau, float *ibw)
{
    const size_t MM = (size_t)dm.M * dm.M, total = (size_t)dm.V * MM, n = (size_t)dm.M * 2 * dm.N;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int v = (int)(idx / MM);
        const size_t ab = idx - (size_t)v * MM;
        const double beff = link_bw[ab] * cong[ab];
        LinkRec r;
        r.t = __ull2double_rn(prof[kAct * dm.V + v]) / beff;
        const uint64_t x = dkey(r.t);
        r.key = x >= kInfKey ? 0xFFFFFFFFu : (uint32_t)count_below(sorted + v * cap, n, x + 1);
        r.lb = __double2float_rd(r.t);
        tau[idx] = r;
        if (v == 0) ibw[ab] = __double2float_rd(__ddiv_rd(1.0, beff));
    }
}

// Congestion factor of each unordered pair a < b: lo + (hi - lo) u, with u a
// 53-bit uniform from words 2(aM+b), 2(aM+b)+1 of the stream (seed, gen, 0, CONG).
__global__ void redraw_kernel(int M, uint64_t seed, uint32_t gen, double lo, double hi, double *cong)
{
    const size_t MM = (size_t)M * M;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < MM;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int a = (int)(idx / M), b = (int)(idx - (size_t)a * M);
        if (a == b) { cong[idx] = 1.0; continue; }
        if (a > b) continue;
        Stream st(seed, gen, 0, kCong);
        const uint32_t w0 = st.word(2u * (uint32_t)idx), w1 = st.word(2u * (uint32_t)idx + 1u);
        const uint64_t u53 = ((uint64_t)(w0 >> 5) << 26) | (uint64_t)(w1 >> 6);
        const double u = (double)u53 * (1.0 / 9007199254740992.0);
        const double span = hi - lo;
        const double t = span * u;
        const double f = lo + t;
        cong[idx] = f;
        cong[(size_t)b * M + a] = f;
    }
}

// An invalid genome (`lane` of `lanes` threads) is replaced by a valid one, the
// identity ordering as one prefill replica, so that no later kernel reads it.
__device__ __forceinline__ void replace_genome(const Dims &dm, const DevPop &p, int g, int32_t *err, int lane, int lanes)
{
    const int M = dm.M, K = dm.K;
    if (lane == 0) atomicMin(err, g);
    for (int i = lane; i < M; i += lanes) p.perm[(size_t)g * M + i] = (uint16_t)i;
    for (int c = lane; c < K; c += lanes) p.sizes[(size_t)g * K + c] = (uint16_t)(c ? 0 : M);
    if (lane == 0) {
        p.nclus[g] = 1;
        p.roles[g] = 0;
    }
}

// A warp per genome: the lanes check the sizes and mark the devices of the
// ordering in a shared bitmap (a device marked before is a repeat).  11 us for
// 16,384 genomes of 512 devices; a thread per genome, with its bitmap in local
// memory and its ordering read element by element, took 73.
constexpr int kValidateWarps = 4;

__global__ void __launch_bounds__(32 * kValidateWarps) validate_kernel(Dims dm, DevPop p, int32_t *err)
{
    after_previous();
    __shared__ uint32_t s_seen[kValidateWarps][kBitmapWords];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int g = blockIdx.x * kValidateWarps + wl;
    if (g >= dm.P) return;
    const int M = dm.M, K = dm.K;
    uint32_t *seen = s_seen[wl];
    for (int w = lane; w < (M + 31) >> 5; w += 32) seen[w] = 0;
    const int R = p.nclus[g];
    const uint64_t roles = p.roles[g];
    bool ok = R >= 1 && R <= K && R <= M;
    int sum = 0;
    for (int c = lane; c < K; c += 32) {
        const int s = p.sizes[(size_t)g * K + c];
        ok = ok && (c < R ? s >= 1 : s == 0);
        sum += s;
    }
    sum = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)sum);   // (by every lane, whatever it found)
    ok = ok && sum == M;
    if (R < 64) ok = ok && (roles >> R) == 0ull;
    __syncwarp();
    for (int i = lane; i < M; i += 32) {
        const int d = p.perm[(size_t)g * M + i];
        if (d >= M) ok = false;
        else if (atomicOr(&seen[d >> 5], 1u << (d & 31)) >> (d & 31) & 1u) ok = false;
    }
    if (!__all_sync(0xFFFFFFFFu, ok)) replace_genome(dm, p, g, err, lane, 32);
}

// Large populations of fleets below 64 devices: a thread per genome, its bitmap one
// word.  A warp each is bound by its chain of loads and barriers and leaves lanes
// idle: an upload of 16,384 genomes of 16 devices 29 us, of 262,144 91, by threads
// 21 and 30; up to 4,096 genomes both take 20.  (At 64 devices, rows of 128 bytes,
// threads take 28 from 64 genomes on.)
constexpr int kValidateThreads = 128;
bool validate_by_threads(int M, int P) { return M < 64 && P >= 8192; }

__global__ void __launch_bounds__(kValidateThreads) validate_small_kernel(Dims dm, DevPop p, int32_t *err)
{
    after_previous();
    const int g = blockIdx.x * kValidateThreads + threadIdx.x;
    if (g >= dm.P) return;
    const int M = dm.M, K = dm.K, R = p.nclus[g];
    const uint64_t roles = p.roles[g];
    bool ok = R >= 1 && R <= K && R <= M;
    if (R < 64) ok = ok && (roles >> R) == 0ull;
    int sum = 0;
    for (int c = 0; c < K; ++c) {
        const int s = p.sizes[(size_t)g * K + c];
        ok = ok && (c < R ? s >= 1 : s == 0);
        sum += s;
    }
    ok = ok && sum == M;
    uint64_t seen = 0;                             // (M distinct devices below M fill the first M bits)
    for (int i = 0; i < M; ++i) {
        const int d = p.perm[(size_t)g * M + i];
        ok = ok && d < M;
        seen |= d < 64 ? 1ull << d : 0ull;
    }
    ok = ok && seen == (1ull << M) - 1ull;
    if (!ok) replace_genome(dm, p, g, err, 0, 1);
}

// Fisher-Yates shuffle of the identity ordering by a warp (word M-1-t draws
// j_t, the position swapped with t, for t = M-1 .. 1).  The element that ends
// at position t is the one at j_t before step t; position p is last written
// before step t by the next larger step that drew p too, whose element came
// from its own position; so every position's element is found by following
// "the next larger step that drew this position" to a position no step drew,
// all of them at once (14 links at most in 1,600 random draws of up to 512).
// w32 [M] and aux [M] are scratch; out[t] = element t.
constexpr uint32_t kNoStep = 0xFFFFu;

__device__ __forceinline__ void random_perm(Stream st, int M, uint32_t *w32, uint16_t *aux, uint16_t *out, int lane)
{
    for (int q = lane; 4 * q < M - 1; q += 32)                    // a lane takes one block of the stream
        for (int i = 4 * q; i < 4 * q + 4 && i < M - 1; ++i) {
            const int t = M - 1 - i;
            w32[t] = below(st.word((uint32_t)i), (uint32_t)t + 1);
        }
    for (int p = lane; p < M; p += 32) aux[p] = (uint16_t)kNoStep;
    __syncwarp();
    // aux[p]: the smallest step seen that drew p; w32[t]: j_t | the next larger step that drew j_t << 16
    for (int base = (M - 1) & ~31; base >= 0; base -= 32) {
        const int t = base + lane;
        const bool step = t >= 1 && t < M;
        const uint32_t j = step ? w32[t] : 0u;
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, step ? j : 0x10000u + (unsigned)lane);
        const unsigned above = peers & ~((2u << lane) - 1u);
        uint32_t nx = kNoStep;
        if (step) nx = above ? (uint32_t)(base + __ffs(above) - 1) : aux[j];
        __syncwarp();
        if (step) {
            w32[t] = j | nx << 16;
            if (lane == __ffs(peers) - 1) aux[j] = (uint16_t)t;
        }
        __syncwarp();
    }
    for (int t = lane; t < M; t += 32) {
        uint32_t p = t ? w32[t] & 0xFFFFu : 0u, x = t ? w32[t] >> 16 : aux[0];
        while (x != kNoStep) {
            p = x;
            const uint32_t f = aux[x];
            x = f == x ? w32[x] >> 16 : f;                        // (a step that drew itself)
        }
        out[t] = (uint16_t)p;
    }
    __syncwarp();
}

// Grouping of Mr devices by a warp: replica count 1 + uniform(min(Kr, Mr)) from
// word 0; the R-1 cut points by sequential selection sampling (candidate cut t
// taken with probability needed/remaining, word t): 32 candidates at a time, up
// to the next one taken.  Writes sizes[0..Kr) (zeros past R), returns R in
// every lane.
template <typename T>
__device__ __forceinline__ int random_grouping(Stream st, int Mr, int Kr, uint32_t *w32, T *sizes, int lane)
{
    for (int q = lane; 4 * q < Mr; q += 32)
        for (int t = 4 * q; t < 4 * q + 4 && t < Mr; ++t) w32[t] = st.word((uint32_t)t);
    for (int c = lane; c < Kr; c += 32) sizes[c] = 0;
    __syncwarp();
    const int cap = Kr < Mr ? Kr : Mr;
    const int R = 1 + (int)below(w32[0], (uint32_t)cap);
    int need = R - 1, prev = 0, c = 0;
    for (int base = 1; base <= Mr - 1 && need > 0; base += 32) {
        const int t = base + lane;
        const uint32_t x = t <= Mr - 1 ? below(w32[t], (uint32_t)(Mr - t)) : 0xFFFFFFFFu;
        unsigned open = 0xFFFFFFFFu;                              // lanes not passed yet
        while (need > 0) {
            const unsigned hit = __ballot_sync(0xFFFFFFFFu, x < (uint32_t)need) & open;
            if (!hit) break;
            const int l = __ffs(hit) - 1;
            if (lane == 0) sizes[c] = (T)(base + l - prev);
            ++c;
            prev = base + l;
            --need;
            open = l == 31 ? 0u : ~0u << (l + 1);
        }
    }
    if (lane == 0) sizes[c] = (T)(Mr - prev);
    __syncwarp();
    return R;
}

__device__ __forceinline__ uint64_t random_roles(Stream st, int R)
{
    const uint64_t bits = (uint64_t)st.word(0) | ((uint64_t)st.word(1) << 32);
    return R >= 64 ? bits : (bits & ((1ull << R) - 1ull));
}

// Shared memory of a warp of the two kernels below: 32-bit words, two 16-bit
// arrays of M, and the sizes.
__host__ __device__ __forceinline__ size_t genome_bytes(int M)
{
    return (4 * (size_t)M + 2 * (size_t)((M + 1) & ~1) * 2 + 2 * E2_MAX_CLUSTERS + 3) & ~(size_t)3;
}

// Large populations of small fleets: a genome per thread, which takes the draws
// one after the other; a warp per genome leaves most lanes idle there (65,536
// genomes of 16 devices 55 us against 24, 262,144 of 8 197 against 18).
__global__ void __launch_bounds__(32) init_small_kernel(Dims dm, DevPop p, uint64_t seed)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= dm.P) return;
    const int M = dm.M, K = dm.K;
    uint16_t *perm = p.perm + (size_t)s * M, *sizes = p.sizes + (size_t)s * K;
    for (int i = 0; i < M; ++i) perm[i] = (uint16_t)i;
    Stream order(seed, 0, (uint32_t)s, kInitPerm);
    for (int t = M - 1; t >= 1; --t) {
        const uint32_t j = below(order.word((uint32_t)(M - 1 - t)), (uint32_t)t + 1);
        const uint16_t x = perm[t];
        perm[t] = perm[j];
        perm[j] = x;
    }
    for (int c = 0; c < K; ++c) sizes[c] = 0;
    Stream group(seed, 0, (uint32_t)s, kInitGroup);
    const int R = 1 + (int)below(group.word(0), (uint32_t)min(K, M));
    int c = 0, prev = 0;
    for (int t = 1; t < M && c < R - 1; ++t)
        if (below(group.word((uint32_t)t), (uint32_t)(M - t)) < (uint32_t)(R - 1 - c)) {
            sizes[c++] = (uint16_t)(t - prev);
            prev = t;
        }
    sizes[c] = (uint16_t)(M - prev);
    p.nclus[s] = (uint8_t)R;
    p.roles[s] = random_roles(Stream(seed, 0, (uint32_t)s, kInitRoles), R);
}

// Whether a thread per genome is about as fast or faster: up to 8 devices always
// (64 genomes 4 us, a warp each 6), then from 4,096 genomes at up to 16 devices (6
// against 8), 16,384 at up to 24 (16 to 20 against 18) and 65,536 at up to 32 (54
// against 57); with a quarter of those genomes it takes 6, 10 and 27 against 6, 8
// and 19.
bool init_by_threads(int M, int P) { return M <= 8 || (M <= 32 && P >= 256 << 2 * ((M + 7) / 8)); }

// A genome per warp.  (A thread per genome, swapping in global memory, took
// 125 us for 8,192 genomes of 256 devices; now 30.)
__global__ void __launch_bounds__(256) init_kernel(Dims dm, DevPop p, uint64_t seed)
{
    extern __shared__ uint32_t ga_smem[];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int s = blockIdx.x * (blockDim.x >> 5) + wl;
    if (s >= dm.P) return;
    const int M = dm.M, K = dm.K;
    uint32_t *w32 = ga_smem + (size_t)wl * (genome_bytes(M) / 4);
    uint16_t *child = reinterpret_cast<uint16_t *>(w32 + M), *aux = child + ((M + 1) & ~1);
    random_perm(Stream(seed, 0, (uint32_t)s, kInitPerm), M, w32, aux, child, lane);
    for (int i = lane; i < M; i += 32) p.perm[(size_t)s * M + i] = child[i];
    uint16_t *sizes = p.sizes + (size_t)s * K;
    const int R = random_grouping(Stream(seed, 0, (uint32_t)s, kInitGroup), M, K, w32, sizes, lane);
    const uint64_t roles = random_roles(Stream(seed, 0, (uint32_t)s, kInitRoles), R);
    if (lane == 0) {
        p.nclus[s] = (uint8_t)R;
        p.roles[s] = roles;
    }
}

// Duplicate test: dup_insert_kernel fills the fingerprint table (elites.cuh) in
// global memory and dup_lookup_kernel looks each genome up, a warp each.
// Below kDupTableFrom genomes one kernel does both (flag_duplicates).
constexpr int kDupTableFrom = 4096;

// (the table is filled with kFreeSlot beforehand)
__global__ void __launch_bounds__(256) dup_insert_kernel(int P, const uint64_t *hash, unsigned long long *tab,
                                                         unsigned mask)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < P) table_insert(tab, mask, hash[g], g);
}

__global__ void __launch_bounds__(256) dup_lookup_kernel(Dims dm, DevPop p, const uint64_t *hash,
                                                         const unsigned long long *tab, unsigned mask, int32_t *dup)
{
    after_previous();
    const int lane = threadIdx.x & 31;
    const int g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (g >= dm.P) return;
    const bool d = is_duplicate(p, tab, mask, hash, g, dm.M, dm.K, lane);
    if (lane == 0) dup[g] = d;
}

// (comparing each genome's keys with every lower-indexed one's took 8 us at
// 1,024 genomes and 28 at 2,048)
__global__ void __launch_bounds__(kDupThreads) dup_kernel(Dims dm, DevPop p, const uint64_t *hash, int32_t *dup,
                                                          unsigned mask)
{
    after_previous();
    extern __shared__ unsigned long long tab[];
    flag_duplicates(tab, mask, p, hash, dup, dm.P, dm.M, dm.K);
}

// An elite goes to slot `rank` of the next population, by the warp that ranked it.
__device__ __forceinline__ void take_elite(const Dims &dm, const double *fit, const DevPop &src, const DevPop &dst,
                                           int32_t *elite, double *elite_fit, int rank, int g, int lane)
{
    const int M = dm.M, K = dm.K;
    for (int j = lane; j < M; j += 32) dst.perm[(size_t)rank * M + j] = src.perm[(size_t)g * M + j];
    for (int j = lane; j < K; j += 32) dst.sizes[(size_t)rank * K + j] = src.sizes[(size_t)g * K + j];
    if (lane < 4) elite_fit[(size_t)rank * 4 + lane] = fit[(size_t)g * 4 + lane];
    if (lane == 0) {
        dst.nclus[rank] = src.nclus[g];
        dst.roles[rank] = src.roles[g];
        elite[rank] = g;
    }
}

// The full ranking, a warp per genome, where the selection does not apply.
__global__ void __launch_bounds__(256) rank_kernel(Dims dm, const double *fit, const int32_t *dup,
                                                   int32_t *elite, double *elite_fit, DevPop src, DevPop dst,
                                                   const unsigned long long *ctl)
{
    after_previous();
    __shared__ EliteTile tile;
    if (ctl[2] != 0) return;                       // elite_cand_rank_kernel took the elites
    rank_all(tile, dm.P, dm.Q, fit, dup, [&](int rank, int g, int lane) {
        take_elite(dm, fit, src, dst, elite, elite_fit, rank, g, lane);
    });
}

// The listed genomes' ranks, a warp each.
__global__ void __launch_bounds__(256) elite_cand_rank_kernel(Dims dm, const double *fit,
                                                              const unsigned long long *ctl, const int32_t *cand,
                                                              int32_t *elite, double *elite_fit, DevPop src, DevPop dst)
{
    after_previous();
    __shared__ EliteTile tile;
    if (ctl[2] == 0) return;
    rank_listed(tile, dm.Q, fit, ctl, cand, [&](int rank, int g, int lane) {
        take_elite(dm, fit, src, dst, elite, elite_fit, rank, g, lane);
    });
}

struct GaThr {
    uint64_t cx, half, mut, k1, k2, k3;
};

__device__ __forceinline__ bool key_before(uint64_t wa, uint64_t pa, int a, uint64_t wb, uint64_t pb, int b)
{
    if (wa != wb) return wa < wb;
    if (pa != pb) return pa < pb;
    return a < b;
}

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// One child per warp (App. A), slots [Q, P).
//  * tournaments: lanes draw the candidates, a warp reduction keeps the
//    fittest (the fitness order is strict, so this is the winner of the
//    sequential tournament);
//  * uniform crossover of the ordering chromosome, a lane per four positions;
//  * repair: first occurrence of each device by shared-memory atomicMin; a
//    later repeat is a hole; the h-th hole (by position) takes the h-th
//    missing device (by id), ranks from warp ballots;
//  * grouping and roles from one parent; then at most one mutation, its
//    sequential draws (Fisher-Yates, selection sampling) resolved by the warp.
// Bound by shared-memory work per position and, before, by the mutations that
// one lane took step by step: 156 us for 15,872 children of 512 devices, now 70.
__global__ void __launch_bounds__(256, 4) ga_kernel(Dims dm, DevPop src, DevPop dst, const double *fit,
                                                 uint64_t seed, uint32_t gen, GaThr thr)
{
    extern __shared__ uint32_t ga_smem[];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5, NWB = blockDim.x >> 5;
    const int M = dm.M, K = dm.K, P = dm.P;
    uint32_t *w32 = ga_smem + (size_t)wl * (genome_bytes(M) / 4);   // first occurrences, then random words
    uint16_t *child = reinterpret_cast<uint16_t *>(w32 + M);
    uint16_t *missing = child + ((M + 1) & ~1);
    uint16_t *ssz = missing + ((M + 1) & ~1);                     // [64] sizes
    const uint64_t *fk = reinterpret_cast<const uint64_t *>(fit);
    for (int s = dm.Q + blockIdx.x * NWB + wl; s < P; s += gridDim.x * NWB) {   // the children
        uint16_t *out_perm = dst.perm + (size_t)s * M;
        uint16_t *cs = dst.sizes + (size_t)s * K;
        // ---- two tournaments
        Stream sel(seed, gen, (uint32_t)s, kSelect);
        int par[2];
        for (int q = 0; q < 2; ++q) {
            uint64_t bw = ~0ull, bp = ~0ull;
            int bi = 0x7FFFFFFF;
            for (int t = lane; t < dm.tournament; t += 32) {
                const int cnd = (int)below(sel.word((uint32_t)(q * dm.tournament + t)), (uint32_t)P);
                const uint64_t cw = fk[(size_t)cnd * 4], cp = fk[(size_t)cnd * 4 + 1];
                if (key_before(cw, cp, cnd, bw, bp, bi)) { bw = cw; bp = cp; bi = cnd; }
            }
            for (int o = dm.tournament > 16 ? 16 : dm.tournament > 4 ? 8 : 2; o; o >>= 1) {   // (lanes past it hold no one)
                const uint64_t w2 = __shfl_xor_sync(0xFFFFFFFFu, bw, o), p2 = __shfl_xor_sync(0xFFFFFFFFu, bp, o);
                const int i2 = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
                if (key_before(w2, p2, i2, bw, bp, bi)) { bw = w2; bp = p2; bi = i2; }
            }
            par[q] = __shfl_sync(0xFFFFFFFFu, bi, 0);
        }
        // ---- uniform crossover and repair
        const uint16_t *pa = src.perm + (size_t)par[0] * M, *pb = src.perm + (size_t)par[1] * M;
        Stream cx(seed, gen, (uint32_t)s, kCross);
        if ((M & 3) == 0) {                                     // rows start on 8 bytes: four positions per load
            for (int q = lane; 4 * q < M; q += 32) {
                const ushort4 a = reinterpret_cast<const ushort4 *>(pa)[q], b = reinterpret_cast<const ushort4 *>(pb)[q];
                ushort4 x;
                x.x = (uint64_t)cx.word(4u * q) < thr.cx ? b.x : a.x;
                x.y = (uint64_t)cx.word(4u * q + 1u) < thr.cx ? b.y : a.y;
                x.z = (uint64_t)cx.word(4u * q + 2u) < thr.cx ? b.z : a.z;
                x.w = (uint64_t)cx.word(4u * q + 3u) < thr.cx ? b.w : a.w;
                reinterpret_cast<ushort2 *>(child)[2 * q] = make_ushort2(x.x, x.y);
                reinterpret_cast<ushort2 *>(child)[2 * q + 1] = make_ushort2(x.z, x.w);
            }
        } else {
            for (int q = lane; 4 * q < M; q += 32)              // a lane takes the 4 positions of one
                for (int i = 4 * q; i < 4 * q + 4 && i < M; ++i)   // block of the stream (one Philox call)
                    child[i] = (uint64_t)cx.word((uint32_t)i) < thr.cx ? pb[i] : pa[i];
        }
        for (int i = lane; i < M; i += 32) w32[i] = 0x7FFFFFFFu;
        __syncwarp();
        for (int i = lane; i < M; i += 32) atomicMin(&w32[child[i]], (uint32_t)i);
        __syncwarp();
        const unsigned lt = lanemask_lt();
        int nmiss = 0;
        for (int base = 0; base < M; base += 32) {
            const int d = base + lane;
            const bool pm = d < M && w32[d] == 0x7FFFFFFFu;
            const unsigned bm = __ballot_sync(0xFFFFFFFFu, pm);
            if (pm) missing[nmiss + __popc(bm & lt)] = (uint16_t)d;
            nmiss += __popc(bm);
        }
        __syncwarp();
        int nh = 0;
        for (int base = 0; base < M && nh < nmiss; base += 32) {   // (as many holes as missing devices)
            const int i = base + lane;
            const bool hole = i < M && w32[child[i]] != (uint32_t)i;
            const unsigned bh = __ballot_sync(0xFFFFFFFFu, hole);
            if (hole) child[i] = missing[nh + __popc(bh & lt)];
            nh += __popc(bh);
        }
        // ---- grouping and roles from one parent
        const int from = (uint64_t)cx.word((uint32_t)M) < thr.half ? par[1] : par[0];
        for (int i = lane; i < K; i += 32) ssz[i] = src.sizes[(size_t)from * K + i];
        int R = src.nclus[from];
        uint64_t rl = src.roles[from];
        __syncwarp();
        // ---- mutation
        Stream mt(seed, gen, (uint32_t)s, kMutate);
        if ((uint64_t)mt.word(0) < thr.mut) {
            const uint64_t kind = mt.word(1);
            if (kind < thr.k1) {                                   // swap two positions
                const uint32_t x = below(mt.word(2), (uint32_t)M), y = below(mt.word(3), (uint32_t)M);
                if (lane == 0) { const uint16_t t = child[x]; child[x] = child[y]; child[y] = t; }
            } else {
                int r = 0;
                if (kind < thr.k2)                                 // regroup from a random replica
                    r = (int)below(mt.word(2), (uint32_t)R);
                else if (kind >= thr.k3)                           // regenerate both chromosomes
                    random_perm(Stream(seed, gen, (uint32_t)s, kMutPerm), M, w32, missing, child, lane);
                int kept = 0;
                for (int c = lane; c < r; c += 32) kept += (int)ssz[c];
                kept = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)kept);
                __syncwarp();
                const int Rn = random_grouping(Stream(seed, gen, (uint32_t)s, kMutGroup), M - kept, K - r, w32, ssz + r, lane);
                const uint64_t nr = random_roles(Stream(seed, gen, (uint32_t)s, kMutRoles), Rn);
                const uint64_t keep = r >= 64 ? ~0ull : ((1ull << r) - 1ull);
                rl = (rl & keep) | (r >= 64 ? 0ull : (nr << r));
                R = r + Rn;
            }
        }
        __syncwarp();
        if ((M & 1) == 0) {
            for (int i = lane; i < M / 2; i += 32)
                reinterpret_cast<uint32_t *>(out_perm)[i] = reinterpret_cast<const uint32_t *>(child)[i];
        } else {
            for (int i = lane; i < M; i += 32) out_perm[i] = child[i];
        }
        for (int i = lane; i < K; i += 32) cs[i] = ssz[i];
        if (lane == 0) { dst.nclus[s] = (uint8_t)R; dst.roles[s] = rl; }
        __syncwarp();
    }
}

// 1D launch helpers
inline unsigned grid_for(size_t n, int threads, size_t cap = 152 * 32)
{
    size_t b = (n + threads - 1) / threads;
    if (b > cap) b = cap;
    return (unsigned)(b ? b : 1);
}

}  // namespace

cudaError_t launch_tables(const e2_ctx *c)
{
    const size_t total = (size_t)c->dm.V * c->dm.M * 2 * c->dm.LS;
    tables_kernel<<<grid_for(total, 256), 256, 0, c->stream>>>(c->dm, c->rate, c->bw, c->mem, c->rate_cpu, c->bw_cpu,
                                                                c->mem_cpu, c->prof, c->leaf);
    const size_t vm = (size_t)c->dm.V * c->dm.M;
    captab_kernel<<<grid_for(vm, 256), 256, 0, c->stream>>>(c->dm, c->rate, c->bw, c->mem, c->rate_cpu, c->bw_cpu,
                                                             c->mem_cpu, c->prof, c->psum, c->leaf, c->capg, c->drec,
                                                             c->prec, c->prech, c->capv, c->fpr);
    c->launches += 2;
    if (c->dm.layered) {
        const size_t lt = (size_t)c->dm.V * c->dm.M * 2 * c->dm.N * c->dm.N;
        layered_tables_kernel<<<grid_for(lt, 256), 256, 0, c->stream>>>(c->dm, c->rate, c->bw, c->mem, c->prof,
                                                                         c->psum, c->lcost);
        ++c->launches;
    }
    return cudaGetLastError();
}

cudaError_t launch_tau(const e2_ctx *c)
{
    const size_t total = (size_t)c->dm.V * c->dm.M * c->dm.M;
    tau_kernel<<<grid_for(total, 256), 256, 0, c->stream>>>(c->dm, c->link_bw, c->cong, c->prof,
                                                            c->leaf_sorted, rank_pow2((size_t)c->dm.M * 2 * c->dm.N), c->tau,
                                                            c->ibw);
    ++c->launches;
    return cudaGetLastError();
}

cudaError_t launch_redraw(const e2_ctx *c, uint64_t seed, uint32_t gen)
{
    const size_t total = (size_t)c->dm.M * c->dm.M;
    redraw_kernel<<<grid_for(total, 256), 256, 0, c->stream>>>(c->dm.M, seed, gen, c->cong_lo, c->cong_hi, c->cong);
    ++c->launches;
    return cudaGetLastError();
}

// Bytes [0, n) of one chunk by T, four loads in flight per thread.
template <class T>
__device__ __forceinline__ void copy_chunk(unsigned char *dst, const unsigned char *src, unsigned n)
{
    const unsigned full = n / sizeof(T);
    const T *s = reinterpret_cast<const T *>(src);
    T *d = reinterpret_cast<T *>(dst);
    constexpr int kUnroll = 4;
    for (unsigned i = threadIdx.x; i < full; i += blockDim.x * kUnroll) {
        T v[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
            if (i + u * blockDim.x < full) v[u] = s[i + u * blockDim.x];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
            if (i + u * blockDim.x < full) d[i + u * blockDim.x] = v[u];
    }
    for (unsigned i = full * sizeof(T) + threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

// The arrays of a population, or of an evaluation's results, to or from the
// caller's device arrays in one launch.  16-byte accesses where both sides
// start on 16 bytes (a chunk is a multiple of that), 4-byte or single ones
// otherwise.  Bound by memory on large populations (107 MB written at 16,384
// genomes of 512 devices: 22 us with the reads, part of them from L2).
__global__ void __launch_bounds__(256) copy_kernel(const __grid_constant__ CopyList l)
{
    int i = 0;
    while (i + 1 < l.n && blockIdx.x >= l.first[i + 1]) ++i;
    const size_t at = (size_t)(blockIdx.x - l.first[i]) * kCopyChunk;
    const unsigned n = (unsigned)min((unsigned long long)kCopyChunk, l.bytes[i] - at);
    const unsigned char *src = l.src[i] + at;
    unsigned char *dst = l.dst[i] + at;
    const uintptr_t bits = reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst);
    if (!(bits & 15)) copy_chunk<uint4>(dst, src, n);
    else if (!(bits & 3)) copy_chunk<uint32_t>(dst, src, n);
    else copy_chunk<unsigned char>(dst, src, n);
    if (blockIdx.x == 0 && threadIdx.x == 0 && l.word) *l.word = kNoBadGenome;
}

cudaError_t launch_copies(const CopyList &l, cudaStream_t st)
{
    copy_kernel<<<l.first[l.n], 256, 0, st>>>(l);
    return cudaGetLastError();
}

cudaError_t launch_validate(const e2_ctx *c, const DevPop &p, bool early)
{
    ++c->launches;
    const bool small = validate_by_threads(c->dm.M, c->dm.P);
    const int threads = small ? kValidateThreads : 32 * kValidateWarps, per = small ? kValidateThreads : kValidateWarps;
    return launch_kernel(small ? validate_small_kernel : validate_kernel, (unsigned)((c->dm.P + per - 1) / per), threads, 0,
                         c->stream, early, c->dm, p, c->err);
}

// Warps per CTA of a kernel with genome_bytes(M) of shared memory per warp: up to
// eight within the 48 KB that any block may use (one at 4,096 devices takes 33).
static int genome_warps(int M)
{
    int nw = 8;
    while (nw > 1 && (size_t)nw * genome_bytes(M) > 48 * 1024) nw >>= 1;
    return nw;
}

cudaError_t launch_init(const e2_ctx *c, const DevPop &p, uint64_t seed)
{
    if (init_by_threads(c->dm.M, c->dm.P)) {
        init_small_kernel<<<(unsigned)((c->dm.P + 31) / 32), 32, 0, c->stream>>>(c->dm, p, seed);
        ++c->launches;
        return cudaGetLastError();
    }
    const int nw = genome_warps(c->dm.M);
    init_kernel<<<(unsigned)((c->dm.P + nw - 1) / nw), 32 * nw, nw * genome_bytes(c->dm.M), c->stream>>>(c->dm, p, seed);
    ++c->launches;
    return cudaGetLastError();
}

// Duplicate flags, then the selection; the elites go to slots [0, Q) of dst.
cudaError_t launch_elites(const e2_ctx *c, const DevPop &p, const DevPop &dst, bool early)
{
    cudaError_t e = cudaSuccess;
    const int P = c->dm.P, Q = c->dm.Q;
    const unsigned blocks = (unsigned)(((size_t)P * 32 + 255) / 256);
    const bool table = P >= kDupTableFrom;
    const unsigned tsize = dup_table_size(P);
    if (table) {
        e = cudaMemsetAsync(c->dup_tab, 0x7F, sizeof(*c->dup_tab) * tsize, c->stream);
        if (e != cudaSuccess) return e;
        dup_insert_kernel<<<(unsigned)((P + 255) / 256), 256, 0, c->stream>>>(P, c->hash, c->dup_tab, tsize - 1);
        e = launch_kernel(dup_lookup_kernel, blocks, 256, 0, c->stream, true, c->dm, p, c->hash, c->dup_tab, tsize - 1, c->dup);
    } else {
        // (four genomes per warp and block: more blocks would fill more tables than they look up in)
        const int per = 4 * kDupThreads / 32;
        const size_t smem = sizeof(unsigned long long) * tsize;
        if (smem > 48 * 1024) {
            e = cudaFuncSetAttribute(dup_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        e = launch_kernel(dup_kernel, (unsigned)((P + per - 1) / per), kDupThreads, smem, c->stream, early, c->dm, p, c->hash,
                          c->dup, tsize - 1);
    }
    if (Q > 0) {
        if (e == cudaSuccess)
            e = launch_kernel(elite_select_kernel<int32_t>, 1, kSelThreads, 0, c->stream, true, P, Q, c->fit, c->dup,
                              c->elite_ctl, c->elite_cand);
        const unsigned rb = (unsigned)((Q + 7) / 8 < 152 * 4 ? (Q + 7) / 8 : 152 * 4);
        if (e == cudaSuccess)
            e = launch_kernel(elite_cand_rank_kernel, rb, 256, 0, c->stream, true, c->dm, c->fit, c->elite_ctl, c->elite_cand,
                              c->elite, c->elite_fit, p, dst);
        if (e == cudaSuccess)
            e = launch_kernel(rank_kernel, blocks, 256, 0, c->stream, true, c->dm, c->fit, c->dup, c->elite, c->elite_fit, p,
                              dst, c->elite_ctl);
    }
    c->launches += (table ? 2 : 1) + (Q > 0 ? 3 : 0);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_ga(const e2_ctx *c, const DevPop &src, const DevPop &dst, uint64_t seed, uint32_t gen,
                      cudaStream_t st)
{
    if (c->dm.P <= c->dm.Q) return cudaSuccess;              // no children
    GaThr thr{c->thr_cx, c->thr_half, c->thr_mut, c->thr_k1, c->thr_k2, c->thr_k3};
    const int nw = genome_warps(c->dm.M);
    const long long blocks = ((long long)(c->dm.P - c->dm.Q) + nw - 1) / nw;
    ga_kernel<<<(unsigned)(blocks < 152 * 64 ? blocks : 152 * 64), 32 * nw, nw * genome_bytes(c->dm.M), st>>>(
        c->dm, src, dst, c->fit, seed, gen, thr);
    ++c->launches;
    return cudaGetLastError();
}

// The generation step: the children (which need only the fitness) on the side
// stream, concurrently with the duplicate test and the ranks (which copy the
// elites) on the context's stream; the context's stream then waits for the
// children.
cudaError_t launch_step(const e2_ctx *c, const DevPop &src, const DevPop &dst, uint64_t seed, uint32_t gen,
                        bool after_eval)
{
    cudaError_t e = cudaEventRecord(c->ev_fork, c->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(c->side, c->ev_fork, 0);
    if (e == cudaSuccess) e = launch_ga(c, src, dst, seed, gen, c->side);
    if (e == cudaSuccess) e = cudaEventRecord(c->ev_join, c->side);
    if (e == cudaSuccess) e = launch_elites(c, src, dst, after_eval);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(c->stream, c->ev_join, 0);
    return e;
}

cudaError_t find_ga_node(cudaGraph_t graph, cudaGraphNode_t *node)
{
    *node = nullptr;
    size_t n = 0;
    cudaError_t e = cudaGraphGetNodes(graph, nullptr, &n);
    if (e != cudaSuccess) return e;
    cudaGraphNode_t nodes[64];
    if (n > 64) return cudaErrorInvalidValue;
    e = cudaGraphGetNodes(graph, nodes, &n);
    if (e != cudaSuccess) return e;
    for (size_t i = 0; i < n; ++i) {
        cudaGraphNodeType t;
        if ((e = cudaGraphNodeGetType(nodes[i], &t)) != cudaSuccess) return e;
        if (t != cudaGraphNodeTypeKernel) continue;
        cudaKernelNodeParams p{};
        if ((e = cudaGraphKernelNodeGetParams(nodes[i], &p)) != cudaSuccess) return e;
        if (p.func == reinterpret_cast<void *>(ga_kernel)) {
            *node = nodes[i];
            return cudaSuccess;
        }
    }
    return cudaErrorInvalidValue;
}

cudaError_t set_ga_node(const e2_ctx *c, cudaGraphExec_t exec, cudaGraphNode_t node, const DevPop &src,
                        const DevPop &dst, uint64_t seed, uint32_t gen)
{
    cudaKernelNodeParams p{};
    cudaError_t e = cudaGraphKernelNodeGetParams(node, &p);     // launch shape as recorded
    if (e != cudaSuccess) return e;
    Dims dm = c->dm;
    DevPop s = src, d = dst;
    const double *fit = c->fit;
    GaThr thr{c->thr_cx, c->thr_half, c->thr_mut, c->thr_k1, c->thr_k2, c->thr_k3};
    void *args[] = {&dm, &s, &d, &fit, &seed, &gen, &thr};
    p.kernelParams = args;
    p.extra = nullptr;
    return cudaGraphExecKernelNodeSetParams(exec, node, &p);
}

}  // namespace e2
