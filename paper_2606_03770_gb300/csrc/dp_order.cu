// dp_order.cu -- DP_Pipe (Alg. 1, Eq. 1-2) for models of identical blocks, one
// DP run per warp, by order statistics instead of columns.
//
// With identical blocks (Sec. 3.2: the premise that lets the paper fix the
// node order) a stage's time depends only on its device, its block count n and
// whether it is the master: two non-decreasing rows per device, l_k(n) and
// l_k^head(n).  A bottleneck T lets device k hold at most cap_k(T) = #{n :
// l_k(n) <= T} blocks, and a partition of B blocks over devices 1..k with
// every stage and link time <= T exists exactly when
//     tau_i <= T, cap_i(T) >= 1 for i <= k, and sum_i cap_i(T) >= B,
// since any n_i between 1 and cap_i(T) that add up to B will do.  So no cell
// of Alg. 1's table has to be computed from its predecessors:
//     D_k[B] = max(links, first-block times, the B-th smallest entry of rows 1..k).
//
// The bottleneck.  Master mu replaces row mu by its head row, so
//     V* = the least T >= links for which some mu has cap^head_mu(T) >= 1,
//          cap_i(T) >= 1 elsewhere, and sum cap - cap_mu + cap^head_mu >= N,
// mu* = the smallest such mu at V* (Alg. 1's first-wins argmin).  Lane k holds
// device k (or devices k, k + 32, ...): an arithmetic estimate of T (Newton on
// the linear costs, in float: no loads) gives each device's count within a
// block or two, and the warp then walks the rows entry by entry, up or down,
// to the exact threshold.  On the repository's workloads the walk is 1.5 to
// 2.4 steps on average and 8 at most; after kMaxWalk steps (costs the estimate
// does not describe) it becomes a bisection over the order keys.
//
// Traceback.  Alg. 1 keeps the smallest split, i.e. device k takes n_k =
// min(cap_k(D_k[B_k]), what leaves one block for each earlier device).  With
// e = sum_{i<=k} cap_i(D_k) - B_k the excess capacity of the prefix, taking
// n_k = cap_k leaves the prefix 1..k-1 with the same excess, and D_{k-1} is
// what remains after dropping the e largest entries of its rows (down to the
// prefix's largest link or first-block time).  e = 0 (most runs): every device
// takes its cap.  Otherwise the threshold changes only where the prefix loses
// the link that set it or enough of the entries tied at it, and the stretch
// between two such places is settled by one warp scan.
//
// Comparisons are between 32-bit order keys (exact ranks of the float64 times,
// ranks.cu); T and Lambda come from the float64 tables, so every result is the
// oracle's to the bit.
//
// Bound by latency and issue: about eight dependent L2 round trips per run and
// a few hundred warp instructions.  The column DP that this replaces did
// O(m W log W) shared-memory probes per run.
#include "e2ga_internal.cuh"

namespace e2 {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr uint32_t kInf = 0xFFFFFFFFu;        // the order key of +inf
constexpr int kMaxWalk = 16;
constexpr int kMaxDrop = 6;                   // entries dropped one threshold at a time in the traceback
// CTAs per SM that the registers are capped for (56, 72, 80, 96 and 255 a thread).
constexpr int order_ctas(int D) { return D == 1 ? 3 : D == 2 ? 7 : D == 3 ? 6 : D == 4 ? 5 : 2; }

// Items per claim at most.  With a device per lane a claim's partitions stay
// in shared memory ([item][device] device | blocks << 16, rows of 33 words
// against bank conflicts) for the latency sums.
constexpr int kClaim = 16, kClaimRow = 33;

// A non-negative double as a float rounded toward zero (0 below the float
// range, a large value above it), without the float64 conversion unit.
__device__ __forceinline__ float trunc_float(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    if (hi < 0x38100000u) return 0.0f;
    if (hi >= 0x47E00000u) return 1e38f;
    return __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
}

// A link's record in one 16-byte load.
__device__ __forceinline__ LinkRec load_link(const Tables &tb, size_t i)
{
    const uint4 x = reinterpret_cast<const uint4 *>(tb.tau)[i];
    LinkRec r;
    r.t = __hiloint2double((int)x.y, (int)x.x);
    r.key = x.z;
    r.lb = __uint_as_float(x.w);
    return r;
}

// Exclusive prefix sums over devices 0..32 D - 1 (lane l holds l, l + 32, ...).
template <int D>
__device__ __forceinline__ void exclusive_sums(const int (&x)[D], int (&ex)[D], int lane)
{
    int carry = 0;
#pragma unroll
    for (int j = 0; j < D; ++j) {
        int inc = x[j];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += y;
        }
        ex[j] = carry + inc - x[j];
        if (j + 1 < D) carry += __shfl_sync(kFull, inc, 31);
    }
}

// The largest device whose flag is set (-1: none).
template <int D>
__device__ __forceinline__ int highest(const bool (&f)[D])
{
    int best = -1;
#pragma unroll
    for (int j = 0; j < D; ++j) {
        const unsigned b = __ballot_sync(kFull, f[j]);
        if (b) best = j * 32 + 31 - __clz(b);
    }
    return best;
}

// Persistent warps over the items of class cls.  An item is one (genome,
// replica, role): a prefill run, or the decode sweep from the largest batch
// the pre-pass kept down to the first that meets Min_TPS (Alg. 2).  A warp
// claims several items at a time and sums their latencies Lambda (a serial
// chain of float64 additions in pipeline order, on a pipe of 2 lanes per SM)
// one item per lane at the end.  Loops that rarely run twice are not unrolled:
// unrolled by the compiler's default they filled the instruction cache (2.2
// cycles per issued instruction waiting for it, now 0.6; class 0 at 512 devices
// 159 -> 150 us).
template <int D, bool OFF>
__global__ void __launch_bounds__(32 * dp_order_warps(D == 1 ? 0 : 1), order_ctas(D)) dp_order_kernel(Dims dm, Tables tb, DevPop pop, EvalOut out, WorkList wl,
                                                       const int32_t *slot_off, SplitOut so, int cls)
{
    after_previous();
    extern __shared__ uint32_t s_dyn[];                    // D == 1: the claim's partitions, per warp
                                                           // D > 1: the run's device ids, per warp
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int K = dm.K, M = dm.M, N = dm.N;
    const uint32_t LS = (uint32_t)dm.LS;
    const uint32_t *lr = tb.leaf_rank;
    uint32_t *part = s_dyn + (size_t)wid * (kClaim * kClaimRow);
    uint16_t *dev = reinterpret_cast<uint16_t *>(s_dyn) + (size_t)wid * (32 * D);
    const unsigned begin = cls ? wl.ctrl[kCtrlEnd] : 0u, end = wl.ctrl[kCtrlEnd + cls];
    // claims of about a quarter of a warp's share (half for the large replicas):
    // the lanes of the latency sums fill up, and the last claims still even out
    const unsigned warps = gridDim.x * (blockDim.x >> 5);
    const unsigned batch = min((unsigned)kClaim, max(1u, (end - begin) / ((D == 1 ? 4u : 2u) * warps)));
    unsigned long long st_runs = 0, st_cells = 0;
    unsigned st_probes = 0;

    for (;;) {
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(&wl.ctrl[kCtrlNext + cls], batch);
        at = __shfl_sync(kFull, at, 0);
        if (at >= end) break;
        const int nb = (int)min(batch, end - at);
        // lane j: item j of the claim
        uint64_t item = 0;
        int my_m = 0, my_off = 0;
        if (lane < nb) {
            item = wl.items[at + lane];
            const size_t slot = (size_t)(item >> 8);
            my_m = pop.sizes[slot];
            my_off = slot_off[slot];
        }
        int acc_m = 0, acc_v = 0, acc_mu = 0;              // lane j: item j's accepted run (m = 0: none)

        for (int ji = 0; ji < nb; ++ji) {
            const uint64_t it = __shfl_sync(kFull, item, ji);
            const int m = __shfl_sync(kFull, my_m, ji), off = __shfl_sync(kFull, my_off, ji);
            const int slot = (int)(it >> 8), role = (int)((it >> 7) & 1u), top = (int)(it & 0x3Fu);
            const int g = slot / K;
            const int W = N - m + 1;
            const size_t sv = (size_t)slot * 2 + role;
            int16_t *lay = dm.role_search ? so.layers + ((size_t)g * 2 + role) * M + off
                                          : out.layers + (size_t)g * M + off;
            // ---- the replica's devices and each one's predecessor in the pipeline
            int d[D], dp[D];
#pragma unroll
            for (int j = 0; j < D; ++j) {
                const int k = lane + 32 * j;
                d[j] = k < m ? pop.perm[(size_t)g * M + off + k] : 0;
            }
            if (D == 1) {
                dp[0] = __shfl_up_sync(kFull, d[0], 1);
            } else {
#pragma unroll
                for (int j = 0; j < D; ++j) dev[lane + 32 * j] = (uint16_t)d[j];
                __syncwarp();
#pragma unroll
                for (int j = 0; j < D; ++j) dp[j] = lane + 32 * j ? dev[lane + 32 * j - 1] : 0;
                __syncwarp();
            }
            bool served = false;
            for (int bit = top; bit >= 0 && !served; --bit) {
                const int v = role ? bit + 1 : 0;
                const size_t vM = (size_t)v * M;
                // ---- per device: capacities, cost estimate, row offset, link key
                uint32_t ro[D];
                int c0[D], c1[D];
                float cinv[D], hb[D], hr[D], gcap[D];
                uint32_t tr[D];
                double tk[D];                              // link times (D > 1: read at the end)
                uint32_t floor_l = 0;
                float tf_l = 0.0f, hmin_l = 3e38f;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    const int k = lane + 32 * j;
                    ro[j] = 0; c0[j] = c1[j] = 0; cinv[j] = hb[j] = hr[j] = gcap[j] = 0.0f; tr[j] = 0; tk[j] = 0.0;
                    if (k < m) {
                        const uint4 rec = tb.drec[vM + d[j]];
                        c0[j] = min((int)(rec.x & 0xFFFFu), W);
                        c1[j] = min((int)(rec.x >> 16), W);
                        cinv[j] = __uint_as_float(rec.y);
                        hb[j] = __uint_as_float(rec.z);
                        if (OFF) {
                            hr[j] = __uint_as_float(rec.w);
                            gcap[j] = (float)tb.capg[(vM + d[j]) * 2];
                        }
                        ro[j] = (uint32_t)(vM + d[j]) * 2u * LS;
                        if (k > 0) {
                            const LinkRec link = load_link(tb, (vM + dp[j]) * M + d[j]);
                            tr[j] = link.key;
                            tf_l = fmaxf(tf_l, link.lb);
                            if (D == 1) tk[j] = link.t;
                        }
                        if (c1[j] >= 1) hmin_l = fminf(hmin_l, hb[j]);
                        if (c0[j] >= 1) tf_l = fmaxf(tf_l, __fdividef(1.0f, cinv[j]));
                    }
                    floor_l = max(floor_l, tr[j]);
                }
                const uint32_t floor_r = __reduce_max_sync(kFull, floor_l);
                // ---- the estimate of a threshold: Newton on sum_k min(T / c_k - 1/2, cap_k) = target
                //      over devices 0..lim-1, from the left (the sum is concave in T); x_of is
                //      device k's count at T, less the head's blocks on the master
                const float fxs = tb.fxs[v];
                int head_at = -1;
                auto x_of = [&](int j, float T, float &slope) -> float {
                    float x = T * cinv[j];
                    slope = cinv[j];
                    if (OFF && x > gcap[j] && hr[j] > 0.0f) {
                        x = gcap[j] + (x - gcap[j]) * hr[j];
                        slope *= hr[j];
                    }
                    return lane + 32 * j == head_at ? x - hb[j] : x;
                };
                auto newton = [&](const int (&cap)[D], int lim, float target) -> float {
                    unsigned a0 = 0;
#pragma unroll
                    for (int j = 0; j < D; ++j)
                        if (lane + 32 * j < lim) a0 += (unsigned)fminf(cinv[j] * fxs, 8388608.0f);
                    a0 = __reduce_add_sync(kFull, a0);
                    float T = (target + 0.5f * (float)lim) * fxs / (float)max(a0, 1u);
#pragma unroll 1
                    for (int itn = 0; itn < 6; ++itn) {
                        int s = 0;
                        unsigned a = 0;
#pragma unroll
                        for (int j = 0; j < D; ++j) {
                            if (lane + 32 * j >= lim) continue;
                            float slope;
                            const float x = x_of(j, T, slope);
                            const bool full = cap[j] == 0 || x >= (float)cap[j] + 0.5f;
                            s += full ? cap[j] * 16 : (int)(x * 16.0f) - 8;
                            a += full ? 0u : (unsigned)fminf(slope * fxs, 8388608.0f);
                        }
                        s = __reduce_add_sync(kFull, s);
                        a = __reduce_add_sync(kFull, a);
                        const float rest = target - (float)s * 0.0625f;
                        if (fabsf(rest) < 0.5f || a == 0) break;
                        T += rest * fxs / (float)a;
                    }
                    return T;
                };
                // V*: a target of N blocks and the least head
                const float t_min = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(tf_l)));
                const float hmin = __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(hmin_l)));
                const float T = fmaxf(newton(c0, m, (float)N + (hmin < 1e6f ? floorf(hmin) : 0.0f)), t_min);
                // ---- counts at the estimate, without and with the head, and the keys around them
                int n[D], nh[D];
                uint32_t lo[D], hi[D], loh[D], hih[D];
                uint32_t r_l = 0;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    float slope;
                    n[j] = min(max((int)x_of(j, T, slope), 1), c0[j]);
                    nh[j] = min(max(n[j] - (int)(hb[j] + 0.5f), 0), c1[j]);
                    lo[j] = n[j] ? lr[ro[j] + n[j] - 1] : 0u;
                    hi[j] = n[j] < c0[j] ? lr[ro[j] + n[j]] : kInf;
                    loh[j] = nh[j] ? lr[ro[j] + LS + nh[j] - 1] : 0u;
                    hih[j] = nh[j] < c1[j] ? lr[ro[j] + LS + nh[j]] : kInf;
#pragma unroll 1
                    while (lo[j] == kInf) {                // (a time that overflowed to +inf)
                        hi[j] = kInf;
                        --n[j];
                        lo[j] = n[j] ? lr[ro[j] + n[j] - 1] : 0u;
                    }
                    r_l = max(r_l, lo[j]);
                    st_probes += 4;
                }
                // ---- the counts of one threshold R: the largest key among them
                uint32_t R = max(min(floor_r, kInf - 1u), __reduce_max_sync(kFull, r_l));
                auto raise = [&](uint32_t to) {            // (to < kInf, so the loops end)
#pragma unroll
                    for (int j = 0; j < D; ++j) {
#pragma unroll 1
                        while (hi[j] <= to) {
                            lo[j] = hi[j];
                            ++n[j];
                            hi[j] = n[j] < c0[j] ? lr[ro[j] + n[j]] : kInf;
                            ++st_probes;
                        }
#pragma unroll 1
                        while (hih[j] <= to) {
                            loh[j] = hih[j];
                            ++nh[j];
                            hih[j] = nh[j] < c1[j] ? lr[ro[j] + LS + nh[j]] : kInf;
                            ++st_probes;
                        }
                    }
                };
#pragma unroll
                for (int j = 0; j < D; ++j)
#pragma unroll 1
                    while (nh[j] > 0 && loh[j] > R) {
                        hih[j] = loh[j];
                        --nh[j];
                        loh[j] = nh[j] ? lr[ro[j] + LS + nh[j] - 1] : 0u;
                        ++st_probes;
                    }
                raise(R);
                // the masters that a set of counts leaves feasible; true if there is one
                auto feasible = [&](const int (&a)[D], const int (&ah)[D], unsigned (&fm)[D]) -> bool {
                    int s = 0;
#pragma unroll
                    for (int j = 0; j < D; ++j) s += a[j] + ((lane + 32 * j < m && a[j] == 0) ? 1 << 20 : 0);
                    s = __reduce_add_sync(kFull, s);
                    const int zero = s >> 20, S = s & 0xFFFFF;
                    bool any = false;
#pragma unroll
                    for (int j = 0; j < D; ++j) {
                        const bool f = ah[j] >= 1 && zero - (a[j] == 0) == 0 && S - a[j] + ah[j] >= N;
                        fm[j] = __ballot_sync(kFull, f);
                        any |= fm[j] != 0;
                    }
                    return any;
                };
                unsigned fm[D];
                bool found = feasible(n, nh, fm);
                int steps = 0;
                uint32_t below = 0;                        // (bisection) largest key known infeasible
                if (floor_r == kInf) {                     // a link of infinite time: no partition
                    found = false;
                } else if (found) {                        // walk down to the least feasible threshold
#pragma unroll 1
                    for (;;) {
                        uint32_t x = 0;
#pragma unroll
                        for (int j = 0; j < D; ++j) x = max(x, max(lo[j], loh[j]));
                        x = __reduce_max_sync(kFull, x);
                        if (x <= floor_r) { R = floor_r; break; }
                        R = x;
                        if (++steps > kMaxWalk) break;
                        int n2[D], nh2[D];
                        uint32_t lo2[D], loh2[D];
#pragma unroll
                        for (int j = 0; j < D; ++j) {
                            n2[j] = n[j]; nh2[j] = nh[j]; lo2[j] = lo[j]; loh2[j] = loh[j];
#pragma unroll 1
                            while (n2[j] > 0 && lo2[j] == R) {
                                --n2[j];
                                lo2[j] = n2[j] ? lr[ro[j] + n2[j] - 1] : 0u;
                                ++st_probes;
                            }
#pragma unroll 1
                            while (nh2[j] > 0 && loh2[j] == R) {
                                --nh2[j];
                                loh2[j] = nh2[j] ? lr[ro[j] + LS + nh2[j] - 1] : 0u;
                                ++st_probes;
                            }
                        }
                        unsigned f2[D];
                        if (!feasible(n2, nh2, f2)) break;
#pragma unroll
                        for (int j = 0; j < D; ++j) {
                            n[j] = n2[j]; nh[j] = nh2[j]; lo[j] = lo2[j]; loh[j] = loh2[j]; fm[j] = f2[j];
                        }
                    }
                    below = floor_r;                       // (not yet known infeasible: tested below)
                } else {                                   // walk up to the first feasible one
#pragma unroll 1
                    while (!found) {
                        uint32_t x = kInf;
#pragma unroll
                        for (int j = 0; j < D; ++j) x = min(x, min(hi[j], hih[j]));
                        x = __reduce_min_sync(kFull, x);
                        if (x == kInf) break;              // no partition
                        if (++steps > kMaxWalk) break;
                        R = x;
                        raise(R);
                        found = feasible(n, nh, fm);
                    }
                    below = R;
                }
                ++st_runs;
                st_cells += m;
                if (steps > kMaxWalk) {
                    // costs that the estimate does not describe: bisection over the keys
                    auto counts_at = [&](uint32_t to) {
#pragma unroll
                        for (int j = 0; j < D; ++j) {
                            int a = 0, b = c0[j];
#pragma unroll 1
                            while (a < b) {
                                const int mid = (a + b) >> 1;
                                if (lr[ro[j] + mid] <= to) a = mid + 1;
                                else b = mid;
                                ++st_probes;
                            }
                            n[j] = a;
                            a = 0; b = c1[j];
#pragma unroll 1
                            while (a < b) {
                                const int mid = (a + b) >> 1;
                                if (lr[ro[j] + LS + mid] <= to) a = mid + 1;
                                else b = mid;
                                ++st_probes;
                            }
                            nh[j] = a;
                        }
                    };
                    uint32_t good = found ? R : kInf - 1u;
                    if (found) {                           // the floor itself may do
                        counts_at(floor_r);
                        if (feasible(n, nh, fm)) good = below = floor_r;
                    } else {
                        counts_at(good);
                        found = feasible(n, nh, fm);
                    }
#pragma unroll 1
                    while (found && good - below > 1u) {
                        const uint32_t mid = below + (good - below) / 2u;
                        counts_at(mid);
                        if (feasible(n, nh, fm)) good = mid;
                        else below = mid;
                    }
                    if (found) {
                        R = good;
                        counts_at(R);
                        feasible(n, nh, fm);
#pragma unroll
                        for (int j = 0; j < D; ++j) {
                            lo[j] = n[j] ? lr[ro[j] + n[j] - 1] : 0u;
                            loh[j] = nh[j] ? lr[ro[j] + LS + nh[j] - 1] : 0u;
                        }
                    }
                }
                if (!found) {
                    // the pre-pass tested this variant's memory exactly, unless the
                    // profile's costs do not grow with the batch: then the batches
                    // below the largest that passed run untested, and may have no
                    // partition.  Otherwise this cannot happen.
                    if (lane == 0 && (dm.grows || !role)) atomicAdd(&out.stats[kStDeviceErrors], 1ull);
                    continue;
                }
                // ---- mu*, its rows, and the excess of the whole pipeline
                int mus = 0;
#pragma unroll
                for (int j = D - 1; j >= 0; --j)
                    if (fm[j]) mus = j * 32 + __ffs(fm[j]) - 1;
                int C[D], nk[D];
                int s_l = 0;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    const bool head = lane + 32 * j == mus;
                    C[j] = head ? nh[j] : n[j];
                    if (head) { lo[j] = loh[j]; ro[j] += LS; }
                    nk[j] = C[j];
                    s_l += C[j];
                }
                head_at = mus;
                int e = (int)__reduce_add_sync(kFull, s_l) - N;
                // ---- a decode batch too slow whatever the traceback does: the partition takes the
                //      counts C less e blocks in all, so Lambda is at least the links and
                //      sum C_k c_k - e max c_k (the head only adds); in fixed point as below.
                //      About three quarters of the batches that fail the test end here.
                if (D == 1 && !OFF && role && dm.lam_fx > 0.0f) {
                    const float x = (float)C[0] * __fdividef(1.0f, cinv[0]) + trunc_float(tk[0]);
                    const unsigned s = __reduce_add_sync(
                        kFull, lane < m ? (unsigned)fminf(x * (1.0f - 3e-6f) * dm.lam_fx, 8388608.0f) : 0u);
                    const float back = fminf((float)e * t_min * (1.0f + 3e-6f) * dm.lam_fx, 1e9f);
                    if (s > (1u << 22) + 64u + (unsigned)back) continue;
                }
                // ---- traceback
                if (e > 0) {
                    // fl[k]: the largest link or first-block key of devices 0..k
                    uint32_t fl[D];
                    uint32_t carry = 0;
#pragma unroll
                    for (int j = 0; j < D; ++j) {
                        const int k = lane + 32 * j;
                        uint32_t x = k < m ? max(tr[j], lr[ro[j]]) : 0u;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const uint32_t y = __shfl_up_sync(kFull, x, o);
                            if (lane >= o) x = max(x, y);
                        }
                        fl[j] = max(x, carry);
                        if (j + 1 < D) carry = __shfl_sync(kFull, fl[j], 31);
                    }
                    int lim = m;                           // devices 0..lim-1 are undecided
#pragma unroll 1
                    for (;;) {
                        uint32_t f = 0;
#pragma unroll
                        for (int j = 0; j < D; ++j) {
                            const uint32_t y = __shfl_sync(kFull, fl[j], (lim - 1) & 31);
                            if (j == (lim - 1) >> 5) f = y;
                        }
                        // drop the e largest entries of the prefix, down to f: many of them by a
                        // new estimate (and up again from there if it dropped too many; the whole
                        // pipeline's threshold is V*, with nothing to drop) ...
                        uint32_t x = 0;
                        int C2[D];
                        if (e > kMaxDrop && lim < m) {
                            int total = 0;
#pragma unroll
                            for (int j = 0; j < D; ++j) total += lane + 32 * j < lim ? C[j] : 0;
                            const int B = __reduce_add_sync(kFull, total) - e;
                            const float Tp = newton(C, lim, (float)B);
                            uint32_t lo2[D], hi2[D];
                            uint32_t r = 0;
#pragma unroll
                            for (int j = 0; j < D; ++j) {
                                C2[j] = 0; lo2[j] = 0; hi2[j] = kInf;
                                if (lane + 32 * j < lim) {
                                    float slope;
                                    C2[j] = min(max((int)x_of(j, Tp, slope), 1), C[j]);
                                    lo2[j] = lr[ro[j] + C2[j] - 1];
                                    if (C2[j] < C[j]) hi2[j] = lr[ro[j] + C2[j]];
                                    st_probes += 2;
                                }
                                r = max(r, lo2[j]);
                            }
                            r = max(f, __reduce_max_sync(kFull, r));
#pragma unroll 1
                            for (;;) {
                                int sum = 0;
#pragma unroll
                                for (int j = 0; j < D; ++j) {
#pragma unroll 1
                                    while (hi2[j] <= r) {
                                        lo2[j] = hi2[j];
                                        ++C2[j];
                                        hi2[j] = C2[j] < C[j] ? lr[ro[j] + C2[j]] : kInf;
                                        ++st_probes;
                                    }
                                    sum += C2[j];
                                }
                                sum = __reduce_add_sync(kFull, sum);
                                e = sum - B;
                                if (e >= 0) break;
                                r = kInf;
#pragma unroll
                                for (int j = 0; j < D; ++j) r = min(r, hi2[j]);
                                r = __reduce_min_sync(kFull, r);   // (finite: the prefix's caps add up to B + e)
                            }
#pragma unroll
                            for (int j = 0; j < D; ++j)
                                if (lane + 32 * j < lim) { C[j] = C2[j]; lo[j] = lo2[j]; }
                        }
                        // ... and the rest one threshold at a time
#pragma unroll 1
                        while (e > 0) {
                            x = 0;
#pragma unroll
                            for (int j = 0; j < D; ++j) if (lane + 32 * j < lim) x = max(x, lo[j]);
                            x = __reduce_max_sync(kFull, x);
                            if (x <= f) break;
                            uint32_t lo2[D];
                            int cnt = 0;
#pragma unroll
                            for (int j = 0; j < D; ++j) {
                                C2[j] = C[j];
                                lo2[j] = lo[j];
                                if (lane + 32 * j < lim)
#pragma unroll 1
                                    while (C2[j] > 0 && lo2[j] == x) {
                                        --C2[j];
                                        lo2[j] = C2[j] ? lr[ro[j] + C2[j] - 1] : 0u;
                                        ++st_probes;
                                    }
                                cnt += C[j] - C2[j];
                            }
                            cnt = __reduce_add_sync(kFull, cnt);
                            if (cnt > e) break;
#pragma unroll
                            for (int j = 0; j < D; ++j) { C[j] = C2[j]; lo[j] = lo2[j]; }
                            e -= cnt;
                        }
                        if (e == 0) {
#pragma unroll
                            for (int j = 0; j < D; ++j) if (lane + 32 * j < lim) nk[j] = C[j];
                            break;
                        }
                        // where the blocks run out (every earlier device keeps one), and
                        // where the threshold next changes
                        int q[D], Q[D];
                        bool fx[D];
#pragma unroll
                        for (int j = 0; j < D; ++j) q[j] = lane + 32 * j < lim ? C[j] - 1 : 0;
                        exclusive_sums<D>(q, Q, lane);
#pragma unroll
                        for (int j = 0; j < D; ++j) fx[j] = lane + 32 * j < lim && Q[j] <= e;
                        const int kx = highest<D>(fx);
                        int next;
                        if (x > f) {                       // more than e entries tied at x: until e are left
                            int t[D], Dx[D];
#pragma unroll
                            for (int j = 0; j < D; ++j) t[j] = C[j] - C2[j];
                            exclusive_sums<D>(t, Dx, lane);
#pragma unroll
                            for (int j = 0; j < D; ++j) fx[j] = lane + 32 * j < lim && Dx[j] <= e;
                            next = highest<D>(fx);
                        } else {                           // until the prefix loses the link that set f
                            next = 0;
#pragma unroll
                            for (int j = 0; j < D; ++j)
                                next += __popc(__ballot_sync(kFull, lane + 32 * j < lim && fl[j] < f));
                        }
                        const int stop = max(next, kx);
#pragma unroll
                        for (int j = 0; j < D; ++j) {
                            const int k = lane + 32 * j;
                            if (k >= stop && k < lim) nk[j] = C[j];
                            if (kx >= next && k < lim) {
                                if (k == kx) nk[j] = Q[j] + C[j] - e;
                                else if (k < kx) nk[j] = 1;
                            }
                        }
                        if (kx >= next) break;
                        lim = next;
                    }
                }
                // ---- T: the largest stage or link time of the partition (equal to V*); the
                //      decode test on Lambda, in fixed point where that decides it
                double lk[D];
                uint64_t tmax = 0;
                float lam_f = 0.0f;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    const int k = lane + 32 * j;
                    lk[j] = 0.0;
                    if (k < m) {
                        lk[j] = tb.leaf[ro[j] + nk[j] - 1];
                        if (D > 1 && k > 0) tk[j] = tb.tau[(vM + dp[j]) * M + d[j]].t;
                    }
                    tmax = umax64(tmax, umax64(dkey(lk[j]), dkey(tk[j])));
                    lam_f += trunc_float(lk[j]) + trunc_float(tk[j]);
                }
                const uint32_t th = (uint32_t)(tmax >> 32), TH = __reduce_max_sync(kFull, th);
                const uint32_t TL = __reduce_max_sync(kFull, th == TH ? (uint32_t)tmax : 0u);
                bool ok = true;
                if (role && dm.lam_max < keyd(kInfKey)) {
                    // the lanes' parts of Lambda / Lambda_max in units of 2^-22, rounded down
                    // (each lane off by less than one unit and 2^-19 relative): well above
                    // or below 2^22 the test is decided, otherwise the exact sum decides
                    unsigned s = 1u << 22;
                    if (dm.lam_fx > 0.0f) s = __reduce_add_sync(kFull, (unsigned)fminf(lam_f * dm.lam_fx, 8388608.0f));
                    if (s + 48u <= 1u << 22 && dm.lam_fx > 0.0f) {
                        ok = true;
                    } else if (s > (1u << 22) + 8u) {
                        ok = false;
                    } else {
                        double lam = 0.0;
#pragma unroll
                        for (int j = 0; j < D; ++j)
                            for (int q = 0; q < 32 && 32 * j + q < m; ++q) {
                                const double lq = __shfl_sync(kFull, lk[j], q), tq = __shfl_sync(kFull, tk[j], q);
                                if (j == 0 && q == 0) lam = lq;
                                else { lam = lam + tq; lam = lam + lq; }
                            }
                        ok = lam <= dm.lam_max;            // 1.0 / lam >= Min_TPS
                    }
                }
                if (!ok) continue;
                served = true;
#pragma unroll
                for (int j = 0; j < D; ++j)
                    if (lane + 32 * j < m) lay[lane + 32 * j] = (int16_t)nk[j];
                if (D == 1) part[ji * kClaimRow + lane] = (uint32_t)d[0] | (uint32_t)nk[0] << 16;
                if (lane == ji) { acc_m = m; acc_v = v; acc_mu = mus; }
                if (lane == 0) {
                    const double Tv = keyd(((uint64_t)TH << 32) | TL);
                    if (dm.role_search) {
                        so.mu[sv] = (int16_t)mus;
                        so.code[sv] = (int16_t)bit;
                        so.T[sv] = Tv;
                    } else {
                        out.master[slot] = (int16_t)mus;
                        out.bsel[slot] = (int16_t)(role ? bit + 1 : 0);
                        out.T[slot] = Tv;
                    }
                }
            }
            if (!served) {
                if (dm.role_search) {
                    if (lane == 0) so.code[sv] = -1;
                } else {
                    for (int k = lane; k < m; k += 32) lay[k] = -1;
                    if (lane == 0) {
                        out.master[slot] = -1; out.bsel[slot] = -1;
                        out.T[slot] = keyd(kInfKey); out.L[slot] = keyd(kInfKey);
                    }
                }
            }
        }
        // ---- Lambda of the accepted runs, lane j item j, in pipeline order
        __syncwarp();
        const int longest = (int)__reduce_max_sync(kFull, (unsigned)acc_m);
        if (longest) {
            const int slot = (int)(item >> 8), role = (int)((item >> 7) & 1u), g = slot / K;
            const size_t vM = (size_t)acc_v * M;
            const uint16_t *pp = pop.perm + (size_t)g * M + my_off;
            const int16_t *lay = dm.role_search ? so.layers + ((size_t)g * 2 + role) * M + my_off
                                                : out.layers + (size_t)g * M + my_off;
            double lam = 0.0, l[4], t[4];
            int dprev = 0;
            auto fetch = [&](int k0) {                     // four devices' times
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int k = k0 + q;
                    l[q] = t[q] = 0.0;
                    if (k < acc_m) {
                        int dk, nb_;
                        if (D == 1) {
                            const uint32_t x = part[lane * kClaimRow + k];
                            dk = (int)(x & 0xFFFFu);
                            nb_ = (int)(x >> 16);
                        } else {
                            dk = pp[k];
                            nb_ = lay[k];
                        }
                        l[q] = tb.leaf[((vM + dk) * 2 + (k == acc_mu)) * LS + nb_ - 1];
                        if (k > 0) t[q] = tb.tau[(vM + dprev) * M + dk].t;
                        dprev = dk;
                    }
                }
            };
            fetch(0);
            for (int k0 = 0; k0 < longest; k0 += 4) {
                double l0[4], t0[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) { l0[q] = l[q]; t0[q] = t[q]; }
                fetch(k0 + 4);                             // in flight during the additions
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (k0 + q < acc_m) {
                        if (k0 + q == 0) lam = l0[0];
                        else { lam = lam + t0[q]; lam = lam + l0[q]; }
                    }
            }
            if (acc_m) {
                if (dm.role_search) so.L[(size_t)slot * 2 + role] = lam;
                else out.L[slot] = lam;
            }
        }
        __syncwarp();
    }
    st_probes = __reduce_add_sync(kFull, st_probes);
    if (lane == 0 && st_runs) {
        atomicAdd(&out.stats[cls ? kStDpRunsSmall : kStDpRuns], st_runs);
        atomicAdd(&out.stats[kStCells], st_cells);
        atomicAdd(&out.stats[kStProbes], (unsigned long long)st_probes);
    }
}

using OrderKernel = void (*)(Dims, Tables, DevPop, EvalOut, WorkList, const int32_t *, SplitOut, int);

template <int D>
OrderKernel pick(bool off) { return off ? dp_order_kernel<D, true> : dp_order_kernel<D, false>; }

// The kernel of replicas of up to mmax devices: 1, 2, 3, 4 or 8 devices per lane.
OrderKernel order_kernel(int mmax, bool off, int *per_lane)
{
    *per_lane = mmax <= 32 ? 1 : mmax <= 64 ? 2 : mmax <= 96 ? 3 : mmax <= 128 ? 4 : 8;
    switch (*per_lane) {
    case 1: return pick<1>(off);
    case 2: return pick<2>(off);
    case 3: return pick<3>(off);
    case 4: return pick<4>(off);
    default: return pick<8>(off);
    }
}

}  // namespace

size_t dp_order_smem(int mmax, int cls)
{
    int per_lane = 1;
    order_kernel(mmax, false, &per_lane);
    const size_t warp = per_lane > 1 ? 32 * (size_t)per_lane * sizeof(uint16_t) : kClaim * kClaimRow * sizeof(uint32_t);
    return warp * dp_order_warps(cls);
}

cudaError_t dp_order_occupancy(int mmax, int cls, bool off, int *per_sm)
{
    int per_lane = 1;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        per_sm, reinterpret_cast<const void *>(order_kernel(mmax, off, &per_lane)), 32 * dp_order_warps(cls),
        dp_order_smem(mmax, cls));
}

cudaError_t dp_order_launch(int grid, int mmax, int cls, cudaStream_t stream, const Dims &dm, const Tables &tb,
                            const DevPop &pop, const EvalOut &out, const WorkList &wl, const int32_t *slot_off,
                            const SplitOut &so, bool early)
{
    int per_lane = 1;
    const OrderKernel k = order_kernel(mmax, dm.offload != 0, &per_lane);
    return launch_kernel(k, (unsigned)grid, 32 * dp_order_warps(cls), dp_order_smem(mmax, cls), stream, early, dm, tb, pop,
                         out, wl, slot_off, so, cls);
}

}  // namespace e2
