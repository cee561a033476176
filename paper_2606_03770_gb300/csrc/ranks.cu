// ranks.cu -- 32-bit order keys for the DP.
//
// The DP of a variant v compares stage times l_d(n, master) of its devices with
// each other and with the largest link time of a chain.  A stage time x is
// replaced by
//     key(x) = 1 + #{ stage times of the variant below x }      (+inf -> 0xFFFFFFFF)
// and a link time t by #{ stage times <= t }, so that key(x) <= key(t) exactly
// when x <= t, and stage keys keep every comparison and tie of the stage times
// among themselves.  (Two link times are never told apart by anything the DP
// decides: a chain's links bound every master alike.)  A comparison is one
// 32-bit instruction, and a warp's minimum or maximum one reduction.  T and
// Lambda come from the float64 times.
//
// The stage times are sorted once per context, by a bitonic network (strides
// of 2,048 and more in global memory, the rest in shared memory); a redraw of
// the links then only searches each link's place in the sorted list, in the
// kernel that computes the link times (ga.cu).  Ranking links and stages
// together, as before, sorted the link bandwidths and rebuilt both key tables
// at every redraw: 90 us per generation for 128 devices, now 10.
#include "e2ga_internal.cuh"

namespace e2 {

namespace {

constexpr int kLocal = 2048;   // elements sorted per CTA in shared memory

__device__ __forceinline__ void cmpx(uint64_t &a, uint64_t &b, bool up)
{
    if ((a > b) == up) { const uint64_t t = a; a = b; b = t; }
}

// Bitonic stages (k, j) with j < kLocal for every k in [k_lo, k_hi], on
// chunks of kLocal elements in shared memory; blockIdx.y selects the array.
__global__ void __launch_bounds__(1024) bitonic_local(uint64_t *data, size_t stride_arrays, size_t k_lo,
                                                      size_t k_hi)
{
    __shared__ uint64_t s[kLocal];
    uint64_t *a = data + blockIdx.y * stride_arrays + (size_t)blockIdx.x * kLocal;
    const size_t base = (size_t)blockIdx.x * kLocal;
    for (int i = threadIdx.x; i < kLocal; i += blockDim.x) s[i] = a[i];
    __syncthreads();
    for (size_t k = k_lo; k <= k_hi; k <<= 1) {
        for (size_t j = (k >> 1) < (size_t)(kLocal >> 1) ? (k >> 1) : (size_t)(kLocal >> 1); j > 0; j >>= 1) {
            for (int t = threadIdx.x; t < kLocal / 2; t += blockDim.x) {
                const size_t i = 2 * j * (t / j) + (t % j);          // lower index of the pair
                const bool up = ((base + i) & k) == 0;
                cmpx(s[i], s[i + j], up);
            }
            __syncthreads();
        }
    }
    for (int i = threadIdx.x; i < kLocal; i += blockDim.x) a[i] = s[i];
}

// One bitonic stage (k, j) with j >= kLocal, in global memory.
__global__ void bitonic_global(uint64_t *data, size_t stride_arrays, size_t n, size_t k, size_t j)
{
    uint64_t *a = data + blockIdx.y * stride_arrays;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n / 2; t += (size_t)gridDim.x * blockDim.x) {
        const size_t i = 2 * j * (t / j) + (t % j);
        cmpx(a[i], a[i + j], (i & k) == 0);
    }
}

// Keys for the stage-time sort: every finite or infinite l_d(n, master) of
// variant v, padded with +inf up to the power of two.
__global__ void leaf_keys(Dims dm, const double *leaf, uint64_t *keys, size_t cap)
{
    const size_t per = (size_t)dm.M * 2 * dm.N;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < (size_t)dm.V * cap;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int v = (int)(idx / cap);
        const size_t i = idx - (size_t)v * cap;
        uint64_t key = ~0ull;
        if (i < per) {
            const size_t row = i / dm.N, n = i - row * dm.N;           // row = d * 2 + master
            key = dkey(leaf[((size_t)v * dm.M * 2 + row) * dm.LS + n]);
        }
        keys[idx] = key;
    }
}

// Keys of the stage times: leaf_rank[v][d][mf][n].
__global__ void leaf_rank_kernel(Dims dm, const double *leaf, const uint64_t *sorted, size_t cap, uint32_t *leaf_rank)
{
    const size_t n = (size_t)dm.M * 2 * dm.N, per = (size_t)dm.M * 2 * dm.LS, total = (size_t)dm.V * per;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const uint64_t x = dkey(leaf[idx]);
        leaf_rank[idx] = x >= kInfKey ? 0xFFFFFFFFu : 1u + (uint32_t)count_below(sorted + (idx / per) * cap, n, x);
    }
}

inline unsigned grid_for(size_t n, int threads, size_t cap = 152 * 32)
{
    size_t b = (n + threads - 1) / threads;
    if (b > cap) b = cap;
    return (unsigned)(b ? b : 1);
}

// Adds its launches to *launches.
cudaError_t bitonic_sort(uint64_t *data, size_t n_pow2, int arrays, cudaStream_t st, unsigned long long *launches)
{
    // n_pow2 >= kLocal, a power of two
    bitonic_local<<<dim3((unsigned)(n_pow2 / kLocal), arrays), 1024, 0, st>>>(data, n_pow2, 2, kLocal);
    ++*launches;
    for (size_t k = 2 * kLocal; k <= n_pow2; k <<= 1) {
        for (size_t j = k >> 1; j >= (size_t)kLocal; j >>= 1) {
            bitonic_global<<<dim3(grid_for(n_pow2 / 2, 256), arrays), 256, 0, st>>>(data, n_pow2, n_pow2, k, j);
            ++*launches;
        }
        bitonic_local<<<dim3((unsigned)(n_pow2 / kLocal), arrays), 1024, 0, st>>>(data, n_pow2, k, k);
        ++*launches;
    }
    return cudaGetLastError();
}

}  // namespace

size_t rank_pow2(size_t n)
{
    size_t p = kLocal;
    while (p < n) p <<= 1;
    return p;
}

cudaError_t build_stage_keys(const e2_ctx *c)
{
    const size_t cap = rank_pow2((size_t)c->dm.M * 2 * c->dm.N);
    leaf_keys<<<grid_for((size_t)c->dm.V * cap, 256), 256, 0, c->stream>>>(c->dm, c->leaf, c->leaf_sorted, cap);
    ++c->launches;
    const cudaError_t e = bitonic_sort(c->leaf_sorted, cap, c->dm.V, c->stream, &c->launches);
    if (e != cudaSuccess) return e;
    const size_t total = (size_t)c->dm.V * c->dm.M * 2 * c->dm.LS;
    leaf_rank_kernel<<<grid_for(total, 256), 256, 0, c->stream>>>(c->dm, c->leaf, c->leaf_sorted, cap, c->leaf_rank);
    ++c->launches;
    return cudaGetLastError();
}

}  // namespace e2
