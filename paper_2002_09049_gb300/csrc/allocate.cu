// Per-channel point counts from the output-error table (Sec. 3.3, Algorithm 2).
//
// Budget mode.  The sequential rule -- hand each extra point to the channel whose next point has
// the largest gain e_k(n_k) - e_k(n_k+1), lowest k on ties, stop when no gain is positive -- is
// computed as one selection.  For channel k and n = 2..k_max let
//   gain_k(n) = e_k(n-1) - e_k(n)      (fp32 subtraction; NaN reads as -inf)
//   p_k(n)    = min_{2<=m<=n} gain_k(m) (prefix minimum)
// and order the pairs (k, n) by (p desc, k asc, n asc).  The sequential loop takes exactly the
// first `extra` pairs of this order that have p > 0: a channel's (n+1)-th gain becomes its head
// only after the n-th was taken, its priority never exceeds the priorities before it, and a head
// at or above every other head is taken next -- so both rules visit the pairs in the same order.
// Each pair becomes one unique 64-bit key (~bits(p) in the high word, k*(k_max-1)+(n-2) in the
// low word); a selection finds the extra-th smallest key T, and n_k = 1 + #{n : key(k, n) <= T}.
// The high words live in shared memory when they fit (they are recomputed from the error table on
// every pass otherwise); no global scratch is used.
//
// One CTA selects, so latency is what counts: barriers, and shared-memory atomics that meet on one
// address.  The keys' own range is cut into 2,048 equal buckets (8-bit digits from the top, tried
// first, put all keys into the few buckets of their common exponents: 40 us for 960 channels x 8
// points), the bucket that holds the wanted rank is cut again if it has more than SEL_LIST keys,
// and the rank inside it comes from counting.  960 x 8: 7.4 us; 64 x 4 keys: 9.1 -> 5.7 us.
#include <math.h>

#include "mpq_internal.cuh"

MPQ_CHECKED_UNIT("allocate.cu");

namespace mpq {
namespace {

constexpr int AB_THREADS = 1024;
constexpr unsigned NO_KEY = ~0u;   // the high word of no key: a selectable p is above 0

// The keys' high words of channel k for n = 2..k_max, in n order, via callback (NO_KEY: no gain).
template <typename F>
__device__ __forceinline__ void channel_keys(const float *__restrict__ err, int k, int k_max, F f)
{
    const float *e = err + (size_t)k * (k_max + 1);
    float p = INFINITY;
    float prev = e[1];
#pragma unroll 4
    for (int n = 2; n <= k_max; ++n) {
        const float cur = e[n];
        float g = __fsub_rn(prev, cur);
        if (isnan(g)) g = -INFINITY;
        p = fminf(p, g);
        prev = cur;
        f(n, p > 0.0f ? ~__float_as_uint(p) : NO_KEY);
    }
}

constexpr int KEY_CACHE = 49152;   // keys' high words held in shared memory (192 KB) when they fit
constexpr int SEL_BUCKETS = 2 * AB_THREADS;
constexpr int SEL_LIST = AB_THREADS;

// One CTA of AB_THREADS threads allocates one layer; skeys: dynamic shared memory for its keys.
__device__ __forceinline__ void allocate_budget_cta(const float *__restrict__ err, int C, int k_max,
                                                    long long extra, int *__restrict__ npoints,
                                                    int *__restrict__ points_used, bool cached,
                                                    unsigned *skeys)
{
    __shared__ unsigned hist[SEL_BUCKETS];
    __shared__ unsigned long long list[SEL_LIST];
    __shared__ unsigned long long w_total[32], s_T;
    __shared__ unsigned w_min[32], w_max[32], w_sum[32];
    __shared__ long long s_rem;
    __shared__ unsigned s_bucket, s_count;
    __shared__ int s_nlist, s_used;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int KM1 = k_max - 1;
    // the cached keys within the launch's shared memory, else read again from err
    if (cached && !MPQ_CHECK_SMEM_END(4 * (size_t)C * KM1)) cached = false;

    if (tid == 0) {
        s_used = 0;
        s_nlist = 0;
    }
    hist[tid] = 0u;
    hist[tid + AB_THREADS] = 0u;
    // the keys; how many there are, and their range
    unsigned long long mine = 0;
    unsigned kmin = NO_KEY, kmax = 0u;
    for (int k = tid; k < C; k += AB_THREADS)
        channel_keys(err, k, k_max, [&](int n, unsigned hi) {
            if (cached) skeys[(size_t)k * KM1 + (n - 2)] = hi;
            if (hi != NO_KEY) {
                ++mine;
                kmin = min(kmin, hi);
                kmax = max(kmax, hi);
            }
        });
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) {
        w_total[warp] = mine;
        w_min[warp] = kmin;
        w_max[warp] = kmax;
    }
    __syncthreads();
    mine = w_total[lane];
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    kmin = __reduce_min_sync(0xffffffffu, w_min[lane]);
    kmax = __reduce_max_sync(0xffffffffu, w_max[lane]);
    const long long total = (long long)mine;
    const long long take = extra < total ? extra : total;

    // visit every selectable key
    auto for_keys = [&](auto f) {
        if (cached) {
            const int nk = C * KM1;
            for (int i = tid; i < nk; i += AB_THREADS) {
                const unsigned hi = skeys[i];
                if (hi != NO_KEY) f(((unsigned long long)hi << 32) | (unsigned)i);
            }
        } else {
            for (int k = tid; k < C; k += AB_THREADS)
                channel_keys(err, k, k_max, [&](int n, unsigned hi) {
                    if (hi != NO_KEY)
                        f(((unsigned long long)hi << 32) |
                          (unsigned)((unsigned long long)k * KM1 + (n - 2)));
                });
        }
    };

    unsigned long long T = 0;   // selected = keys <= T (when take > 0)
    if (take > 0 && take == total) {
        T = ~0ULL;
    } else if (take > 0) {
        long long rem = take;   // 1-based rank of the wanted key among the `count` in [base, base + width]
        unsigned long long count = (unsigned long long)total;
        unsigned long long base = (unsigned long long)kmin << 32;
        unsigned long long width = ((unsigned long long)(kmax - kmin) << 32) | 0xFFFFFFFFull;
        while (count > SEL_LIST) {
            // (hist is clear) buckets of 2^shift: at most SEL_BUCKETS of them
            const int shift = max(0, 64 - __clzll((long long)width) - 11);
            for_keys([&](unsigned long long key) {
                if (key - base <= width) atomicAdd(&hist[(unsigned)((key - base) >> shift)], 1u);
            });
            __syncthreads();
            // the bucket that holds the rem-th key
            const unsigned c0 = hist[2 * tid], c1 = hist[2 * tid + 1];
            unsigned incl = c0 + c1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) w_sum[warp] = incl;
            __syncthreads();
            const unsigned long long before =
                __reduce_add_sync(0xffffffffu, lane < warp ? w_sum[lane] : 0u) +
                (unsigned long long)(incl - c0 - c1);
            const long long want = rem - (long long)before;
            if (want > 0 && want <= (long long)(c0 + c1)) {
                const bool second = want > (long long)c0;
                s_bucket = 2 * tid + (second ? 1 : 0);
                s_count = second ? c1 : c0;
                s_rem = want - (second ? (long long)c0 : 0);
            }
            hist[2 * tid] = 0u;
            hist[2 * tid + 1] = 0u;
            __syncthreads();
            rem = s_rem;
            count = s_count;
            base += (unsigned long long)s_bucket << shift;
            width = shift > 0 ? (1ULL << shift) - 1 : 0;
        }
        // the keys left, and the one with rem - 1 smaller ones
        for_keys([&](unsigned long long key) {
            if (key - base <= width) {
                const int at = atomicAdd(&s_nlist, 1);
                if (MPQ_IN(at, SEL_LIST)) list[at] = key;
            }
        });
        __syncthreads();
        const int m = (int)count;
        if (tid < m) {
            const unsigned long long key = list[tid];
            int smaller = 0;
#pragma unroll 8
            for (int i = 0; i < m; ++i) smaller += list[i] < key;
            if (smaller == (int)(rem - 1)) s_T = key;
        }
        __syncthreads();
        T = s_T;
    }

    // n_k = 1 + number of selected keys of channel k (a prefix n = 2..n_k, since p is monotone)
    int used = 0;
    for (int k = tid; k < C; k += AB_THREADS) {
        int n_k = 1;
        if (take > 0) {
            const unsigned long long first = (unsigned long long)k * KM1;
            auto selected = [&](int n, unsigned hi) {
                n_k += hi != NO_KEY &&
                       (((unsigned long long)hi << 32) | (unsigned)(first + (n - 2))) <= T;
            };
            if (cached) {
                for (int n = 2; n <= k_max; ++n) selected(n, skeys[first + (n - 2)]);
            } else {
                channel_keys(err, k, k_max, selected);
            }
        }
        npoints[k] = n_k;
        used += n_k;
    }
    if (points_used) {
        used = __reduce_add_sync(0xffffffffu, used);
        if (lane == 0) atomicAdd(&s_used, used);   // integer sum: order-free
        __syncthreads();
        if (tid == 0) *points_used = s_used;
    }
}

__global__ void __launch_bounds__(AB_THREADS)
allocate_budget_kernel(const float *__restrict__ err, int C, int k_max, long long extra,
                       int *__restrict__ npoints, int *__restrict__ points_used, bool cached)
{
    extern __shared__ unsigned skeys[];   // [C * (k_max - 1)] when cached
    allocate_budget_cta(err, C, k_max, extra, npoints, points_used, cached, skeys);
}

// Threshold mode (Algorithm 2 as printed) for one layer by one CTA, the total by a block sum.
__device__ __forceinline__ void allocate_threshold_cta(const float *__restrict__ err, int C,
                                                       int k_max, double eps,
                                                       int *__restrict__ npoints,
                                                       int *__restrict__ points_used)
{
    __shared__ int s_used;
    if (threadIdx.x == 0) s_used = 0;
    __syncthreads();
    int used = 0;
    for (int k = threadIdx.x; k < C; k += blockDim.x) {
        const float *e = err + (size_t)k * (k_max + 1);
        int n = k_max;
        for (int m = 1; m <= k_max; ++m) {
            if ((double)e[m] < eps) {
                n = m;
                break;
            }
        }
        npoints[k] = n;
        used += n;
    }
    if (points_used) {
        for (int o = 16; o > 0; o >>= 1) used += __shfl_xor_sync(0xffffffffu, used, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(&s_used, used);   // integer sum: order-free
        __syncthreads();
        if (threadIdx.x == 0) *points_used = s_used;
    }
}

// Several layers in one launch: CTA b allocates layer order[b] (largest first, so the longest
// CTAs start first).
struct AllocBatch {
    const float *err[MPQ_MAX_BATCH];
    int *npoints[MPQ_MAX_BATCH];
    int *points_used[MPQ_MAX_BATCH];
    double param[MPQ_MAX_BATCH];     // threshold mode: eps
    long long extra[MPQ_MAX_BATCH];  // budget mode
    int C[MPQ_MAX_BATCH];
    unsigned char cached[MPQ_MAX_BATCH];
    unsigned char order[MPQ_MAX_BATCH];
};

__global__ void __launch_bounds__(AB_THREADS)
allocate_batch_kernel(const __grid_constant__ AllocBatch b, int k_max, int mode)
{
    extern __shared__ unsigned skeys[];
    if (!MPQ_IN(blockIdx.x, MPQ_MAX_BATCH) || !MPQ_IN(b.order[blockIdx.x], MPQ_MAX_BATCH)) return;
    const int l = b.order[blockIdx.x];
    if (mode == MPQ_ALLOC_BUDGET)
        allocate_budget_cta(b.err[l], b.C[l], k_max, b.extra[l], b.npoints[l], b.points_used[l],
                            b.cached[l] != 0, skeys);
    else
        allocate_threshold_cta(b.err[l], b.C[l], k_max, b.param[l], b.npoints[l],
                               b.points_used[l]);
}

constexpr int AT_THREADS = 256;

__global__ void __launch_bounds__(AT_THREADS)
allocate_threshold_kernel(const float *__restrict__ err, int C, int k_max, double eps,
                          int *__restrict__ npoints, int *__restrict__ points_used)
{
    int used = 0;
    for (int k = blockIdx.x * AT_THREADS + threadIdx.x; k < C; k += gridDim.x * AT_THREADS) {
        const float *e = err + (size_t)k * (k_max + 1);
        int n = k_max;
        for (int m = 1; m <= k_max; ++m) {
            if ((double)e[m] < eps) {
                n = m;
                break;
            }
        }
        npoints[k] = n;
        used += n;
    }
    if (points_used) {
        for (int o = 16; o > 0; o >>= 1) used += __shfl_xor_sync(0xffffffffu, used, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(points_used, used);  // integer sum: order-free
    }
}

}  // namespace

mpq_status launch_allocate_budget(const float *err, int C, int k_max, long long extra,
                                  int *npoints, int *points_used, cudaStream_t stream)
{
    const long long nkeys = (long long)C * (k_max - 1);
    const bool cached = nkeys <= KEY_CACHE;
    const size_t smem = cached ? (size_t)nkeys * sizeof(unsigned) : 0;
    static std::atomic<int> limit[kMaxDevices];
    const cudaError_t e = allow_smem(reinterpret_cast<const void *>(allocate_budget_kernel), limit, smem);
    if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute");
    allocate_budget_kernel<<<1, AB_THREADS, smem, stream>>>(err, C, k_max, extra, npoints,
                                                            points_used, cached);
    return cuda_status(cudaGetLastError(), "allocation kernel launch");
}

mpq_status launch_allocate_batch(int n, const float *const *err, const int *C, int k_max,
                                 int mode, const long long *extra, const double *eps,
                                 int *const *npoints, int *const *points_used, cudaStream_t stream)
{
    AllocBatch b;
    size_t smem = 0;
    int m = 0;
    for (int l = 0; l < n; ++l) {
        if (C[l] == 0) continue;   // nothing to allocate (points_used zeroed by the caller)
        b.err[l] = err[l];
        b.npoints[l] = npoints[l];
        b.points_used[l] = points_used ? points_used[l] : nullptr;
        b.C[l] = C[l];
        b.extra[l] = extra ? extra[l] : 0;
        b.param[l] = eps ? eps[l] : 0.0;
        const long long nkeys = (long long)C[l] * (k_max - 1);
        const bool cached = mode == MPQ_ALLOC_BUDGET && nkeys <= KEY_CACHE;
        b.cached[l] = cached;
        if (cached && (size_t)nkeys * sizeof(unsigned) > smem) smem = (size_t)nkeys * sizeof(unsigned);
        b.order[m++] = (unsigned char)l;
    }
    if (m == 0) return MPQ_OK;
    // largest layers first
    for (int i = 1; i < m; ++i)
        for (int j = i; j > 0 && b.C[b.order[j]] > b.C[b.order[j - 1]]; --j) {
            const unsigned char t = b.order[j];
            b.order[j] = b.order[j - 1];
            b.order[j - 1] = t;
        }
    static std::atomic<int> limit[kMaxDevices];
    const cudaError_t e = allow_smem(reinterpret_cast<const void *>(allocate_batch_kernel), limit, smem);
    if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute");
    allocate_batch_kernel<<<m, AB_THREADS, smem, stream>>>(b, k_max, mode);
    return cuda_status(cudaGetLastError(), "batched allocation kernel launch");
}

mpq_status launch_allocate_threshold(const float *err, int C, int k_max, double eps,
                                     int *npoints, int *points_used, cudaStream_t stream)
{
    if (points_used) {
        cudaError_t e = cudaMemsetAsync(points_used, 0, sizeof(int), stream);
        if (e != cudaSuccess) return cuda_status(e, "cudaMemsetAsync");
    }
    int blocks = (C + AT_THREADS - 1) / AT_THREADS;
    const int cap = sm_count() * 4;
    if (blocks > cap) blocks = cap;
    allocate_threshold_kernel<<<blocks, AT_THREADS, 0, stream>>>(err, C, k_max, eps, npoints,
                                                                  points_used);
    return cuda_status(cudaGetLastError(), "allocation kernel launch");
}

}  // namespace mpq
