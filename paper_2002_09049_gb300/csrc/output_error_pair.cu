// Output error (Sec. 3.3, Eq. 11) on the tensor cores: the operand ranges, the scratch and the
// dispatch of output_error_chain.cu's contraction, and the host helpers it shares with the clipping
// search (tile maps, stream-ordered scratch).
//
// The contraction scales each operand by a power of two, so it needs max|X| and max|r| of every
// residual vector.  The greedy search hands the latter over (rmax); without it pair_range_kernel
// regenerates the residuals and measures them.  With pooled scratch, X is split ahead into fp16
// planes; the entry point with a fixed range table lets the contraction's producers split it.
//
// Tile copies want rows of whole 16 bytes.  Other rows (d not a multiple of 16, or buffers off a
// 16-byte boundary) go through copies of W and the codes with padded rows, made by blocks of the
// range pass (the planes of X are padded anyway); with fixed scratch the contraction gathers them
// itself.  The padding is zeros, which add nothing to any product.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <math.h>

#include <algorithm>
#include <atomic>

#include "mpq_internal.cuh"
#include "pair_common.cuh"
#include "slow_channels.cuh"
#include "sm100.cuh"

MPQ_CHECKED_UNIT("output_error_pair.cu");

namespace mpq {
namespace {

__device__ __forceinline__ float max_abs4(float4 v)
{
    return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
}

// Ranges for the fp16 operand scales, folded with atomicMax into a zeroed range[] (float bits of
// non-negative values order like unsigned integers): blocks [0, xb) take max|X| into range[0], four
// independent 16-byte loads in flight per thread; blocks [xb, xb + cb) give each channel `split`
// warps, each over a 1/split share of the row, for max_j |r_{k,n+1,j}| of every residual vector
// (the same fp32 recursion of Eq. 7 as the contraction's producers) into
// range[1 + k (k_max + 1) + n]; the blocks from xb + cb on copy W and the codes to rows of dp
// elements (pad), a warp per row.
template <int KP1>
__device__ __forceinline__ void range_step(float4 r, const int8_t *__restrict__ codes, size_t plane,
                                           size_t row, int j, const float (&sc)[KP1 > 1 ? KP1 - 1 : 1],
                                           float (&mx)[KP1])
{
    mx[0] = fmaxf(mx[0], max_abs4(r));
#pragma unroll
    for (int n = 0; n < KP1 - 1; ++n) {
        const char4 q = __ldg(reinterpret_cast<const char4 *>(codes + n * plane + row) + j);
        r.x = __fmaf_rn(-sc[n], (float)q.x, r.x);
        r.y = __fmaf_rn(-sc[n], (float)q.y, r.y);
        r.z = __fmaf_rn(-sc[n], (float)q.z, r.z);
        r.w = __fmaf_rn(-sc[n], (float)q.w, r.w);
        mx[n + 1] = fmaxf(mx[n + 1], max_abs4(r));
    }
}

template <int KP1>
__global__ void __launch_bounds__(256)
pair_range_kernel(const float *__restrict__ X, long long nx, int xb, int cb,
                  const float *__restrict__ W, const int8_t *__restrict__ codes,
                  const float *__restrict__ scales, int C, int d, int split,
                  unsigned *__restrict__ range, unsigned *__restrict__ count, int n_count,
                  const PadRows pad)
{
    constexpr int K = KP1 - 1;
    sm100::griddep_launch();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n_count; i += gridDim.x * 256) count[i] = 0u;
    if ((int)blockIdx.x < xb) {
        float m = 0.0f;
        const long long stride = (long long)xb * blockDim.x;
        long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        // elements before the first 16-byte boundary and after the last one, then the rest
        const long long head = min(nx, (long long)((0u - ((unsigned)(uintptr_t)X >> 2)) & 3u));
        const long long nx4 = (nx - head) / 4, tail = head + 4 * nx4;
        if (i < head) m = fabsf(__ldg(X + i));
        if (i < nx - tail) m = fmaxf(m, fabsf(__ldg(X + tail + i)));
        const float4 *x4 = reinterpret_cast<const float4 *>(X + head);
        for (; i + 3 * stride < nx4; i += 4 * stride) {
            const float4 a = __ldg(x4 + i), b = __ldg(x4 + i + stride);
            const float4 c = __ldg(x4 + i + 2 * stride), e = __ldg(x4 + i + 3 * stride);
            m = fmaxf(m, fmaxf(fmaxf(max_abs4(a), max_abs4(b)), fmaxf(max_abs4(c), max_abs4(e))));
        }
        for (; i < nx4; i += stride) m = fmaxf(m, max_abs4(__ldg(x4 + i)));
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) atomicMax(range, __float_as_uint(m));
        return;
    }
    if ((int)blockIdx.x >= xb + cb) {
        // rows 0 .. C - 1 of the copy are W's, row C (n + 1) + k is point n's codes of channel k
        const long long row = (long long)((int)blockIdx.x - xb - cb) * 8 + warp;
        if (row >= (long long)C * KP1) return;
        if (row < C) {
            const float *src = W + row * d;
            float *dst = pad.W + row * pad.dp;
#pragma unroll 4
            for (int j = lane; j < pad.dp; j += 32) dst[j] = j < d ? __ldg(src + j) : 0.0f;
        } else {
            const int8_t *src = codes + (row - C) * d;
            char4 *dst = reinterpret_cast<char4 *>(pad.codes + (row - C) * pad.dp);
#pragma unroll 2
            for (int j = 4 * lane; j < pad.dp; j += 128) {
                char4 q;
                q.x = j < d ? __ldg(src + j) : (int8_t)0;
                q.y = j + 1 < d ? __ldg(src + j + 1) : (int8_t)0;
                q.z = j + 2 < d ? __ldg(src + j + 2) : (int8_t)0;
                q.w = j + 3 < d ? __ldg(src + j + 3) : (int8_t)0;
                dst[j >> 2] = q;
            }
        }
        return;
    }
    const int gw = ((int)blockIdx.x - xb) * 8 + warp;
    const int k = gw / split, part = gw - k * split;
    if (k >= C) return;
    float sc[K > 0 ? K : 1], mx[KP1];
#pragma unroll
    for (int n = 0; n < K; ++n) sc[n] = __ldg(scales + (size_t)k * K + n);
#pragma unroll
    for (int n = 0; n < KP1; ++n) mx[n] = 0.0f;
    const size_t plane = (size_t)C * d, row = (size_t)k * d;
    const int step = 32 * split;
    int j = part * 32 + lane;
    // 16-byte row loads and 4-byte code loads need d % 4 == 0 and aligned bases
    if ((d & 3) == 0 && ((uintptr_t)W & 15) == 0 && ((uintptr_t)codes & 3) == 0) {
        const float4 *w4 = reinterpret_cast<const float4 *>(W + row);
        const int d4 = d / 4;
        for (; j + step < d4; j += 2 * step) {      // two rows' worth of loads in flight
            const float4 a = __ldg(w4 + j), b = __ldg(w4 + j + step);
            range_step<KP1>(a, codes, plane, row, j, sc, mx);
            range_step<KP1>(b, codes, plane, row, j + step, sc, mx);
        }
        if (j < d4) range_step<KP1>(__ldg(w4 + j), codes, plane, row, j, sc, mx);
    } else {
#pragma unroll 2
        for (; j < d; j += step) {
            float r = __ldg(W + row + j);
            mx[0] = fmaxf(mx[0], fabsf(r));
#pragma unroll
            for (int n = 0; n < K; ++n) {
                r = __fmaf_rn(-sc[n], (float)__ldg(codes + n * plane + row + j), r);
                mx[n + 1] = fmaxf(mx[n + 1], fabsf(r));
            }
        }
    }
#pragma unroll
    for (int n = 0; n < KP1; ++n) {
        float m = mx[n];
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0 && MPQ_IN((size_t)k * KP1 + n, (size_t)C * KP1))
            atomicMax(range + 1 + (size_t)k * KP1 + n, __float_as_uint(m));
    }
}

// The range pre-pass into `range` (zeroed here): max|X| into range[0] and, with `residuals`, max|r|
// of every residual vector into range[1 + k (k_max+1) + n]; the contraction's counters zeroed
// (count, nullable); W and codes copied to padded rows (pad.W nullable).
template <int KP1>
cudaError_t launch_ranges(const float *X, int N, const float *W, const int8_t *codes,
                          const float *scales, int C, int d, bool residuals, unsigned *range,
                          unsigned *count, int n_count, const PadRows &pad, cudaStream_t stream)
{
    const size_t words = residuals ? 1 + (size_t)C * KP1 : 1;
    const long long nx = (long long)N * d;
    const int xb = (int)std::min<long long>(std::max(1LL, (nx / 4 + 1023) / 1024), 4LL * sm_count());
    const int rsplit = std::min(8, std::max(1, (d / 4 + 255) / 256));   // >= 8 loads per lane
    const long long cb = residuals ? ((long long)C * rsplit + 7) / 8 : 0;
    const long long pb = pad.W ? ((long long)C * KP1 + 7) / 8 : 0;
    cudaError_t e = cudaMemsetAsync(range, 0, words * sizeof(unsigned), stream);
    if (e != cudaSuccess) return e;
    pair_range_kernel<KP1><<<(unsigned)(xb + cb + pb), 256, 0, stream>>>(
        X, nx, xb, (int)cb, W, codes, scales, C, d, rsplit, range, count, n_count, pad);
    return cudaGetLastError();
}

// Ranges, split X planes (pooled scratch only: ext_range NULL) and the contraction, with the range
// table, the partial sums and the planes in one block.  ext_range: the caller's fixed scratch
// (the range table, then CHAIN_FIXED_SCRATCH bytes after MPQ_NOALLOC_RANGE_WORDS words).
template <int KP1>
mpq_status launch_pair(const float *X, int N, const float *W, const int8_t *codes,
                       const float *scales, int C, int d, float *err, cudaStream_t stream,
                       unsigned *ext_range, const float *rmax)
{
    unsigned *range = ext_range;
    char *part = nullptr;
    uint16_t *xs = nullptr;
    const int tiles = chain_tiles(C, KP1 - 1);
    const int dp = (d + 15) / 16 * 16;
    const bool copies = !output_error_pair_ok(X, W, codes, d) && !ext_range;   // padded rows
    PadRows pad = {nullptr, nullptr, dp};
    size_t part_bytes = CHAIN_FIXED_SCRATCH;
    if (ext_range) {
        part = reinterpret_cast<char *>(ext_range + MPQ_NOALLOC_RANGE_WORDS);
    } else {
        const size_t words = rmax ? 1 : 1 + (size_t)C * KP1;
        const size_t range_bytes = (words * sizeof(unsigned) + 255) / 256 * 256;
        void *scratch = nullptr;
        // no more for partial sums than the fixed scratch holds: both entry points then take the
        // same schedule, and so the same order of sums
        part_bytes = std::max(chain_count_bytes(tiles),
                              std::min(chain_scratch_bytes(tiles, chain_max_gang(N)),
                                       (size_t)CHAIN_FIXED_SCRATCH));
        const size_t plane_bytes = (size_t)N * dp * 2 * sizeof(uint16_t);
        const size_t w_bytes = copies ? (size_t)C * dp * sizeof(float) : 0;
        const size_t q_bytes = copies ? (size_t)C * dp * (KP1 - 1) : 0;
        const mpq_status st = pool_scratch(
            &scratch, range_bytes + part_bytes + plane_bytes + w_bytes + q_bytes, stream);
        if (st != MPQ_OK) return st;
        range = static_cast<unsigned *>(scratch);
        part = static_cast<char *>(scratch) + range_bytes;
        xs = reinterpret_cast<uint16_t *>(part + part_bytes);
        if (copies) {   // (each part a multiple of 16 bytes)
            pad.W = reinterpret_cast<float *>(part + part_bytes + plane_bytes);
            pad.codes = reinterpret_cast<int8_t *>(part + part_bytes + plane_bytes + w_bytes);
        }
    }
    mpq_status r = cuda_status(
        launch_ranges<KP1>(X, N, W, codes, scales, C, d, rmax == nullptr, range,
                           reinterpret_cast<unsigned *>(part), 2 * tiles, pad, stream),
        "output-error range pre-pass");
    const unsigned *vr = rmax ? reinterpret_cast<const unsigned *>(rmax) : range + 1;
    if (r == MPQ_OK && xs) {
        const SlowLayer slow = {X, W, codes, scales, vr, err, rmax ? 0 : C, N, d, KP1 - 1};
        r = cuda_status(launch_x_split(X, N, d, range, xs, slow, stream), "X split kernel launch");
    }
    if (r == MPQ_OK)
        r = launch_output_error_chain(X, N, W, codes, scales, C, d, KP1 - 1, err, range, vr,
                                      rmax != nullptr, xs, pad, part, part_bytes, stream);
    if (!ext_range) {
        const cudaError_t ef = cudaFreeAsync(range, stream);
        if (r == MPQ_OK) r = cuda_status(ef, "scratch release (cudaFreeAsync)");
    }
    return r;
}

}  // namespace

namespace {
PFN_cuTensorMapEncodeTiled_v12000 tile_map_encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        return (PFN_cuTensorMapEncodeTiled_v12000) nullptr;
    }();
    return fn;
}
}  // namespace

bool encode_tile_map(CUtensorMap *m, CUtensorMapDataType type, int rank, const void *base,
                     const cuuint64_t *dims, const cuuint64_t *strides, const cuuint32_t *box,
                     CUtensorMapSwizzle swizzle)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = tile_map_encoder();
    if (!enc) return false;
    const cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, type, (cuuint32_t)rank, const_cast<void *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Scratch (the fp16 contraction's range table, the adaptive grid's event lists) comes from the device's stream-ordered pool (allocated and
// freed on the call's stream, so concurrent calls on other streams never share it; inside a CUDA
// graph capture these become the graph's own allocation nodes).  Freed blocks stay cached in the
// pool instead of going back to the driver at every synchronisation (set on the first call made
// outside a stream capture, where a pool attribute may not be changed).
mpq_status pool_scratch(void **p, size_t bytes, cudaStream_t stream)
{
    static std::atomic<int> pool_set{0};
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusActive;
    if (cudaStreamIsCapturing(stream, &cs) != cudaSuccess) {
        (void)cudaGetLastError();
        cs = cudaStreamCaptureStatusActive;
    }
    if (cs == cudaStreamCaptureStatusNone && !pool_set.exchange(1)) {
        int dev = 0;
        cudaMemPool_t pool;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
            uint64_t keep = UINT64_MAX;
            (void)cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        }
        (void)cudaGetLastError();
    }
    const cudaError_t e = cudaMallocAsync(p, bytes, stream);
    if (e == cudaErrorMemoryAllocation) {
        (void)cudaGetLastError();
        set_error("no %zu bytes of scratch in the stream-ordered pool", bytes);
        return MPQ_ERR_NOMEM;
    }
    return cuda_status(e, "scratch allocation (cudaMallocAsync)");
}

// Other rows: the chain through padded copies or the gather, or the single-CTA tf32 kernel.  Both
// entry points take the same side, so that they give the same errors bit for bit: the gather
// wants 4-byte aligned codes and its range table, and the lines are drawn where it, the slower of
// the two, breaks even.  us, tf32 -> padded copies / gather:
//   short rows (the chain is four launches): 64 x 147, k_max = 4, N = 256 28 -> 24 / 30;
//     64 x 201 35 -> 24 / 34; 512 x 601 91 -> 28 / 63; 5245 x 1859, k_max = 5, N = 939 2313 -> 229 / 1120;
//   a channel tile that is hardly filled: 64 x 301, k_max = 1, N = 1024 30 -> 27 / 38; 8 x 301,
//     k_max = 4 33 -> 26 / 36; 8 x 601 57 -> 26 / 55; 16 x 4607, k_max = 8, N = 64 556 -> 69 / 349;
//   half of the rows idle, over several rounds of channel tiles: 4096 x 601, k_max = 4, N = 64
//     90 -> 42 / 108, N = 256 167 -> 44 / 108; one round: 512 x 601, N = 64 88 -> 29 / 63.
bool output_error_rows_ok(int N, const int8_t *codes, int C, int d, int k_max)
{
    const long long rows = (long long)C * (k_max + 2);   // operand rows; a pair's tile holds 256
    return ((uintptr_t)codes & 3) == 0 &&
           1 + (size_t)C * (k_max + 1) <= (size_t)MPQ_NOALLOC_RANGE_WORDS && d >= 192 &&
           (rows >= 256 || (k_max >= 4 && d >= 600)) &&
           (N > 128 || 2 * chain_tiles(C, k_max) <= sm_count());
}

bool output_error_pair_ok(const float *X, const float *W, const int8_t *codes, int d)
{
    return tile_rows_ok(X, W, codes, d);
}

mpq_status launch_output_error_pair(const float *X, int N, const float *W, const int8_t *codes,
                                    const float *scales, int C, int d, int k_max, float *err,
                                    cudaStream_t stream, unsigned *range, const float *rmax)
{
    switch (k_max + 1) {
#define MPQ_CASE(n) \
    case n: return launch_pair<n>(X, N, W, codes, scales, C, d, err, stream, range, rmax);
        MPQ_CASE(2) MPQ_CASE(3) MPQ_CASE(4) MPQ_CASE(5) MPQ_CASE(6) MPQ_CASE(7) MPQ_CASE(8)
        MPQ_CASE(9) MPQ_CASE(10) MPQ_CASE(11) MPQ_CASE(12) MPQ_CASE(13) MPQ_CASE(14) MPQ_CASE(15)
        MPQ_CASE(16) MPQ_CASE(17)
#undef MPQ_CASE
    }
    set_error("k_max = %d unsupported", k_max);
    return MPQ_ERR_UNSUPPORTED;
}

mpq_status launch_x_range(const float *X, int N, int d, unsigned *range, unsigned *count,
                          int n_count, cudaStream_t stream)
{
    return cuda_status(launch_ranges<2>(X, N, nullptr, nullptr, nullptr, 0, d, false, range,
                                        count, n_count, PadRows{nullptr, nullptr, 0}, stream),
                       "X range pass");
}

}  // namespace mpq
