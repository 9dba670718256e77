// Output error of every channel for every point count (Sec. 3.3, Eq. 11):
//   err[k][n] = (1/N) sum_t (x_t . r_{k,n+1})^2,  n = 0..k_max,
// with the residuals r_{k,n+1} regenerated on chip from W, codes and scales by the recursion of
// Eq. 7 (never materialised in global memory).
//
// Shared input (groups = 1) is a dense contraction and runs on the tensor cores: the CTA pairs of
// output_error_chain.cu (through output_error_pair.cu) where rows are whole aligned 16 bytes
// (tile_rows_ok) or long and many enough for padded copies (output_error_rows_ok), else, and where
// the pool has no room for those copies, the single-CTA kernel (output_error_tc.cu).  Per-channel
// input (groups = C, depthwise convolution, d = 9): one CTA per channel, its k_max+1 residuals in
// shared memory, the channel's own rows of X staged through shared memory with coalesced reads
// (each read once), threads over the rows; rows of up to 32 elements two a thread.
#include <math.h>

#include <algorithm>

#include "mpq_internal.cuh"
#include "sm100.cuh"

MPQ_CHECKED_UNIT("output_error.cu");

namespace mpq {
namespace {

constexpr int GR_THREADS = 256;

// Short rows (every depthwise kernel in use: 9, 25, 49): two rows a thread, so that the k_max+1
// residuals of an element, read as 16-byte words, serve both, and chunks of X copied with
// cp.async into one of two buffers while the other is used.  Bound by the latency of the first
// chunk, then by X's bytes: 960 x 9, k_max = 8, N = 1024 13.0 us (35 MB: 5 us), 1536 x 25 45 us
// (157 MB: 23 us); the kernel below, one row a thread and a residual per load, is bound by its
// shared-memory reads: 19.4 and 85 us.
constexpr int SR_THREADS = 128, SR_ROWS = 2;
// longer rows come with too few CTAs an SM (two chunks of 256 rows each: 49 elements 23 us either
// way at 512 channels, N = 512, k_max = 4), and even ones with bank conflicts for both rows
constexpr int SR_MAX_D = 32;
constexpr int SR_CHUNK = SR_ROWS * SR_THREADS;    // rows of a chunk

template <int KP1>
__global__ void __launch_bounds__(SR_THREADS, KP1 <= 9 ? 7 : 4)
output_error_short_rows_kernel(const float *__restrict__ X, int N, const float *__restrict__ W,
                               const int8_t *__restrict__ codes, const float *__restrict__ scales,
                               int C, int d, float *__restrict__ err)
{
    constexpr int K = KP1 - 1, KP = (KP1 + 3) / 4 * 4;
    constexpr int chunk = SR_CHUNK;
    extern __shared__ __align__(16) float xs[];       // two buffers of chunk * d + 4 floats
    __shared__ __align__(16) float rsh[SR_MAX_D][KP];
    __shared__ float red[SR_THREADS / 32][KP1];
    const int k = blockIdx.x, tid = threadIdx.x;
    const int buffer = chunk * d + 4;
    if (!MPQ_IN(k, C) || !MPQ_CHECK(d <= SR_MAX_D) || !MPQ_CHECK_SMEM_END(8 * (size_t)buffer)) return;
    const uintptr_t x0 = (uintptr_t)X, xk = x0 + (size_t)k * N * d * 4;
    const int n_chunks = (N + chunk - 1) / chunk;
    // chunk c into buffer c & 1: the aligned 16 bytes that hold it (none read beyond its end or,
    // where X itself starts off a boundary, before X)
    auto copy = [&](int c) {
        const uintptr_t at = xk + (size_t)c * chunk * d * 4;
        const int nr = min(chunk, N - c * chunk), off = (int)(at & 15);
        const int bytes = off + nr * d * 4;
        const uint32_t dst = sm100::smem_u32(xs + (c & 1) * buffer);
        const uintptr_t from = at - (unsigned)off;
        for (int b = 16 * tid; b < bytes; b += 16 * SR_THREADS) {
            if (from + (unsigned)b < x0) {
                for (int o = off; o < min(16, bytes); o += 4)
                    sm100::cp_async4(dst + b + o, reinterpret_cast<const void *>(from + b + o), 4u);
            } else {
                sm100::cp_async16(dst + b, reinterpret_cast<const void *>(from + b),
                                  (uint32_t)min(16, bytes - b));
            }
        }
        sm100::cp_async_commit();
    };
    copy(0);
    if (n_chunks > 1) copy(1);

    for (int j = tid; j < d; j += SR_THREADS) {
        const size_t at = (size_t)k * d + j, plane = (size_t)C * d;
        float q[K];
#pragma unroll
        for (int n = 0; n < K; ++n) q[n] = (float)__ldg(codes + n * plane + at);
        float r = __ldg(W + at);
        rsh[j][0] = r;
#pragma unroll
        for (int n = 0; n < K; ++n) {
            r = __fmaf_rn(-__ldg(scales + (size_t)k * K + n), q[n], r);
            rsh[j][n + 1] = r;
        }
#pragma unroll
        for (int n = KP1; n < KP; ++n) rsh[j][n] = 0.0f;
    }

    // squares as in the kernel below: a thread's rows compensated, then a tree over the threads
    float acc[KP1], comp[KP1];
#pragma unroll
    for (int n = 0; n < KP1; ++n) {
        acc[n] = 0.0f;
        comp[n] = 0.0f;
    }
    for (int c = 0; c < n_chunks; ++c) {
        if (c + 1 < n_chunks)
            sm100::cp_async_wait<1>();
        else
            sm100::cp_async_wait<0>();
        __syncthreads();   // this chunk (and the residuals) from every thread
        const int nr = min(chunk, N - c * chunk);
        const float *xc = xs + (c & 1) * buffer + ((xk + (size_t)c * chunk * d * 4) & 15) / 4;
        for (int t = tid; t < nr; t += SR_ROWS * SR_THREADS) {
            const bool two = t + SR_THREADS < nr;
            const float *xa = xc + t * d, *xb = two ? xa + SR_THREADS * d : xa;
            float y[KP], z[KP];
#pragma unroll
            for (int n = 0; n < KP; ++n) {
                y[n] = 0.0f;
                z[n] = 0.0f;
            }
#pragma unroll 3
            for (int j = 0; j < d; ++j) {
                const float a = xa[j], b = xb[j];
#pragma unroll
                for (int n = 0; n < KP; n += 4) {
                    const float4 r = *reinterpret_cast<const float4 *>(&rsh[j][n]);
                    y[n] = fmaf(a, r.x, y[n]);
                    z[n] = fmaf(b, r.x, z[n]);
                    if (n + 1 < KP1) {
                        y[n + 1] = fmaf(a, r.y, y[n + 1]);
                        z[n + 1] = fmaf(b, r.y, z[n + 1]);
                    }
                    if (n + 2 < KP1) {
                        y[n + 2] = fmaf(a, r.z, y[n + 2]);
                        z[n + 2] = fmaf(b, r.z, z[n + 2]);
                    }
                    if (n + 3 < KP1) {
                        y[n + 3] = fmaf(a, r.w, y[n + 3]);
                        z[n + 3] = fmaf(b, r.w, z[n + 3]);
                    }
                }
            }
#pragma unroll
            for (int n = 0; n < KP1; ++n) {
                const float p = __fmul_rn(y[n], y[n]);
                kahan_add(acc[n], comp[n], two ? fmaf(z[n], z[n], p) : p);
            }
        }
        if (c + 2 < n_chunks) {
            __syncthreads();   // this buffer is no longer read
            copy(c + 2);
        }
    }
    const int lane = tid & 31, wp = tid >> 5;
#pragma unroll
    for (int n = 0; n < KP1; ++n) {
        kahan_add(acc[n], comp[n], 0.0f);
        float v = acc[n];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[wp][n] = v;
    }
    __syncthreads();
    if (tid < KP1 && MPQ_IN((size_t)k * KP1 + tid, (size_t)C * KP1))
        err[(size_t)k * KP1 + tid] =
            mean_of_sum((red[0][tid] + red[2][tid]) + (red[1][tid] + red[3][tid]), N);
}

constexpr int GR_X_FLOATS = 4096;                 // 16 KB of calibration rows staged at a time

template <int KP1>
__global__ void __launch_bounds__(GR_THREADS)
output_error_grouped_kernel(const float *__restrict__ X, int N, const float *__restrict__ W,
                            const int8_t *__restrict__ codes, const float *__restrict__ scales,
                            int C, int d, float *__restrict__ err)
{
    extern __shared__ __align__(16) float Rsh[];   // [KP1][d], then rows of X [GR_X_FLOATS]
    __shared__ float red[GR_THREADS / 32][KP1];
    const int k = blockIdx.x;
    const int tid = threadIdx.x;
    const int k_max = KP1 - 1;
    const size_t plane = (size_t)C * d;
    // the residual rows and one staged chunk of X within the launch's shared memory
    if (!MPQ_IN(k, C) || !MPQ_CHECK(d <= GR_X_FLOATS) ||
        !MPQ_CHECK_SMEM_END(4 * ((size_t)((KP1 * d + 3) & ~3) + GR_X_FLOATS)))
        return;

    for (int j = tid; j < d; j += GR_THREADS) {
        float r = W[(size_t)k * d + j];
        Rsh[j] = r;
        for (int i = 0; i < k_max; ++i) {
            r = __fmaf_rn(-scales[(size_t)k * k_max + i], (float)codes[(size_t)i * plane + (size_t)k * d + j], r);
            Rsh[(size_t)(i + 1) * d + j] = r;
        }
    }
    __syncthreads();

    const float *Xk = X + (size_t)k * N * d;
    float *Xsh = Rsh + ((KP1 * d + 3) & ~3);
    const int chunk = GR_X_FLOATS / d;               // rows per staged chunk (d <= GR_X_FLOATS)
    // All in fp32 (the part's fp64 rate is a small fraction of its fp32 rate, and fp64 work per
    // row, or fp64 warp reductions, bound the kernel): squares summed over at most ERR_FOLD rows of
    // a thread, folded into a compensated (Kahan) sum, then a tree over the threads and one
    // division -- relative error below (ERR_FOLD + 2 + 8 + 1) * 2^-24 in all.
    constexpr int ERR_FOLD = 16;
    float acc[KP1], comp[KP1], part[KP1];
#pragma unroll
    for (int n = 0; n < KP1; ++n) {
        acc[n] = 0.0f;
        comp[n] = 0.0f;
        part[n] = 0.0f;
    }
    int rows = 0;
    for (int t0 = 0; t0 < N; t0 += chunk) {
        // the channel's next rows of X, read with consecutive threads on consecutive words
        const int nr = min(chunk, N - t0);
        __syncthreads();   // the previous chunk is no longer read
        for (int i = tid; i < nr * d; i += GR_THREADS) Xsh[i] = Xk[(size_t)t0 * d + i];
        __syncthreads();
        for (int t = tid; t < nr; t += GR_THREADS) {
            float y[KP1];
#pragma unroll
            for (int n = 0; n < KP1; ++n) y[n] = 0.0f;
            const float *x = Xsh + t * d;
            for (int j = 0; j < d; ++j) {
                const float xv = x[j];
#pragma unroll
                for (int n = 0; n < KP1; ++n) y[n] = fmaf(xv, Rsh[n * d + j], y[n]);
            }
#pragma unroll
            for (int n = 0; n < KP1; ++n) part[n] = fmaf(y[n], y[n], part[n]);
            if (++rows == ERR_FOLD) {
#pragma unroll
                for (int n = 0; n < KP1; ++n) {
                    kahan_add(acc[n], comp[n], part[n]);
                    part[n] = 0.0f;
                }
                rows = 0;
            }
        }
    }
    const int lane = tid & 31, wp = tid >> 5;
#pragma unroll
    for (int n = 0; n < KP1; ++n) {
        kahan_add(acc[n], comp[n], part[n]);
        float v = acc[n];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[wp][n] = v;
    }
    __syncthreads();
    if (tid < KP1) {
        float v[GR_THREADS / 32];
        for (int i = 0; i < GR_THREADS / 32; ++i) v[i] = red[i][tid];
        for (int w = GR_THREADS / 64; w > 0; w >>= 1)   // tree over the warps
            for (int i = 0; i < w; ++i) v[i] += v[i + w];
        if (MPQ_IN((size_t)k * KP1 + tid, (size_t)C * KP1))
            err[(size_t)k * KP1 + tid] = mean_of_sum(v[0], N);
    }
}

template <int KP1>
mpq_status launch_grouped(const float *X, int N, const float *W, const int8_t *codes,
                          const float *scales, int C, int d, float *err, cudaStream_t stream)
{
    if (d <= SR_MAX_D) {
        const int bytes = 2 * (SR_CHUNK * d + 4) * (int)sizeof(float);   // 66 KB at most
        static std::atomic<int> limit[kMaxDevices];
        const cudaError_t e = allow_smem(
            reinterpret_cast<const void *>(output_error_short_rows_kernel<KP1>), limit, bytes);
        if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute");
        output_error_short_rows_kernel<KP1><<<C, SR_THREADS, bytes, stream>>>(X, N, W, codes, scales, C,
                                                                             d, err);
        return cuda_status(cudaGetLastError(), "grouped output-error kernel launch");
    }
    const size_t smem = ((size_t)(KP1 * d + 3) / 4 * 4 + GR_X_FLOATS) * sizeof(float);
    if (d > GR_X_FLOATS || (long long)smem > max_smem_optin()) {
        set_error("groups = C with d = %d and k_max = %d needs %zu bytes of shared memory", d,
                  KP1 - 1, smem);
        return MPQ_ERR_UNSUPPORTED;
    }
    static std::atomic<int> limit[kMaxDevices];
    cudaError_t e = allow_smem(reinterpret_cast<const void *>(output_error_grouped_kernel<KP1>), limit,
                               smem);
    if (e == cudaSuccess) {
        output_error_grouped_kernel<KP1><<<C, GR_THREADS, smem, stream>>>(X, N, W, codes, scales,
                                                                          C, d, err);
        e = cudaGetLastError();
    }
    return cuda_status(e, "grouped output-error kernel launch");
}

}  // namespace

size_t output_error_scratch_words(const float *X, int N, int groups, const float *W,
                                  const int8_t *codes, int C, int d, int k_max)
{
    return (groups == 1 && (output_error_pair_ok(X, W, codes, d) ||
                            output_error_rows_ok(N, codes, C, d, k_max)))
               ? 1 + (size_t)C * (k_max + 1)
               : 0;
}

mpq_status launch_output_error(const float *X, int N, int groups, const float *W,
                               const int8_t *codes, const float *scales, int C, int d, int k_max,
                               float *err, cudaStream_t stream, unsigned *range,
                               const float *rmax)
{
    if (groups == 1) {
        if (output_error_pair_ok(X, W, codes, d))
            return launch_output_error_pair(X, N, W, codes, scales, C, d, k_max, err, stream,
                                            range, rmax);
        if (output_error_rows_ok(N, codes, C, d, k_max)) {
            const mpq_status st = launch_output_error_pair(X, N, W, codes, scales, C, d, k_max, err,
                                                           stream, range, rmax);
            if (st != MPQ_ERR_NOMEM) return st;   // nothing enqueued: the kernel without scratch
            clear_error();
        }
        return launch_output_error_tc(X, N, W, codes, scales, C, d, k_max, err, stream);
    }
    switch (k_max + 1) {
#define MPQ_CASE(n) \
    case n: return launch_grouped<n>(X, N, W, codes, scales, C, d, err, stream);
        MPQ_CASE(2) MPQ_CASE(3) MPQ_CASE(4) MPQ_CASE(5) MPQ_CASE(6) MPQ_CASE(7) MPQ_CASE(8)
        MPQ_CASE(9) MPQ_CASE(10) MPQ_CASE(11) MPQ_CASE(12) MPQ_CASE(13) MPQ_CASE(14) MPQ_CASE(15)
        MPQ_CASE(16) MPQ_CASE(17)
#undef MPQ_CASE
    }
    set_error("k_max = %d unsupported", k_max);
    return MPQ_ERR_UNSUPPORTED;
}

}  // namespace mpq
