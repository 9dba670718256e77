// Output-error-driven clipping factor (Sec. 3.3, Eq. 12):
//   K* = argmin_K sum_{w in W} E_x (w^T x - w~^T x)^2,   w~ = [w]_Q,  Q = K x [-1 : eps_b : 1],
// over the candidate grid K_c = (c+1)/n_cand x max|w| (n_cand = 20: the experiments' grid
// [0.05 : 0.05 : 1] x max|w|), with W one channel (per-channel sets) or the whole layer (one K).
// The quantized weight is s q with s = K / Qmax and q the exact codes of Eq. 8, and its residual
// fmaf(-s, q, w) feeds the output error of Eq. 11.
//
// Three steps, all on the device:
//   1. candidates: one warp per channel takes max|w| (NaN if a weight is non-finite); per-layer
//      sets reduce the channels' maxima in one CTA;
//   2. errors: the CTA-pair tensor-core contraction over the candidates' residuals, written once as
//      fp16 hi/lo planes (output_error_f16.cu; each residual vector scaled by a power of two from
//      the bound max(min(max|w|, s/2), max|w| - Qmax s) on its elements), or,
//      for shared inputs whose rows are not 16-byte multiples, register tiles of 64 residual
//      vectors by 128 calibration rows in fp32 (clip_rows_kernel), or, for per-channel inputs, one
//      CTA per channel and candidate chunk with the residuals in shared memory and threads over
//      the calibration rows;
//   3. argmin: per channel, or per layer over the channel sums (double, channels in order).
#include <math.h>

#include <algorithm>

#include "mpq_internal.cuh"
#include "rounding.cuh"
#include "sm100.cuh"

MPQ_CHECKED_UNIT("clip.cu");

namespace mpq {
namespace {

constexpr int CL_THREADS = 256;
constexpr int CL_CHUNK = 8;   // candidates per CTA in the shared-memory path

__device__ __forceinline__ float candidate_fraction(int c, int n_cand)
{
    return __fdiv_rn((float)(c + 1), (float)n_cand);
}

// One warp per channel: m = max|w| (NaN when a weight is not finite), also into chmax[k] when
// given.  Per channel, the candidate row K_c = f_c m; per layer, m is parked in column 0 for
// clip_layer_kernel.
__global__ void clip_channel_kernel(const float *__restrict__ W, int C, int d, int n_cand, int mode,
                                    float *__restrict__ clip, float *__restrict__ chmax)
{
    const int k = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (k >= C) return;
    const float *w = W + (size_t)k * d;
    float m = 0.0f;
    int bad = 0;
    for (int j = lane; j < d; j += 32) {
        const float v = w[j];
        bad |= !isfinite(v);
        m = fmaxf(m, fabsf(v));
    }
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    }
    if (bad) m = NAN;
    if (chmax && lane == 0) chmax[k] = m;
    if (mode == MPQ_CLIP_PER_CHANNEL) {
        for (int c = lane; c < n_cand; c += 32)
            clip[(size_t)k * n_cand + c] = __fmul_rn(candidate_fraction(c, n_cand), m);
    } else if (lane == 0) {
        clip[(size_t)k * n_cand] = m;
    }
}

// One CTA: the layer's m = max over the channels (NaN if any channel's is), then every row.
__global__ void clip_layer_kernel(int C, int n_cand, float *__restrict__ clip)
{
    __shared__ float wm[32];
    __shared__ int wb[32];
    float m = 0.0f;
    int bad = 0;
    for (int k = threadIdx.x; k < C; k += blockDim.x) {
        const float v = clip[(size_t)k * n_cand];
        bad |= isnan(v);
        m = fmaxf(m, v);
    }
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        wm[warp] = m;
        wb[warp] = bad;
    }
    __syncthreads();   // every read of column 0 is done before the rows are written
    m = 0.0f;
    bad = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
        m = fmaxf(m, wm[i]);
        bad |= wb[i];
    }
    if (bad) m = NAN;
    for (size_t i = threadIdx.x; i < (size_t)C * n_cand; i += blockDim.x)
        clip[i] = __fmul_rn(candidate_fraction((int)(i % n_cand), n_cand), m);
}

// One CTA per (channel, chunk of CL_CHUNK candidates): residuals r_c = fmaf(-s_c, q_c, w) in
// shared memory, threads over the calibration rows, fp32 dot products, squares summed in fp32
// (16-row partial sums, a compensated sum per thread, a tree over the threads).
__global__ void __launch_bounds__(CL_THREADS)
clip_errors_kernel(const float *__restrict__ X, int N, const float *__restrict__ W,
                   int C, int d, int qmax, int n_cand, const float *__restrict__ clip,
                   float *__restrict__ err)
{
    extern __shared__ __align__(16) float R[];   // [CL_CHUNK][d]
    __shared__ float red[CL_THREADS / 32][CL_CHUNK];
    const int k = blockIdx.x, c0 = blockIdx.y * CL_CHUNK;
    const int nc = min(CL_CHUNK, n_cand - c0);
    if (!MPQ_IN(k, C) || !MPQ_CHECK(nc >= 1) || !MPQ_CHECK_SMEM_END(4 * (size_t)nc * d)) return;
    const float qmaxf = (float)qmax;
    const float *w = W + (size_t)k * d;
    for (int i = threadIdx.x; i < nc * d; i += CL_THREADS) {
        const int c = i / d, j = i % d;
        const float s = __fdiv_rn(clip[(size_t)k * n_cand + c0 + c], qmaxf);
        const float v = w[j];
        const float q = s > 0.0f ? copysignf((float)code_mag(fabsf(v), s, qmaxf), v) : 0.0f;
        R[i] = __fmaf_rn(-s, q, v);
    }
    __syncthreads();
    const float *Xk = X + (size_t)k * N * d;
    // all in fp32 (fp64 throughput is a small fraction of fp32's on this part): squares summed over
    // at most 16 rows of a thread, folded into a compensated sum, then a tree over the threads
    float acc[CL_CHUNK], comp[CL_CHUNK], part[CL_CHUNK];
#pragma unroll
    for (int c = 0; c < CL_CHUNK; ++c) {
        acc[c] = 0.0f;
        comp[c] = 0.0f;
        part[c] = 0.0f;
    }
    int rows = 0;
    for (int t = threadIdx.x; t < N; t += CL_THREADS) {
        const float *x = Xk + (size_t)t * d;
        float y[CL_CHUNK];
#pragma unroll
        for (int c = 0; c < CL_CHUNK; ++c) y[c] = 0.0f;
        for (int j = 0; j < d; ++j) {
            const float xv = x[j];
#pragma unroll
            for (int c = 0; c < CL_CHUNK; ++c)
                if (c < nc) y[c] = fmaf(xv, R[c * d + j], y[c]);
        }
#pragma unroll
        for (int c = 0; c < CL_CHUNK; ++c) part[c] = fmaf(y[c], y[c], part[c]);
        if (++rows == 16) {
#pragma unroll
            for (int c = 0; c < CL_CHUNK; ++c) {
                kahan_add(acc[c], comp[c], part[c]);
                part[c] = 0.0f;
            }
            rows = 0;
        }
    }
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < CL_CHUNK; ++c) {
        kahan_add(acc[c], comp[c], part[c]);
        float v = acc[c];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[wp][c] = v;
    }
    __syncthreads();
    if (threadIdx.x < nc) {
        float v[CL_THREADS / 32];
        for (int i = 0; i < CL_THREADS / 32; ++i) v[i] = red[i][threadIdx.x];
        for (int w = CL_THREADS / 64; w > 0; w >>= 1)   // tree over the warps
            for (int i = 0; i < w; ++i) v[i] += v[i + w];
        if (MPQ_IN((size_t)k * n_cand + c0 + threadIdx.x, (size_t)C * n_cand))
            err[(size_t)k * n_cand + c0 + threadIdx.x] = mean_of_sum(v[0], N);
    }
}

// Shared input, rows of any length and alignment: a fp32 contraction of 64 residual vectors (channel,
// candidate) by 16 R calibration rows per CTA, 8 x R products a thread (as 8 x R/2 pairs of rows,
// two fused multiply-adds an instruction), chunks of 16 elements through two shared buffers while
// the next chunk's elements are read into registers.  Residuals are made from W as they are
// stored: about a tenth of the instructions at 128 rows, and no scratch.  Each product sum runs
// over the row in order in one fp32 accumulator (as the thread-per-row kernel's below, whose
// 1e-7 from 64-bit sums the fp16 contraction's truncating accumulators do not reach: 1.5e-6);
// squares are summed 8 at a time, compensated over a thread's row tiles, and in double over the
// threads and over the CTAs of a cluster, which share a vector tile's row tiles.
// Bound by the fp32 pipes: 2048 x 1859, N = 939, 20 candidates 22.7 -> 4.1 ms (35 TFLOP/s);
// 64 x 147, N = 1024 93 -> 42 us.
constexpr int CR_VEC = 64, CR_K = 16, CR_THREADS = 128;
constexpr int CR_LDR = CR_VEC + 4;             // (rows of 16-byte multiples; fewer conflicts)

__device__ __forceinline__ unsigned long long pair2(float a)
{
    unsigned long long v;
    asm("mov.b64 %0, {%1, %1};" : "=l"(v) : "f"(a));
    return v;
}

__device__ __forceinline__ void fma2(unsigned long long &c, unsigned long long a, unsigned long long b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

template <int R>   // 8, 4 or 2
__global__ void __launch_bounds__(CR_THREADS, 3)
clip_rows_kernel(const float *__restrict__ X, int N, const float *__restrict__ W, int C, int d,
                 int qmax, int n_cand, const float *__restrict__ clip, float *__restrict__ err)
{
    constexpr int ROWS = 16 * R, PAIRS = R / 2;
    __shared__ __align__(16) float xs[2][CR_K][ROWS + 4];
    __shared__ __align__(16) float rs[2][CR_K][CR_LDR];
    __shared__ float scale[CR_VEC], inverse[CR_VEC];
    __shared__ int chan[CR_VEC];               // -1: beyond the last vector
    __shared__ double red[2][CR_VEC];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long m0 = (long long)blockIdx.x * CR_VEC, M = (long long)C * n_cand;
    const int rank = (int)blockIdx.y, split = (int)gridDim.y;
    const int n_rt = (N + ROWS - 1) / ROWS, n_ch = (d + CR_K - 1) / CR_K;
    const int rt0 = (int)((long long)n_rt * rank / split);
    const long long total = ((long long)n_rt * (rank + 1) / split - rt0) * n_ch;   // chunks
    const float qmaxf = (float)qmax, qlim = qmaxf + 1.0f;
    const float tband = 0.5f - MPQ_FAST_REL * (qlim + 1.0f);
    if (tid < CR_VEC) {
        const long long m = m0 + tid;
        float s = 0.0f, inv = 0.0f;
        int k = -1;
        if (m < M) {
            k = (int)(m / n_cand);
            s = __fdiv_rn(__ldg(clip + m), qmaxf);
            // the fast codes' bound holds for normal 1/s; NaN marks scales that take the division
            if (s > 0.0f) inv = s > 0x1p-120f && s < 0x1p120f ? __frcp_rn(s) : NAN;
        }
        scale[tid] = s;
        inverse[tid] = inv;
        chan[tid] = k;
    }
    __syncthreads();

    // loads: element lk of the chunk, rows lg + 8 i of X, vectors lg + 8 i
    const int lk = tid & (CR_K - 1), lg = tid / CR_K;
    float xr[ROWS / 8], wr[CR_VEC / 8];
    int c = 0, rt = rt0;                        // chunk and row tile of the next load
    auto load = [&]() {
        const int j = c * CR_K + lk;
        const float *x = X + (size_t)(rt * (long long)ROWS + lg) * d + j;
        const int rows = N - rt * ROWS - lg;
#pragma unroll
        for (int i = 0; i < ROWS / 8; ++i)
            xr[i] = j < d && 8 * i < rows ? __ldg(x + (size_t)(8 * i) * d) : 0.0f;
#pragma unroll
        for (int i = 0; i < CR_VEC / 8; ++i) {
            const int k = chan[lg + 8 * i];
            wr[i] = j < d && k >= 0 ? __ldg(W + (size_t)k * d + j) : 0.0f;
        }
        if (++c == n_ch) {
            c = 0;
            ++rt;
        }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int i = 0; i < ROWS / 8; ++i) xs[b][lk][lg + 8 * i] = xr[i];
#pragma unroll
        for (int i = 0; i < CR_VEC / 8; ++i) {
            const float s = scale[lg + 8 * i], inv = inverse[lg + 8 * i];
            bool unsure = isnan(inv);
            float q = code_signed_fast(wr[i], inv, qmaxf, qlim, tband, unsure);
            if (unsure) q = code_signed_exact(wr[i], s, qmaxf);
            rs[b][lk][lg + 8 * i] = __fmaf_rn(-s, q, wr[i]);
        }
    };

    // products: rows 4 rg + {0..3} and (R = 8) 64 more, or (R = 2) 2 rg + {0, 1}, vectors 4 vg + {0..3} and 32 more
    const int rg = (lane & 7) + 8 * (warp & 1), vg = (lane >> 3) + 4 * (warp >> 1);
    unsigned long long y[8][PAIRS];
    float acc[8], comp[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        acc[v] = 0.0f;
        comp[v] = 0.0f;
#pragma unroll
        for (int r = 0; r < PAIRS; ++r) y[v][r] = 0ull;
    }
    if (total > 0) {
        load();
        store(0);
    }
    __syncthreads();
    int cc = 0;                                 // chunk of the row tile
    for (long long it = 0; it < total; ++it) {
        const int b = (int)(it & 1);
        if (it + 1 < total) load();
#pragma unroll
        for (int k = 0; k < CR_K; ++k) {
            unsigned long long x[PAIRS];
            if (R == 2) {
                x[0] = *reinterpret_cast<const unsigned long long *>(&xs[b][k][2 * rg]);
            } else {
#pragma unroll
                for (int i = 0; i < PAIRS; i += 2) {
                    const ulonglong2 p = *reinterpret_cast<const ulonglong2 *>(&xs[b][k][32 * i + 4 * rg]);
                    x[i] = p.x;
                    x[(i + 1) % PAIRS] = p.y;
                }
            }
            const float4 r0 = *reinterpret_cast<const float4 *>(&rs[b][k][4 * vg]);
            const float4 r1 = *reinterpret_cast<const float4 *>(&rs[b][k][32 + 4 * vg]);
            const float r[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const unsigned long long rr = pair2(r[v]);
#pragma unroll
                for (int i = 0; i < PAIRS; ++i) fma2(y[v][i], x[i], rr);
            }
        }
        if (++cc == n_ch) {                     // the row tile's squares (rows beyond N: y = 0)
            cc = 0;
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                float p = 0.0f;
#pragma unroll
                for (int r = 0; r < PAIRS; ++r) {
                    const float a = __uint_as_float((unsigned)y[v][r]);
                    const float e = __uint_as_float((unsigned)(y[v][r] >> 32));
                    p = fmaf(e, e, fmaf(a, a, p));
                    y[v][r] = 0ull;
                }
                kahan_add(acc[v], comp[v], p);
                if (!isfinite(acc[v])) comp[v] = 0.0f;   // (inf - inf)
            }
        }
        if (it + 1 < total) store(b ^ 1);
        __syncthreads();
    }

    // sums over the 16 threads of a vector, then over the cluster in rank order
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        double s = (double)acc[v] - (double)comp[v];
        for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((lane & 7) == 0) red[warp & 1][4 * vg + (v & 3) + 32 * (v >> 2)] = s;
    }
    __syncthreads();
    if (tid < CR_VEC) red[0][tid] += red[1][tid];
    sm100::cluster_sync();
    if (rank == 0 && tid < CR_VEC && m0 + tid < M && MPQ_IN((size_t)(m0 + tid), (size_t)M)) {
        double s = red[0][tid];
        for (int p = 1; p < split; ++p) s += sm100::ld_dsmem_f64(&red[0][tid], (uint32_t)p);
        err[m0 + tid] = (float)(s / (double)N);
    }
    sm100::cluster_sync();                      // no CTA leaves while its sums are read
}

// Per channel: the lowest c with the smallest err[k][c]; NaN never wins, none finite gives -1.
__global__ void clip_select_channel_kernel(const float *__restrict__ err, int C, int n_cand,
                                           int *__restrict__ best)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= C) return;
    int b = -1;
    float bv = 0.0f;
    for (int c = 0; c < n_cand; ++c) {
        const float v = err[(size_t)k * n_cand + c];
        if (isnan(v)) continue;
        if (b < 0 || v < bv) {
            b = c;
            bv = v;
        }
    }
    best[k] = b;
}

// Per layer (one CTA): lane c sums column c over the channels in order (double); the lowest c with
// the smallest sum goes to every channel.
__global__ void clip_select_layer_kernel(const float *__restrict__ err, int C, int n_cand,
                                         int *__restrict__ best)
{
    __shared__ int pick;
    if (threadIdx.x < 32) {
        const int c = threadIdx.x;
        double e = 0.0;
        if (c < n_cand)
            for (int k = 0; k < C; ++k) e += (double)err[(size_t)k * n_cand + c];
        const bool ok = c < n_cand && !isnan(e);
        int b = -1;
        double bv = 0.0;
        for (int i = 0; i < n_cand; ++i) {   // in candidate order: the lowest index keeps ties
            const double ei = __shfl_sync(0xffffffffu, e, i);
            const int oki = __shfl_sync(0xffffffffu, (int)ok, i);
            if (oki && (b < 0 || ei < bv)) {
                b = i;
                bv = ei;
            }
        }
        if (threadIdx.x == 0) pick = b;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < C; k += blockDim.x) best[k] = pick;
}

}  // namespace

mpq_status launch_clip(const float *X, int N, int groups, const float *W, int C, int d, int qmax,
                       int n_cand, int mode, float *clip, float *err, int *best,
                       cudaStream_t stream)
{
    // the tensor-core path takes all its scratch from the stream-ordered pool before anything is
    // enqueued: channel maxima, then the contraction's (X range and planes, residual planes)
    const bool tc = groups == 1 && output_error_pair_ok(X, W, reinterpret_cast<const int8_t *>(W), d);
    const size_t max_bytes = ((size_t)C * sizeof(float) + 255) / 256 * 256;
    char *scratch = nullptr;
    if (tc) {
        const mpq_status st = pool_scratch(reinterpret_cast<void **>(&scratch),
                                           max_bytes + clip_f16_scratch_bytes(C, N, d, n_cand),
                                           stream);
        if (st != MPQ_OK) return st;
    }
    float *chmax = reinterpret_cast<float *>(scratch);
    const unsigned blocks = (unsigned)(((size_t)C * 32 + CL_THREADS - 1) / CL_THREADS);
    clip_channel_kernel<<<blocks, CL_THREADS, 0, stream>>>(W, C, d, n_cand, mode, clip, chmax);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && mode == MPQ_CLIP_PER_LAYER) {
        clip_layer_kernel<<<1, 1024, 0, stream>>>(C, n_cand, clip);
        e = cudaGetLastError();
    }
    if (tc) {
        mpq_status st = cuda_status(e, "clip candidate kernel launch");
        if (st == MPQ_OK)
            st = launch_clip_f16(X, N, W, clip, chmax, C, d, qmax, n_cand, err, scratch + max_bytes,
                                 stream);
        const cudaError_t ef = cudaFreeAsync(scratch, stream);
        if (st == MPQ_OK) st = cuda_status(ef, "scratch release (cudaFreeAsync)");
        if (st != MPQ_OK) return st;
    } else {
        if (e != cudaSuccess) return cuda_status(e, "clip candidate kernel launch");
        if (groups == 1) {
            // the rows a thread and the split of the row tiles over a cluster's CTAs with the least
            // work on one SM, a chunk costing R products and about 4 more's time for its residuals
            // and the hand-over; ties to the larger split (more warps resident), then the larger
            // R.  100 x 333, N = 100, 10 candidates: 51 us with R = 8 only, 40 so (a CTA per channel and 8
            // candidates, a thread per row: 44); 64 x 147, N = 300, 20: 49, 30 (47).
            const long long tiles = ((long long)C * n_cand + CR_VEC - 1) / CR_VEC;
            const int sms = sm_count();
            int split = 1, rows = 8;
            long long best = -1;
            for (int r = 8; r >= 2; r /= 2) {
                const long long n_rt = (N + 16LL * r - 1) / (16 * r);
                for (int s = 1; s <= 8 && s <= n_rt; ++s) {
                    const long long cost =
                        (tiles * s + sms - 1) / sms * ((n_rt + s - 1) / s) * (r + 4);
                    if (best < 0 || cost < best || (cost == best && r == rows)) {
                        best = cost;
                        split = s;
                        rows = r;
                    }
                }
            }
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)tiles, (unsigned)split, 1);
            cfg.blockDim = dim3(CR_THREADS, 1, 1);
            cfg.stream = stream;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 1;
            attr[0].val.clusterDim.y = (unsigned)split;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            e = cudaLaunchKernelEx(&cfg, rows == 8   ? clip_rows_kernel<8>
                                         : rows == 4 ? clip_rows_kernel<4>
                                                     : clip_rows_kernel<2>, X, N, W, C, d, qmax, n_cand,
                                   (const float *)clip, err);
        } else {
            const size_t smem = (size_t)CL_CHUNK * d * sizeof(float);
            constexpr int fixed = CL_THREADS / 32 * CL_CHUNK * (int)sizeof(float);
            if ((long long)smem > max_smem_optin() - fixed) {
                set_error("clip search with d = %d needs %zu bytes of shared memory", d, smem);
                return MPQ_ERR_UNSUPPORTED;
            }
            static std::atomic<int> limit[kMaxDevices];
            e = allow_smem(reinterpret_cast<const void *>(clip_errors_kernel), limit, smem);
            if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute");
            const dim3 grid((unsigned)C, (unsigned)((n_cand + CL_CHUNK - 1) / CL_CHUNK));
            clip_errors_kernel<<<grid, CL_THREADS, smem, stream>>>(X, N, W, C, d, qmax, n_cand, clip,
                                                                  err);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return cuda_status(e, "clip error kernel launch");
    }

    if (mode == MPQ_CLIP_PER_CHANNEL)
        clip_select_channel_kernel<<<(C + CL_THREADS - 1) / CL_THREADS, CL_THREADS, 0, stream>>>(
            err, C, n_cand, best);
    else
        clip_select_layer_kernel<<<1, 1024, 0, stream>>>(err, C, n_cand, best);
    e = cudaGetLastError();
    return cuda_status(e, "clip select kernel launch");
}

}  // namespace mpq
