// Output errors (Sec. 3.3, Eq. 11) of channels that the chain of points (output_error_chain.cu) cannot
// compute: those whose residuals grow, as no nearest codes (Eq. 8) make them, or whose scales end in
// NaN.  Plain fp32 dot products with the residuals themselves, a fallback that takes hundreds of
// microseconds a channel.  Layers with every channel so (256 x 4096, N = 2048, k_max = 8 / 1024 x 1024,
// N = 1024, k_max = 4 / 64 x 576, N = 512, k_max = 4): 68 / 15 / 0.43 ms by blocks of the pass that splits
// X, 345 / 37 / 11 ms by the pair that has the channel in the contraction (a thread a calibration row,
// as it was first: 515 / 65 / 21 ms); nearest codes 0.12 / 0.046 / 0.024 ms.
#pragma once

#include <math.h>

#include "mpq_internal.cuh"
#include "sm100.cuh"

namespace mpq {

// Everything a slow channel is computed from; vrange: max|r| per residual vector, float bits.
struct SlowLayer {
    const float *X, *W;
    const int8_t *codes;
    const float *scales;
    const unsigned *vrange;
    float *err;
    int C, N, d, K;
};

// The growth of a residual's largest magnitude that a point may make: K of them stay within a factor
// of 4.
__host__ __device__ constexpr float growth_limit(int K)
{
    constexpr float root[17] = {4.0f,    4.0f,    2.0f,    1.5874f, 1.4142f, 1.3195f,
                                1.2599f, 1.2190f, 1.1892f, 1.1665f, 1.1487f, 1.1343f,
                                1.1225f, 1.1125f, 1.1041f, 1.0968f, 1.0905f};
    return root[K < 16 ? K : 16];
}

// Whether the chain cannot take a point: the largest magnitudes before and after it, its scale.  (A
// channel with a non-finite weight has only NaN scales and errors, and stays with the chain.)
__device__ __forceinline__ bool slow_point(float vr, float vn, float s, float limit)
{
    return vn > limit * vr || fabsf(s) > 4.0f * vr || (isnan(s) && vr < INFINITY);
}

__device__ __forceinline__ bool is_slow(const SlowLayer &l, int k)
{
    const float *s = l.scales + (size_t)k * l.K;
    const unsigned *v = l.vrange + (size_t)k * (l.K + 1);
    const float limit = growth_limit(l.K);
    bool slow = false;
#pragma unroll 8
    for (int n = 0; n < l.K; ++n)
        slow |= slow_point(__uint_as_float(sm100::ld_after_wait(v + n)),
                           __uint_as_float(sm100::ld_after_wait(v + n + 1)), __ldg(s + n), limit);
    return slow;
}

// Error n of slow channel k by a warp: S_ROWS calibration rows at a time, an element of X a lane (whole
// lines), the residual's element regenerated for them.  Every lane sums its elements in order, the
// lanes are added as a tree, squares in double in row order.  No shared memory and no barriers: the
// kernels that call it share SMs with contractions that leave none.
constexpr int S_ROWS = 8, S_WARPS = 8;   // (warps: those that take a channel's errors in turn)

static __device__ __noinline__ void slow_error(const SlowLayer &l, int k, int n, int lane)
{
    const int N = l.N, d = l.d;
    const float *w = l.W + (size_t)k * d, *s = l.scales + (size_t)k * l.K;
    const int8_t *codes = l.codes + (size_t)k * d;
    const size_t plane = (size_t)l.C * d;
    double acc = 0.0;
#pragma unroll 1
    for (int t0 = 0; t0 < N; t0 += S_ROWS) {
        float y[S_ROWS];
#pragma unroll
        for (int u = 0; u < S_ROWS; ++u) y[u] = 0.0f;
        const float *x0 = l.X + (size_t)t0 * d;
#pragma unroll 2
        for (int j = lane; j < d; j += 32) {
            float x[S_ROWS];
#pragma unroll
            for (int u = 0; u < S_ROWS; ++u) x[u] = __ldg(x0 + min(u, N - 1 - t0) * d + j);
            float r = __ldg(w + j);
#pragma unroll 4
            for (int i = 0; i < n; ++i)
                r = __fmaf_rn(-__ldg(s + i), (float)__ldg(codes + i * plane + j), r);
#pragma unroll
            for (int u = 0; u < S_ROWS; ++u) y[u] = fmaf(x[u], r, y[u]);
        }
#pragma unroll
        for (int u = 0; u < S_ROWS; ++u) {
            float v = y[u];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (t0 + u < N) acc += (double)v * (double)v;
        }
    }
    const size_t at = (size_t)k * (l.K + 1) + n;
    if (lane == 0 && MPQ_IN(at, (size_t)l.C * (l.K + 1))) l.err[at] = (float)(acc / (double)N);
}

}  // namespace mpq
