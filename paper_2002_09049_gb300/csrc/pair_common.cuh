// Pieces shared by the CTA-pair output-error kernels (Sec. 3.3, Eq. 11 and 12): the power-of-two
// scaling and fp16 hi/lo split of the contraction's operands, and tile-map encoding for the TMA
// copies.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <math.h>
#include <stdint.h>

#include "mpq.h"

namespace mpq {

// fp16 operands: exponent e with m * 2^e in [2^14, 2^15) for the largest magnitude m of a residual
// vector or of X, so that the vector's hi and lo halves are normal fp16 numbers down to 2^-7 of its
// largest element (and nothing overflows).  0 for m = 0, NaN or inf (which then propagate); capped
// at 126 so that 2^e stays a normal float (only vectors below 2^-111 are scaled less).
__device__ __forceinline__ int f16_scale_exp(float m)
{
    if (!(m > 0.0f) || !isfinite(m)) return 0;
    int E;
    (void)frexpf(m, &E);              // m = f 2^E, f in [0.5, 1)
    return min(15 - E, 126);
}

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

__device__ __forceinline__ double pow2d(int e)
{
    return __longlong_as_double((long long)(1023 + e) << 52);
}

// x * 2^e (exact) split into fp16 hi + lo: hi = fl16(x), lo = fl16(x - hi) (x - hi is exact in fp32).
__device__ __forceinline__ void split_f16x2(float a, float b, uint32_t &hi, uint32_t &lo)
{
    const __half2 h = __floats2half2_rn(a, b);
    const float2 hf = __half22float2(h);
    const __half2 l = __floats2half2_rn(__fsub_rn(a, hf.x), __fsub_rn(b, hf.y));
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}

// Host: launch attribute of a kernel that starts with griddep_wait and directly follows, on its stream,
// a kernel of the same call.
inline cudaLaunchAttribute after_previous_kernel()
{
    cudaLaunchAttribute a = {};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    return a;
}

// Host: tile map over a row-major tensor (dims[0] contiguous, byte strides for dims 1..), zero
// fill out of range, the given shared-memory swizzle.  False if the driver entry point is missing
// or rejects the arguments.
bool encode_tile_map(CUtensorMap *m, CUtensorMapDataType type, int rank, const void *base,
                     const cuuint64_t *dims, const cuuint64_t *strides, const cuuint32_t *box,
                     CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_NONE);

// Copies of W and the codes with rows of dp elements, a multiple of 16 (W NULL: none).
struct PadRows {
    float *W;        // [C][dp]
    int8_t *codes;   // [k_max][C][dp]
    int dp;
};

// Rows that a tile copy can address: whole multiples of 16 bytes in every array, aligned bases.
__host__ __device__ inline bool tile_rows_ok(const float *X, const float *W, const int8_t *codes,
                                             int d)
{
    return (d & 15) == 0 && (((uintptr_t)X | (uintptr_t)W | (uintptr_t)codes) & 15) == 0;
}

// Host: max|X| (float bits) into range[0], zeroed first, and n_count zeros into count.
mpq_status launch_x_range(const float *X, int N, int d, unsigned *range, unsigned *count,
                          int n_count, cudaStream_t stream);

// Host: X * 2^e (e from xrange[0]) split into the fp16 hi and lo planes xs ([2][N][dp], dp = d
// rounded up to 16, the rest of a row zero), and the errors of a layer's slow channels
// (slow_channels.cuh; C = 0: none).
struct SlowLayer;
cudaError_t launch_x_split(const float *X, int N, int d, const unsigned *xrange, uint16_t *xs,
                           const SlowLayer &slow, cudaStream_t stream);

// Host: the output error of the greedy points (output_error_chain.cu), with its ranges ready on
// `stream` (xrange[0] = max|X|, vrange = max|r| per residual vector, float bits); nearest: the codes are
// nearest values (else slow channels are left out, or with xs NULL computed here); xs: the split X
// planes, or NULL (the contraction then splits X itself); pad: padded copies of W and the codes,
// or none (with xs, W and codes are then rows a tile copy can address); part: part_bytes of 256-byte aligned
// scratch for partial sums, at least chain_count_bytes(tiles) and that much of it zeroed on
// `stream` (chain_scratch_bytes(tiles, chain_max_gang(N)) is all it can use).
mpq_status launch_output_error_chain(const float *X, int N, const float *W, const int8_t *codes,
                                     const float *scales, int C, int d, int k_max, float *err,
                                     const unsigned *xrange, const unsigned *vrange,
                                     bool nearest, const uint16_t *xs, const PadRows &pad, void *part,
                                     size_t part_bytes, cudaStream_t stream);
int chain_tiles(int C, int k_max);   // channel tiles of a CTA pair
size_t chain_count_bytes(int tiles);
size_t chain_scratch_bytes(int tiles, int gang);
int chain_max_gang(int N);

}  // namespace mpq
