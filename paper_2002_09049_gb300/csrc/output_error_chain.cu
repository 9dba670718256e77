// Output error (Sec. 3.3, Eq. 11) of the greedy residuals on the tensor cores:
//   err[k][n] = (1/N) sum_t (x_t . r_{k,n+1})^2,  n = 0..k_max,
// from the points themselves.  By Eq. 7, r_{n+1} = r_n - s_n q_n, so with P_i = x . q_i
//   x . r_{n} = x . r_{n+1} + s_n P_n,
// a chain that starts at the last residual and adds one point at a time.  The codes are small
// integers, exact in fp16 as they are: a channel's operand rows are its k_max code rows and the
// last residual's fp16 hi and lo halves (k_max + 2 rows), each multiplied with X's hi and lo halves
// -- 2 (k_max + 2) row passes where k_max + 1 residual vectors of hi/lo halves take 3 (k_max + 1)
// (hi*hi, hi*lo, lo*hi): 20 against 27 at k_max = 8, 12 against 15 at k_max = 4.
//
// Precision.  Codes are exact, X and the last residual carry 22 significant bits (scaled by powers
// of two that put their largest element in [2^14, 2^15), as fp16 hi + lo; the residual's lo times
// X's lo is kept too).  Codes of Eq. 8 are nearest values, so no element of a residual grows
// (|r_{n+1}| <= |r_n|, |s_n q_n| <= 2 |r_n|): the chain adds terms of the size of its result and
// loses nothing.  fp32 accumulation restarts every 256 elements of d (the tensor core's
// accumulation truncates) and the epilogue adds the segments into fp32 running sums.  Every vector
// has its own power of two 2^e_n (from its largest magnitude): the chain runs on
// y_n 2^e_n = y_{n+1} 2^{e_{n+1}} * 2^{e_n - e_{n+1}} + (s_n 2^e_n) P_n, so neither the values nor
// their squares leave fp32's range before the exact rescaling in double at the end.
// Codes that are not nearest values (a caller's own) can make a residual grow, and the chain then ends in
// differences: where a later residual's largest magnitude is g times an earlier one's, that one's
// error is g times as far from 64-bit sums (4e-7 g; the contraction of residual vectors: 1.5e-6).  A
// channel that can reach g = 4, whose scale exceeds four times its residual, or whose scales end in NaN
// (a refused step of the adaptive grid: the errors before it are wanted) is computed by plain fp32
// sums over its residuals instead (slow_channels.cuh): by blocks of the pass that splits X, or here
// with RAWX, which has no such pass.  Where the caller has the ranges from the greedy search, whose
// codes are nearest values, no channel is looked at.
//
// Layout.  Two CTAs on neighbouring SMs (a cluster) issue MMAs of M = 256 calibration rows by
// N = 256 operand rows: each CTA holds 128 calibration rows (hi and lo tiles) and 128 operand rows
// (whole channels), and receives its 128 calibration rows by all 256 operand rows in its tensor
// memory.  A thread of the epilogue holds one calibration row (TMEM lane) and 128 operand rows
// (columns), so a channel's chain runs inside a thread.
//
// Schedule.  One resident pair per two SMs.  Either `gang` neighbouring pairs share the row tiles of a
// channel tile and go through the same range of channel tiles, so its W and codes are read from
// memory once for all of them (the pairs of a gang run at about the same pace); or every pair takes
// an equal contiguous run of the (channel tile, row tile) units (gang 0), where that leaves less on
// the busiest pair.  Where several pairs have a part of a channel tile, each leaves its sums in
// global scratch and the last one to arrive adds them in pair order (nobody waits).  Measured on an
// 11008 x 4096 layer (N = 2048, k_max = 8): contiguous runs 2.18 ms (each pair reads its W and codes
// again for every row tile), gangs of four 2.08 ms; row tiles split over clusters of 2, 4 or 8 CTAs
// 2.4 ms (whole waves of clusters, which do not fill the GPU's SM groups).  On 2009 x 432 (N = 636,
// k_max = 8; 3.3 units a pair) gangs leave 6 units on a pair, contiguous runs 4.
//
// What bounds it: with the operand rows not written the same layer takes 2.02 ms, with W and codes
// from one place of memory as well 1.77 ms, which is the MMAs alone (8 per step, 147 cycles each).
// Shared memory is the co-bound (about 1,050 wavefronts a step against 1,180 cycles of MMAs). The
// three-pass contraction of residual vectors took 2.69 ms (12 MMAs a step, 14 channels a CTA for
// 12), and its errors were 2 to 4 times as far from 64-bit sums (1.5e-6 against 4e-7).
//
// Warps: 0-5 producers (operand rows from W, codes and scales), 6 tile copies, 7 the MMA issuer
// (lane 0 of the even CTA), 8-15 the epilogue (lane quarter warp % 4, column half).  Steps of 64
// elements: X tiles land straight in their slots (split ahead into fp16 planes), W and codes in a
// ring that the producers read.  RAWX (the entry point with fixed scratch): X lands unsplit in that
// ring, and the producers and, between their folds, the epilogue warps split it; same operands, same
// MMAs in the same order, so the results are bit-identical.  Every wait is bounded; on a timeout the kernel records
// MPQ_TIMEOUT_OUTPUT_ERROR, waits for what it issued, and the outputs read NaN.
#include <cuda.h>
#include <cuda_fp16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <atomic>

#include "mpq_internal.cuh"
#include "pair_common.cuh"
#include "slow_channels.cuh"
#include "sm100.cuh"
#include "tf32_operands.cuh"
#include "waits.cuh"

MPQ_CHECKED_UNIT("output_error_chain.cu");

namespace mpq {
namespace {

using namespace sm100;

constexpr int E_VEC = 128;                 // operand rows per CTA (half of the UMMA's N)
constexpr int E_ROWS = 128;                // calibration rows per CTA (half of its M, TMEM lanes)
constexpr int E_M = 2 * E_ROWS;            // calibration rows per pair row tile
constexpr int E_N = 2 * E_VEC;
constexpr int E_KS = 64;                   // elements per step: one 128-byte fp16 row
constexpr int E_SEG = 4;                   // steps per accumulation segment (256 elements)
constexpr int E_PROD_WARPS = 6;
constexpr int E_PT = E_PROD_WARPS * 32;    // producer threads
constexpr int E_COPY_WARP = 6;
constexpr int E_MMA_WARP = 7;
constexpr int E_EPI_WARP0 = 8;             // a multiple of 4: warp % 4 is the TMEM lane quarter
constexpr int E_EPI_WARPS = 8;
constexpr int E_THREADS = 512;
// RAWX: X items of a step split by the epilogue warps (11008 x 4096 3.79 ms, 512 x 4608 237 us; none:
// 4.07 and 271, 6 * 256: 4.20 and 209)
constexpr int E_X_EPI = 4 * 256;
// registers per thread after setmaxnreg: warpgroups 0-1 and 2-3 (epilogue); together exactly what
// the launch holds (512 threads x 128).  With many points the producers bound a step as much as the
// MMAs do, and get what the epilogue's sums leave: k_max = 8, 11008 x 4096 2.12 ms with 80 and 176,
// 2.065 with 96 and 160; 2048 x 2048, N = 1024 k_max = 16 246 and 212 us, k_max = 4 88 and 90.  RAWX
// has the epilogue split X as well.
template <int K, bool RAWX>
struct ERegs {
    static constexpr int LOW = RAWX || K <= 4 ? 80 : 96, HIGH = 256 - LOW;
    static_assert(256 * LOW + 256 * HIGH == E_THREADS * 128, "register split");
};
constexpr int E_TILE = 128 * 128;          // 16 KB: 128 rows of 128 bytes (128-byte swizzle)
constexpr int E_XSET = 2 * E_TILE;         // hi and lo tiles of X
constexpr int E_MAX_STAGES = 3;            // operand-row tiles
constexpr int E_MAX_XSLOTS = 4;
constexpr int E_MAX_RAW = 4;
constexpr uint32_t E_TMEM_COLS = 512;
constexpr int E_MAX_PAIRS = 128;           // resident CTA pairs of a launch, at most
constexpr int E_MAX_GANG = 8;              // pairs that have a part of a channel tile, at most
// what the end of a channel tile costs its pair, and leaving its sums to other pairs as well, in
// steps of 64 elements (about 0.6 us each on the tensor cores)
constexpr int E_TILE_COST = 1, E_PART_COST = 2;
constexpr int E_GATHERERS = E_PROD_WARPS + 1;
// bytes of a gathered row of X or W, and of codes: 64 elements from any offset into 16 bytes
constexpr int E_GATHER_F = E_KS * 4 + 16, E_GATHER_Q = E_KS + 16;
constexpr int E_SMEM_LIMIT = 232448;       // opt-in shared memory per CTA on sm_100 parts

struct ChainCtrl {
    uint64_t full[E_MAX_STAGES];    // even CTA: both CTAs' producer warps (rows written, X landed)
    uint64_t empty[E_MAX_STAGES];   // both CTAs: pair MMA commit (stage free)
    uint64_t xfull[E_MAX_XSLOTS];   // this CTA's X tile copy
    uint64_t xempty[E_MAX_XSLOTS];  // both CTAs: pair MMA commit (X slot free)
    uint64_t raw_full[E_MAX_RAW];   // this CTA's raw tile copies
    uint64_t raw_empty[E_MAX_RAW];  // this CTA's producer warps
    uint64_t segfull[2];            // both CTAs: pair MMA commit, per accumulator
    uint64_t segempty[2];           // even CTA: both CTAs' epilogue warps, per accumulator
    uint64_t done;                  // even CTA: every MMA complete
    uint64_t shared;                // the peer's sums of a tile are in `recv`
    uint32_t tmem_base;
    int abort;
    int xexp;
    int last[2];                    // this CTA was the last to leave a tile's sums
    float2 coef[E_N];               // per operand row of the pair: (2^{e_n - e_{n+1}}, s_n 2^e_n)
    int any_slow;                   // some channel of this CTA is left to slow_error (RAWX)
    int slow[E_VEC];                // per channel of this CTA: 1 + the last pair tile where it is
    double part[4][E_N];            // per lane quarter: sum over the rows' y^2
    double recv[2][E_VEC];          // the peer's sums for this CTA's channels (alternate tiles)
};
constexpr int E_CTRL_BYTES = (sizeof(ChainCtrl) + 1023) / 1024 * 1024;
constexpr int E_BASE_SMEM = 1024 /* alignment slack */ + E_CTRL_BYTES;

// Per-k_max geometry.  Raw slot, as the tile copies write it: W step [CH][64] fp32, codes
// [K][CH][64] int8, and (RAWX) X step [128][64] fp32 first; a gathered slot's rows are
// E_GATHER_F or E_GATHER_Q bytes.  X slots: as many as leave room for three operand
// stages and at least two raw slots.
template <int KP1, bool RAWX>
struct EGeo {
    static constexpr int K = KP1 - 1;
    static constexpr int R = KP1 + 1;                    // operand rows per channel
    static constexpr int CH = E_VEC / R;                 // channels per CTA
    static constexpr int ITEMS = (CH * 16 + E_PT - 1) / E_PT;   // 16 items of 4 elements per channel
    static constexpr int F_ROW = RAWX ? E_GATHER_F : E_KS * 4;   // reserved for a row
    static constexpr int RAW_W = RAWX ? E_ROWS * F_ROW : 0;
    static constexpr int RAW_Q = (RAW_W + CH * F_ROW + 127) / 128 * 128;
    static constexpr uint32_t RAW_TX = ((RAWX ? E_ROWS : 0) + CH) * E_KS * 4 + K * CH * E_KS;
    static constexpr int RAW_BYTES =
        (RAW_Q + K * CH * (RAWX ? E_GATHER_Q : E_KS) + 1023) / 1024 * 1024;
    static constexpr int NS = RAWX ? 2 : 3;              // operand stages
    // RAWX: the producers write X's tiles beside the operand rows, stage by stage
    static constexpr int NX =
        RAWX ? NS
             : (E_BASE_SMEM + 3 * E_TILE + 4 * E_XSET + 3 * RAW_BYTES <= E_SMEM_LIMIT ? 4 : 3);
    static constexpr int BASE = E_BASE_SMEM + NS * E_TILE + NX * E_XSET;
    static constexpr int RAW_FIT = (E_SMEM_LIMIT - BASE) / RAW_BYTES;
    static constexpr int RAW = RAW_FIT < E_MAX_RAW ? RAW_FIT : E_MAX_RAW;
    static constexpr int SMEM = BASE + RAW * RAW_BYTES;
    static_assert(K >= 1 && CH >= 1, "at least one point, one channel");
    static_assert(RAW >= 2, "raw ring needs two slots");
};

// Four biased codes (int8 XOR 0x80 per byte) as exact fp16 values, two per word: the byte becomes
// the low mantissa byte of 1024, and subtracting 1024 + 128 is exact.
__device__ __forceinline__ void codes_f16x4(uint32_t biased, uint32_t &c01, uint32_t &c23)
{
    const __half2 off = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));   // 1152
    const uint32_t a = __byte_perm(biased, 0x64646464u, 0x4140u);
    const uint32_t b = __byte_perm(biased, 0x64646464u, 0x4342u);
    const __half2 x = __hsub2(*reinterpret_cast<const __half2 *>(&a), off);
    const __half2 y = __hsub2(*reinterpret_cast<const __half2 *>(&b), off);
    c01 = *reinterpret_cast<const uint32_t *>(&x);
    c23 = *reinterpret_cast<const uint32_t *>(&y);
}

// 16 bytes of a gathered row, from any word.
__device__ __forceinline__ float4 ld_gathered(uint32_t a)
{
    float4 v;
    v.x = __uint_as_float(ld_shared_u32(a));
    v.y = __uint_as_float(ld_shared_u32(a + 4u));
    v.z = __uint_as_float(ld_shared_u32(a + 8u));
    v.w = __uint_as_float(ld_shared_u32(a + 12u));
    return v;
}

// Raw slot -> the operand rows of one step (tile `dst`): for every (channel, 4 contiguous
// elements) item the codes of every point as fp16, then the last residual (Eq. 7's recursion in
// fp32) scaled by 2^e and split into hi and lo.  Every shared-memory read before the stores; a
// half warp's 8-byte stores fill one 128-byte row.  gather: the slot's rows are the aligned 16 bytes
// around the elements; w0: address of W's row of the CTA's first channel, q0 of its codes of point 1,
// d: row length, plane: codes of a point (all of these count by their low four bits only, and a
// step starts a multiple of 64 elements into the row).
template <int KP1, bool RAWX>
__device__ __forceinline__ void chain_rows(uint32_t slot, uint32_t dst, int pt, int nch, bool gather,
                                           uint32_t w0, uint32_t q0, uint32_t d, uint32_t plane,
                                           const float (&sc)[EGeo<KP1, RAWX>::ITEMS][KP1 - 1],
                                           const float (&vf)[EGeo<KP1, RAWX>::ITEMS])
{
    using G = EGeo<KP1, RAWX>;
    constexpr int K = G::K;
#pragma unroll
    for (int i = 0; i < G::ITEMS; ++i) {
        const int p = pt + i * E_PT;
        if (p < nch * 16) {
            const int ch = p >> 4, e4 = p & 15;
            float4 r;
            if (RAWX && gather)
                r = ld_gathered(slot + G::RAW_W + (uint32_t)(ch * E_GATHER_F + e4 * 16) +
                                ((w0 + (uint32_t)ch * d * 4u) & 15u));
            else
                r = ld_shared_v4(slot + G::RAW_W + (uint32_t)(ch * E_KS + e4 * 4) * 4u);
            uint32_t qb[K];
#pragma unroll
            for (int n = 0; n < K; ++n) {
                if (RAWX && gather) {
                    const uint32_t at = q0 + (uint32_t)n * plane + (uint32_t)ch * d;
                    const uint32_t a = slot + G::RAW_Q + (at & 12u) +
                                       (uint32_t)((n * G::CH + ch) * E_GATHER_Q + e4 * 4);
                    qb[n] = __funnelshift_r(ld_shared_u32(a), ld_shared_u32(a + 4u), 8u * (at & 3u));
                } else {
                    qb[n] = ld_shared_u32(slot + G::RAW_Q +
                                          (uint32_t)((n * G::CH + ch) * E_KS + e4 * 4));
                }
                qb[n] ^= 0x80808080u;
            }
            const uint32_t cofs = (uint32_t)(e4 & 1) * 8u;   // 4 elements = 8 bytes of a 16-byte chunk
            const int row = ch * G::R;
#pragma unroll
            for (int n = 0; n < K; ++n) {
                uint32_t c01, c23;
                codes_f16x4(qb[n], c01, c23);
                st_shared_v2u(dst + sw128_offset(row + n, e4 >> 1) + cofs, c01, c23);
                const float sn = sc[i][n];
                r.x = __fmaf_rn(-sn, code_from_biased(qb[n], 0), r.x);
                r.y = __fmaf_rn(-sn, code_from_biased(qb[n], 1), r.y);
                r.z = __fmaf_rn(-sn, code_from_biased(qb[n], 2), r.z);
                r.w = __fmaf_rn(-sn, code_from_biased(qb[n], 3), r.w);
            }
            uint32_t h0, l0, h1, l1;
            split_f16x2(__fmul_rn(r.x, vf[i]), __fmul_rn(r.y, vf[i]), h0, l0);
            split_f16x2(__fmul_rn(r.z, vf[i]), __fmul_rn(r.w, vf[i]), h1, l1);
            st_shared_v2u(dst + sw128_offset(row + K, e4 >> 1) + cofs, h0, h1);
            st_shared_v2u(dst + sw128_offset(row + K + 1, e4 >> 1) + cofs, l0, l1);
        }
    }
}

// RAWX: items [p0, p1) of the step's X rows (row p / 16, 4 elements), `stride` threads apart, scaled
// by 2^e and split into the hi and lo tiles (the same values as f16_split_kernel's planes).
// gather: the slot's rows are the aligned 16 bytes around the elements, x0 the address of X and d the
// row length, by their low bits (a row tile starts a multiple of 128 rows into X).
template <int U>
__device__ __forceinline__ void chain_x(uint32_t slot, uint32_t xset, int p0, int p1, int stride,
                                        float xs, bool gather, uint32_t x0, uint32_t d)
{
    for (; p0 < p1; p0 += U * stride) {   // U reads in flight, all before their stores
        float4 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (const int p = p0 + u * stride; p < p1) {
                const uint32_t row = (uint32_t)p >> 4;
                x[u] = gather ? ld_gathered(slot + row * E_GATHER_F + ((uint32_t)p & 15u) * 16u +
                                            ((x0 + row * d * 4u) & 15u))
                              : ld_shared_v4(slot + (uint32_t)p * 16u);
            }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = p0 + u * stride, row = p >> 4, e4 = p & 15;
            if (p >= p1) break;
            uint32_t h0, l0, h1, l1;
            split_f16x2(__fmul_rn(x[u].x, xs), __fmul_rn(x[u].y, xs), h0, l0);
            split_f16x2(__fmul_rn(x[u].z, xs), __fmul_rn(x[u].w, xs), h1, l1);
            const uint32_t off = sw128_offset(row, e4 >> 1) + (uint32_t)(e4 & 1) * 8u;
            st_shared_v2u(xset + off, h0, h1);
            st_shared_v2u(xset + E_TILE + off, l0, l1);
        }
    }
}

// RAWX, rows that a tile copy cannot address: the producer warps and the copy warp each copy a share
// (part 0 .. E_GATHERERS - 1) of the raw slot of a step (columns x .. x + 63, X rows row0 .. + 127,
// channels k0 .. + nch - 1), for every row the aligned 16 bytes that hold its 64 elements, and arrive
// on `bar` with every lane.  Zeros from the row's end on and outside the arrays; what lies before
// the first element is not used.  No read outside an array: at its start, where the aligned 16
// bytes may begin before it, the words inside are copied one by one (X, W and codes are 4-byte
// aligned); at a row's end a copy reads no further.  (5245 x 1859, k_max = 5, N = 939: 1.12 ms; 4
// bytes at a time 1.55 ms, and all by one warp 3.0 ms.)
template <int PIECES>   // of 16 bytes, of which the last only where the row's offset needs it
__device__ __forceinline__ void gather_rows(uint32_t dst, uintptr_t base, uintptr_t row0,
                                            uint32_t row_bytes, uint32_t xb, int n, int valid, int th)
{
    constexpr int STEP = E_GATHERERS * 32 / PIECES;   // rows a pass; the threads left over idle
    int r = th / PIECES;
    const int c = th - r * PIECES;
    if (r >= STEP) return;
    uintptr_t at = row0 + (size_t)r * row_bytes + xb;
    dst += (uint32_t)th * 16u;
#pragma unroll 2
    for (; r < n; r += STEP, at += (size_t)STEP * row_bytes, dst += STEP * PIECES * 16u) {
        const int off = (int)(at & 15);
        const uintptr_t from = at - (unsigned)off + 16u * (unsigned)c;
        const int left = (int)(row_bytes - xb) + off - 16 * c;
        const bool need = r < valid && (c < PIECES - 1 || off);
        const uint32_t bytes = need ? (uint32_t)max(0, min(16, left)) : 0u;
        if (bytes && from < base) {
#pragma unroll 1
            for (uint32_t o = (uint32_t)(base - from); o < 16u; o += 4u) {
                const uint32_t b = o < bytes ? min(4u, bytes - o) : 0u;
                cp_async4(dst + o, reinterpret_cast<const void *>(b ? from + o : base), b);
            }
        } else {
            cp_async16(dst, reinterpret_cast<const void *>(bytes ? from : base & ~(uintptr_t)15),
                       bytes);
        }
    }
}

template <int KP1>
__device__ __noinline__ void gather_slot(int part, uint32_t slot, const float *__restrict__ X, int N,
                                         const float *__restrict__ W,
                                         const int8_t *__restrict__ codes, int C, int d, int x,
                                         int row0, int k0, int nch, int lane, uint64_t *bar)
{
    using G = EGeo<KP1, true>;
    const uintptr_t xp = (uintptr_t)X, wp = (uintptr_t)W, qp = (uintptr_t)codes;
    const uint32_t fb = (uint32_t)d * 4u, xb = (uint32_t)x * 4u;
    const int th = part * 32 + lane;
    gather_rows<E_GATHER_F / 16>(slot, xp, xp + (size_t)row0 * fb, fb, xb, E_ROWS, N - row0, th);
    gather_rows<E_GATHER_F / 16>(slot + G::RAW_W, wp, wp + (size_t)k0 * fb, fb, xb, nch, nch, th);
#pragma unroll 1
    for (int n = 0; n < G::K; ++n)
        gather_rows<E_GATHER_Q / 16>(slot + G::RAW_Q + (uint32_t)(n * G::CH * E_GATHER_Q), qp,
                                     qp + ((size_t)n * C + (size_t)k0) * d, (uint32_t)d, (uint32_t)x,
                                     nch, nch, th);
    cp_async_arrive(bar);
}

// Sum over the warp's 32 lanes of each of 32 values: lane l returns the sum of v[l].  Each exchange
// halves the values a lane carries (31 shuffles in all); a fixed tree, so deterministic.
__device__ __forceinline__ float warp_transpose_sum(float (&v)[32], int lane)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if (i < o) {
                const float keep = up ? v[i + o] : v[i];
                const float give = up ? v[i] : v[i + o];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
        }
    }
    return v[0];
}

// The 256 epilogue threads' barrier, and that of 128 of them (the owners of one CTA's channels).
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void own_sync() { asm volatile("bar.sync 2, 128;" ::: "memory"); }

// Partial sums of the pairs that have a part of a channel tile, in global scratch, by tile and CTA of
// the pair: how many have arrived (zeroed before the launch), and E_VEC sums per pair.
struct ChainScratch {
    unsigned *count;   // [tiles][2]
    double *slot;      // [tiles][parts][2][E_VEC]
    int parts;
};

// scales: [C][k_max] point scales; xrange[0], vrange: max|X| and max|r| per residual vector, as
// float bits; X, W, codes: read only by gathers and slow_error.  tiles: channel tiles of a pair
// (2 CH channels).  nearest: every channel's codes are nearest values.  tmX: the split X planes [2][N][d] fp16 (RAWX: X itself), tmW: W, tmQ: the codes.
template <int KP1, bool RAWX>
__global__ void __launch_bounds__(E_THREADS, 1)
output_error_chain_kernel(const float *__restrict__ X, const float *__restrict__ W,
                          const int8_t *__restrict__ codes, const float *__restrict__ scales, int C,
                          int N, int d, const unsigned *__restrict__ xrange,
                          const unsigned *__restrict__ vrange, float *__restrict__ err,
                          int tiles, int gang, bool nearest, const ChainScratch part,
                          const WaitCtl wc, const __grid_constant__ CUtensorMap tmX,
                          const __grid_constant__ CUtensorMap tmW,
                          const __grid_constant__ CUtensorMap tmQ)
{
    using G = EGeo<KP1, RAWX>;
    constexpr int K = G::K, NS = G::NS, NX = G::NX, RAW = G::RAW, R = G::R, CH = G::CH;
    // warps that write a stage's operands (RAWX: the epilogue warps split X between their folds)
    constexpr int SPLIT_WARPS = E_PROD_WARPS + (RAWX ? E_EPI_WARPS : 0);
    constexpr unsigned KBIT = MPQ_TIMEOUT_OUTPUT_ERROR;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw_u32 = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw_u32 & 1023u)) & 1023u;
    ChainCtrl &ctl = *reinterpret_cast<ChainCtrl *>(smem_raw + pad);
    const uint32_t x_u32 = raw_u32 + pad + E_CTRL_BYTES;
    const uint32_t v_u32 = x_u32 + NX * E_XSET;
    const uint32_t ring_u32 = v_u32 + NS * E_TILE;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool gather = RAWX && !tile_rows_ok(X, W, codes, d);
    const uint32_t crank = cluster_ctarank();
    const int half = (int)crank;                     // 0: even CTA (issues the MMAs), 1: its peer
    const uint16_t pair_mask = 3u;
    const int n_rt = (N + E_M - 1) / E_M;
    const int n_ks = (d + E_KS - 1) / E_KS;          // steps per row tile
    const int nseg = (n_ks + E_SEG - 1) / E_SEG;
    // this pair's channel tiles [tile0, tile1) and its row tiles of each: with a gang the same
    // [rt0, rt1) of every one; else from rt0 on of the first and up to rt1 of the last
    const int pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
    int tile0, tile1, rt0, rt1, member = 0;
    long long total;   // steps
    if (gang > 0) {
        const int n_gangs = n_pairs / gang, gid = pair / gang;
        member = pair - gid * gang;
        tile0 = (int)((long long)tiles * gid / n_gangs);
        tile1 = (int)((long long)tiles * (gid + 1) / n_gangs);
        rt0 = (int)((long long)n_rt * member / gang);
        rt1 = (int)((long long)n_rt * (member + 1) / gang);
        total = (long long)(tile1 - tile0) * (rt1 - rt0) * n_ks;
    } else {
        const long long units = (long long)tiles * n_rt;
        const long long u0 = units * pair / n_pairs, u1 = units * (pair + 1) / n_pairs;
        tile0 = (int)(u0 / n_rt);
        tile1 = (int)((u1 - 1) / n_rt) + 1;
        rt0 = (int)(u0 - (long long)tile0 * n_rt);
        rt1 = (int)(u1 - (long long)(tile1 - 1) * n_rt);
        total = (u1 - u0) * n_ks;
    }
    auto rt_lo = [&](int tile) { return gang > 0 || tile == tile0 ? rt0 : 0; };
    auto rt_hi = [&](int tile) { return gang > 0 || tile == tile1 - 1 ? rt1 : n_rt; };
    // first channel of this CTA in a pair tile, and how many of its channels exist
    auto chan0 = [&](int tile) { return (tile * 2 + half) * CH; };
    auto n_chan = [&](int tile) { return max(0, min(CH, C - chan0(tile))); };
    // control block, tiles and the raw ring within the launch's shared memory (the same in every
    // CTA, so the whole cluster leaves together)
    if (!MPQ_CHECK_SMEM_END((size_t)pad + E_CTRL_BYTES + (size_t)NX * E_XSET + (size_t)NS * E_TILE +
                            (size_t)RAW * G::RAW_BYTES))
        return;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(&ctl.full[s], 2 * SPLIT_WARPS);
            mbar_init(&ctl.empty[s], 1);
        }
        for (int s = 0; s < NX; ++s) {
            mbar_init(&ctl.xfull[s], 1);
            mbar_init(&ctl.xempty[s], 1);
        }
        for (int r = 0; r < RAW; ++r) {
            mbar_init(&ctl.raw_full[r], gather ? E_GATHERERS * 32 : 1);   // who copies the slot
            mbar_init(&ctl.raw_empty[r], SPLIT_WARPS);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&ctl.segfull[b], 1);
            mbar_init(&ctl.segempty[b], 2 * E_EPI_WARPS);
        }
        mbar_init(&ctl.done, 1);
        mbar_init(&ctl.shared, E_VEC);
        ctl.abort = 0;
        ctl.any_slow = 0;
        fence_barrier_init();
    }
    if (threadIdx.x < E_VEC) ctl.slow[threadIdx.x] = 0;
    if (warp == E_MMA_WARP) {
        tmem_alloc_pair(&ctl.tmem_base, E_TMEM_COLS);
        tc_fence_before();
    }
    griddep_wait();                     // nothing above reads global memory
    if (threadIdx.x == 0) ctl.xexp = f16_scale_exp(__uint_as_float(ld_after_wait(xrange)));
    cluster_sync();                     // barriers of both CTAs initialised, TMEM allocated
    tc_fence_after();
    const uint32_t tmem = ctl.tmem_base;
    volatile int *abort_flag = &ctl.abort;

    // RAWX with gathered rows, by every warp of the producers and the copy warp: this warp's share of
    // the steps before `upto`, each once its slot is free (false: give up; warp-uniform)
    long long gf = 0;
    int gks = 0, grt = rt0, gtile = tile0, gslot = 0;
    uint32_t gph = 1;
    auto gather_to = [&](long long upto) -> bool {
        for (; gf < upto && gf < total; ++gf) {
            bool ok = !*abort_flag;
            if (ok && gf >= RAW) {
                ok = mbar_wait(&ctl.raw_empty[gslot], gph, wc.budget);
                if (!ok) note_timeout(wc, KBIT);
            }
            if (__any_sync(0xffffffffu, !ok)) {
                *abort_flag = 1;
                return false;
            }
            gather_slot<KP1>(warp, ring_u32 + gslot * G::RAW_BYTES, X, N, W, codes, C, d, gks * E_KS,
                             grt * E_M + half * E_ROWS, chan0(gtile), n_chan(gtile), lane,
                             &ctl.raw_full[gslot]);
            if (++gks == n_ks) {
                gks = 0;
                if (++grt == rt_hi(gtile)) {
                    ++gtile;
                    grt = rt_lo(gtile);
                }
            }
            if (++gslot == RAW) {
                gslot = 0;
                gph ^= 1u;
            }
        }
        return true;
    };

    // one setmaxnreg per warpgroup: 0-1 give registers to 2-3 (epilogue)
    if (warp < E_EPI_WARP0) {
        setmaxnreg_dec<ERegs<K, RAWX>::LOW>();
        if (warp < E_PROD_WARPS) {
            // ------------------------------------------------------------ producers
            const int pt = threadIdx.x;
            float sc[G::ITEMS][K];      // scales of this thread's items in the current tile
            float vf[G::ITEMS];         // 2^e of the items' last residual
            int nch = 0;
            const float xs = pow2f(ctl.xexp);
            int s = 0, slot = 0, sx = 0;
            uint32_t sph = 0, rph = 0, xph = 0;    // phase parities of stage s, raw slot, X slot sx
            long long left = 0;         // steps left in the tile
            int tile = tile0 - 1, k0 = 0;
            for (long long it = 0; it < total; ++it) {
                if (left-- == 0) {
                    // a new tile's channels
                    ++tile;
                    left = (long long)(rt_hi(tile) - rt_lo(tile)) * n_ks - 1;
                    nch = n_chan(tile);
                    k0 = chan0(tile);
#pragma unroll
                    for (int i = 0; i < G::ITEMS; ++i) {
                        const int p = pt + i * E_PT, c = p >> 4;
                        const bool own = p < nch * 16;
#pragma unroll
                        for (int n = 0; n < K; ++n)
                            sc[i][n] = own ? __ldg(scales + (size_t)(k0 + c) * K + n) : 0.0f;
                        vf[i] = own ? pow2f(f16_scale_exp(__uint_as_float(
                                          ld_after_wait(vrange + (size_t)(k0 + c) * KP1 + K))))
                                    : 0.0f;
                    }
                }
                if constexpr (RAWX) {
                    if (gather && !gather_to(it + RAW)) break;
                }
                bool ok = mbar_wait(&ctl.raw_full[slot], rph, wc.budget) &&
                          mbar_wait_cluster(&ctl.empty[s], sph ^ 1u, wc.budget);
                if (!ok) {
                    *abort_flag = 1;
                    note_timeout(wc, KBIT);
                }
                if (__any_sync(0xffffffffu, !ok || *abort_flag)) break;   // warp-uniform
                const uint32_t src = ring_u32 + slot * G::RAW_BYTES;
                chain_rows<KP1, RAWX>(src, v_u32 + s * E_TILE, pt, nch, gather,
                                      (uint32_t)(uintptr_t)W + (uint32_t)k0 * (uint32_t)d * 4u,
                                      (uint32_t)(uintptr_t)codes + (uint32_t)k0 * (uint32_t)d,
                                      (uint32_t)d, (uint32_t)C * (uint32_t)d, sc, vf);
                if constexpr (RAWX)
                    chain_x<3>(src, x_u32 + s * E_XSET, E_X_EPI + pt, E_ROWS * 16, E_PT, xs, gather,
                               (uint32_t)(uintptr_t)X, (uint32_t)d);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl.raw_empty[slot]);
                if constexpr (!RAWX) {
                    // the step's X tiles have landed too before the stage is reported full
                    ok = mbar_wait(&ctl.xfull[sx], xph, wc.budget);
                    if (!ok) {
                        *abort_flag = 1;
                        note_timeout(wc, KBIT);
                    }
                    if (__any_sync(0xffffffffu, !ok || *abort_flag)) break;
                }
                if (lane == 0) mbar_arrive_cluster(&ctl.full[s], 0);
                if (++s == NS) {
                    s = 0;
                    sph ^= 1u;
                }
                if (++slot == RAW) {
                    slot = 0;
                    rph ^= 1u;
                }
                if (++sx == NX) {
                    sx = 0;
                    xph ^= 1u;
                }
            }
            if (RAWX && gather) cp_async_wait_all();
        } else if (warp == E_COPY_WARP) {
            // ------------------------------------------------------------ tile copies
            // raw tiles of step f into slot f % RAW once the producers have released step f - RAW,
            // X rows of step f into X slot f % NX once the MMAs of step f - NX have completed
            if (gather && wc.withhold == 0) {
                if constexpr (RAWX) {
                    (void)gather_to(total);
                    cp_async_wait_all();
                }
            } else if (lane == 0 && wc.withhold == 0) {
                prefetch_tensormap(&tmX);
                prefetch_tensormap(&tmW);
                prefetch_tensormap(&tmQ);
                long long raw_issued = 0, x_issued = 0;
                int ks = 0, rt = rt0, tile = tile0, rslot = 0, xslot = 0;
                uint32_t rph = 1, xph = 1;   // parities of the waits for a free slot
                for (long long f = 0; f < total && !*abort_flag; ++f) {
                    const int x = ks * E_KS, row0 = rt * E_M + half * E_ROWS, k0 = chan0(tile);
                    const uint32_t rdst = ring_u32 + rslot * G::RAW_BYTES;
                    const uint32_t xdst = x_u32 + xslot * E_XSET;
                    // a tile copy starts 16-byte aligned (x counts int8 codes in the code map)
                    // into an aligned destination, or is not issued and the launch ends through
                    // the bounded waits
                    bool ok = MPQ_CHECK((x & 15) == 0 && (rdst & 127u) == 0u &&
                                        (xdst & 1023u) == 0u && x < d);
                    if (!ok) {
                        *abort_flag = 1;
                        break;
                    }
                    if (f >= RAW)
                        ok = mbar_wait(&ctl.raw_empty[rslot], rph, wc.budget);
                    if (ok) {
                        mbar_arrive_expect_tx(&ctl.raw_full[rslot], G::RAW_TX);
                        if constexpr (RAWX) tma_load_2d(rdst, &tmX, x, row0, &ctl.raw_full[rslot]);
                        tma_load_2d(rdst + G::RAW_W, &tmW, x, k0, &ctl.raw_full[rslot]);
                        tma_load_3d(rdst + G::RAW_Q, &tmQ, x, k0, 0, &ctl.raw_full[rslot]);
                        raw_issued = f + 1;
                    }
                    if constexpr (!RAWX) {
                        if (ok && f >= NX)
                            ok = mbar_wait_cluster(&ctl.xempty[xslot], xph, wc.budget);
                        if (ok) {
                            mbar_arrive_expect_tx(&ctl.xfull[xslot], E_XSET);
                            tma_load_3d(xdst, &tmX, x, row0, 0, &ctl.xfull[xslot]);
                            x_issued = f + 1;
                        }
                    }
                    if (!ok) {
                        *abort_flag = 1;
                        note_timeout(wc, KBIT);
                        break;
                    }
                    if (++ks == n_ks) {
                        ks = 0;
                        if (++rt == rt_hi(tile)) {
                            ++tile;
                            rt = rt_lo(tile);
                        }
                    }
                    if (++rslot == RAW) {
                        rslot = 0;
                        rph ^= 1u;
                    }
                    if (++xslot == NX) {
                        xslot = 0;
                        xph ^= 1u;
                    }
                }
                // no copy lands after the CTA is gone: the last copy of every slot
                for (long long f = raw_issued - RAW > 0 ? raw_issued - RAW : 0; f < raw_issued; ++f)
                    drain_wait(&ctl.raw_full[f % RAW], (uint32_t)(f / RAW) & 1u, wc, KBIT);
                for (long long f = x_issued - NX > 0 ? x_issued - NX : 0; f < x_issued; ++f)
                    drain_wait(&ctl.xfull[f % NX], (uint32_t)(f / NX) & 1u, wc, KBIT);
            }
        } else if (half == 0 && lane == 0) {
            // ------------------------------------------------------------ MMA issuer (even CTA)
            constexpr uint32_t idesc = idesc_f16(E_M, E_N);
            bool ok = true;
            // step it = (row tile, step ks), stage s, X slot sx, segment g (accumulator g & 1)
            int ks = 0, s = 0, sx = 0, g = 0, sk = 0;
            uint32_t sph = 0;
            for (long long it = 0; it < total && ok && !*abort_flag; ++it) {
                const bool seg_start = sk == 0;
                const uint32_t b = (uint32_t)g & 1u;
                if (seg_start) {
                    // this accumulator's previous segment has been folded by both epilogues
                    if (!mbar_wait_cluster(&ctl.segempty[b], ((uint32_t)(g >> 1) & 1u) ^ 1u,
                                           wc.budget)) {
                        note_timeout(wc, KBIT);
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                }
                if (!mbar_wait_cluster(&ctl.full[s], sph, wc.budget)) {
                    note_timeout(wc, KBIT);
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t xset = x_u32 + sx * E_XSET;
                const uint64_t xh = smem_desc_sw128(xset), xl = smem_desc_sw128(xset + E_TILE);
                const uint64_t v = smem_desc_sw128(v_u32 + s * E_TILE);
                const uint32_t dt = tmem + b * (E_TMEM_COLS / 2);
                // 64 fp16 elements = four K = 16 steps, 32 bytes apart in the 128-byte rows
                // (16-byte units); per K step X's lo, then its hi half
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint64_t o = (uint64_t)(kk * 2);
                    mma_f16_pair(dt, xl + o, v + o, idesc, (seg_start && kk == 0) ? 0u : 1u);
                    mma_f16_pair(dt, xh + o, v + o, idesc, 1u);
                }
                mma_commit_pair(&ctl.empty[s], pair_mask);
                if constexpr (!RAWX) mma_commit_pair(&ctl.xempty[sx], pair_mask);
                ++ks;
                if (++sk == E_SEG || ks == n_ks) {
                    mma_commit_pair(&ctl.segfull[b], pair_mask);
                    sk = 0;
                    ++g;
                }
                if (ks == n_ks) ks = 0;
                if (++s == NS) {
                    s = 0;
                    sph ^= 1u;
                }
                if (++sx == NX) sx = 0;
            }
            if (!ok) *abort_flag = 1;
            // drain: every MMA issued above completes before tensor memory is released
            mma_commit_pair(&ctl.done, (uint16_t)1u);
            drain_wait_cluster(&ctl.done, 0, wc, KBIT);
        }
        __syncwarp();
    } else {
        setmaxnreg_inc<ERegs<K, RAWX>::HIGH>();
        // ---------------------------------------------------------------- epilogue
        // lane quarter q (the TMEM lanes this warp may access) and column half h (that CTA's
        // channels); the running sums of this thread's calibration row stay in registers
        const int ew = warp - E_EPI_WARP0, q = ew & 3, h = ew >> 2;
        const int et = ew * 32 + lane;                  // operand row et of the pair's 256
        const int m = et & (E_VEC - 1), mc = m / R, mn = m - mc * R;   // its channel and point
        const bool mine = (et >> 7) == half;            // one of this CTA's channels
        const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * E_VEC);
        float sums[E_VEC];
        double acc[4];              // operand rows 32 i + lane of this half
        unsigned g = 0;             // segment
        bool stop = false;
        // RAWX: this thread's share of X's split, step by step and at most NS steps beyond the
        // segment that is folded next
        long long made = 0, seg_end = 0;   // steps split, steps up to that segment's end
        int xslot = 0, xstage = 0;
        uint32_t xrph = 0, xsph = 0;
        auto split_x = [&](long long upto) {
            const float xs = pow2f(ctl.xexp);
            for (; made < upto && !stop; ++made) {
                const bool ok = mbar_wait(&ctl.raw_full[xslot], xrph, wc.budget) &&
                                mbar_wait_cluster(&ctl.empty[xstage], xsph ^ 1u, wc.budget);
                if (!ok) {
                    *abort_flag = 1;
                    note_timeout(wc, KBIT);
                }
                stop = __any_sync(0xffffffffu, !ok || *abort_flag);   // warp-uniform
                if (stop) break;
                chain_x<2>(ring_u32 + xslot * G::RAW_BYTES, x_u32 + xstage * E_XSET, et, E_X_EPI,
                           256, xs, gather, (uint32_t)(uintptr_t)X, (uint32_t)d);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&ctl.raw_empty[xslot]);
                    mbar_arrive_cluster(&ctl.full[xstage], 0);
                }
                if (++xslot == RAW) {
                    xslot = 0;
                    xrph ^= 1u;
                }
                if (++xstage == NS) {
                    xstage = 0;
                    xsph ^= 1u;
                }
            }
        };
        for (int tile = tile0; tile < tile1; ++tile) {
            int me = 0;
            bool slow = false;
            // a new tile: the chain's constants of both CTAs' operand rows, this CTA's slow
            // channels (every warp is done with the last tile's: the barrier at its end)
            float2 cf = make_float2(0.0f, 0.0f);
            const int k = (tile * 2 + (et >> 7)) * CH + mc;
            if (mc < CH && k < C && mn <= K && MPQ_IN((size_t)k * KP1 + mn, (size_t)C * KP1)) {
                const float vr = __uint_as_float(ld_after_wait(vrange + (size_t)k * KP1 + mn));
                me = f16_scale_exp(vr);
                if (mn < K) {
                    const float vn = __uint_as_float(ld_after_wait(vrange + (size_t)k * KP1 + mn + 1));
                    const float sn = __ldg(scales + (size_t)k * K + mn);
                    const int de = me - f16_scale_exp(vn);
                    // (beyond 2^-126 the later residuals are nothing beside this one; a
                    // growing residual is a slow channel's)
                    cf = make_float2(de < -126 ? 0.0f : pow2f(min(de, 126)),
                                     __fmul_rn(sn, pow2f(me)));
                    if (mine && !nearest && slow_point(vr, vn, sn, growth_limit(K))) {
                        ctl.slow[mc] = tile + 1;
                        if constexpr (RAWX) ctl.any_slow = 1;
                    }
                }
            }
            ctl.coef[et] = cf;
            epi_sync();
            slow = mine && mc < CH && ctl.slow[mc] == tile + 1;
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = 0.0;
            for (int rt = rt_lo(tile); rt < rt_hi(tile); ++rt) {
#pragma unroll
                for (int i = 0; i < E_VEC; ++i) sums[i] = 0.0f;
                for (int sg = 0; sg < nseg; ++sg, ++g) {
                    const uint32_t b = g & 1u, par = (g >> 1) & 1u;
                    if constexpr (RAWX) {
                        seg_end += min(E_SEG, n_ks - sg * E_SEG);
                        split_x(min(total, seg_end + NS));
                    }
                    if (stop) break;
                    const bool ok = mbar_wait_cluster(&ctl.segfull[b], par, wc.budget);
                    if (!ok) {
                        *abort_flag = 1;
                        note_timeout(wc, KBIT);
                    }
                    stop = __any_sync(0xffffffffu, !ok || *abort_flag);   // warp-uniform
                    if (stop) break;
                    tc_fence_after();
                    // (a row tile's sums start from zero: 0 + v = v, up to the sign of a zero, which
                    // the squares below do not see)
#pragma unroll
                    for (int cb = 0; cb < E_VEC / 16; ++cb) {   // (32 columns at a time spill registers)
                        float v[16];
                        tmem_ld_32x32b_x16(lane_base + b * (E_TMEM_COLS / 2) + (uint32_t)(cb * 16), v);
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            sums[cb * 16 + i] = __fadd_rn(v[i], sums[cb * 16 + i]);
                    }
                    // the accumulator is free again (the loads have completed)
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(&ctl.segempty[b], 0);
                }
                // (after a timeout every warp still goes through the tiles' barriers, with NaN)
                // the chain of every channel, from its last residual up: the row tile's squares in
                // place of the sums, then over the warp's rows
                const float2 *cf = ctl.coef + h * E_VEC;
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    float y = __fadd_rn(sums[c * R + K + 1], sums[c * R + K]);
                    sums[c * R + K + 1] = 0.0f;
                    sums[c * R + K] = __fmul_rn(y, y);
#pragma unroll
                    for (int n = K - 1; n >= 0; --n) {
                        const float2 f = cf[c * R + n];
                        y = __fmaf_rn(y, f.x, __fmul_rn(f.y, sums[c * R + n]));
                        sums[c * R + n] = __fmul_rn(y, y);
                    }
                }
#pragma unroll
                for (int cb = 0; cb < E_VEC / 32; ++cb) {
                    float v[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = sums[cb * 32 + i];
                    acc[cb] += (double)warp_transpose_sum(v, lane);
                }
            }
            // ---- the end of the tile: the sums over the lane quarters, exchanged so that each CTA
            // has its own channels' over both CTAs' rows
#pragma unroll
            for (int cb = 0; cb < 4; ++cb) ctl.part[q][h * E_VEC + cb * 32 + lane] = acc[cb];
            epi_sync();
            double s = ((ctl.part[0][et] + ctl.part[1][et]) + ctl.part[2][et]) + ctl.part[3][et];
            if (*abort_flag) s = (double)NAN;
            const int rb = (tile - tile0) & 1;
            if (!mine) {
                st_dsmem_f64(&ctl.recv[rb][m], (uint32_t)(half ^ 1), s);
                mbar_arrive_release_cluster(&ctl.shared, (uint32_t)(half ^ 1));
            } else {
                if (mbar_wait_cluster(&ctl.shared, (uint32_t)rb, wc.budget)) {
                    s = half == 0 ? s + ctl.recv[rb][m] : ctl.recv[rb][m] + s;
                } else {
                    *abort_flag = 1;
                    note_timeout(wc, KBIT);
                    s = (double)NAN;
                }
                // which of the pairs that have a part of this tile this one is
                int n_parts = gang, part_at = member;
                if (gang == 0) {
                    n_parts = 1;
                    if (rt_lo(tile) > 0 || rt_hi(tile) < n_rt) {
                        // (unit u is pair ((u + 1) n_pairs - 1) / units's)
                        const long long units = (long long)tiles * n_rt, ut = (long long)tile * n_rt;
                        const int p0 = (int)(((ut + 1) * n_pairs - 1) / units);
                        n_parts = (int)(((ut + n_rt) * n_pairs - 1) / units) - p0 + 1;
                        part_at = pair - p0;
                    }
                }
                bool write = true;
                if (n_parts > 1) {   // this pair's share into scratch; the last one adds them
                    double *slots = part.slot + ((size_t)tile * part.parts * 2 + half) * E_VEC + m;
                    slots[(size_t)part_at * 2 * E_VEC] = s;
                    __threadfence();
                    own_sync();
                    if (m == 0)
                        ctl.last[rb] = atomicAdd(part.count + 2 * (size_t)tile + half, 1u) ==
                                       (unsigned)(n_parts - 1);
                    own_sync();
                    write = ctl.last[rb] != 0;
                    if (write) {
                        __threadfence();
                        s = 0.0;
                        for (int p = 0; p < n_parts; ++p)
                            s += __ldcg(slots + (size_t)p * 2 * E_VEC);
                    }
                }
                const int k = chan0(tile) + mc;
                if (write && mc < n_chan(tile) && mn <= K && !slow &&
                    MPQ_IN((size_t)k * KP1 + mn, (size_t)C * KP1)) {
                    // exact: undo the operand scales
                    err[(size_t)k * KP1 + mn] =
                        (float)(s / (double)N * pow2d(-2 * (ctl.xexp + me)));
                }
            }
            stop = __any_sync(0xffffffffu, stop || *abort_flag);
        }
        __syncwarp();
    }

    cluster_sync();   // nothing of the pair's is in flight: the peer's sums have been read
    if constexpr (RAWX) {
        if (warp >= E_EPI_WARP0 && ctl.any_slow && !*abort_flag) {
            // slow channels, by the pair that has a tile's first row tile
            const SlowLayer layer = {X, W, codes, scales, vrange, err, C, N, d, K};
            for (int tl = tile0; tl < tile1; ++tl) {
                if (rt_lo(tl) != 0) continue;
                for (int c = 0; c < n_chan(tl); ++c) {
                    if (!is_slow(layer, chan0(tl) + c)) continue;
                    for (int n = warp - E_EPI_WARP0; n <= K; n += S_WARPS)
                        slow_error(layer, chan0(tl) + c, n, lane);
                }
            }
        }
    }
    if (warp == E_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, E_TMEM_COLS);
    }
}

// A: X (RAWX) or its split planes.
template <int KP1, bool RAWX>
mpq_status launch_chain(const float *X, const void *A, int N, const float *W, const int8_t *codes,
                        const float *scales, int C, int d, float *err, const unsigned *xrange,
                        const unsigned *vrange, bool nearest, const PadRows &pad, void *part,
                        size_t part_bytes, cudaStream_t stream)
{
    using G = EGeo<KP1, RAWX>;
    const int n_rt = (int)((N + (long long)E_M - 1) / E_M);
    const int tiles = chain_tiles(C, KP1 - 1), n_ks = (d + E_KS - 1) / E_KS;

    CUtensorMap tmX, tmW, tmQ;
    memset(&tmX, 0, sizeof(tmX));
    memset(&tmW, 0, sizeof(tmW));
    memset(&tmQ, 0, sizeof(tmQ));
    bool maps = true;
    const bool gather = RAWX && !tile_rows_ok(X, W, codes, d);   // no tile copies at all
    const int dp = (d + 15) / 16 * 16;                           // a row of the planes and copies
    const float *wt = pad.W ? pad.W : W;
    const int8_t *qt = pad.W ? pad.codes : codes;
    if constexpr (RAWX) {
        const cuuint64_t dx[2] = {(cuuint64_t)d, (cuuint64_t)N}, sx[1] = {(cuuint64_t)d * 4};
        const cuuint32_t bx[2] = {E_KS, E_ROWS};
        if (!gather) maps = encode_tile_map(&tmX, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, A, dx, sx, bx);
    } else {
        const cuuint64_t dx[3] = {(cuuint64_t)dp, (cuuint64_t)N, 2};
        const cuuint64_t sx[2] = {(cuuint64_t)dp * 2, (cuuint64_t)N * dp * 2};
        const cuuint32_t bx[3] = {E_KS, E_ROWS, 2};
        maps = encode_tile_map(&tmX, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, A, dx, sx, bx,
                               CU_TENSOR_MAP_SWIZZLE_128B);
    }
    const cuuint64_t dw[2] = {(cuuint64_t)dp, (cuuint64_t)C}, sw[1] = {(cuuint64_t)dp * 4};
    const cuuint32_t bw[2] = {E_KS, (cuuint32_t)G::CH};
    const cuuint64_t dq[3] = {(cuuint64_t)dp, (cuuint64_t)C, (cuuint64_t)G::K};
    const cuuint64_t sq[2] = {(cuuint64_t)dp, (cuuint64_t)C * dp};
    const cuuint32_t bq[3] = {E_KS, (cuuint32_t)G::CH, (cuuint32_t)G::K};
    if (!gather)
        maps = maps && encode_tile_map(&tmW, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, wt, dw, sw, bw) &&
               encode_tile_map(&tmQ, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, qt, dq, sq, bq);
    if (!maps) {
        set_error("output error: tensor map encoding failed");
        return MPQ_ERR_CUDA;
    }
    if ((long long)G::SMEM > max_smem_optin()) {
        set_error("output error needs %d bytes of shared memory", G::SMEM);
        return MPQ_ERR_UNSUPPORTED;
    }
    static std::atomic<int> limit[kMaxDevices];
    cudaError_t e = allow_smem(reinterpret_cast<const void *>(output_error_chain_kernel<KP1, RAWX>),
                               limit, G::SMEM);
    if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute");

    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(E_THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)G::SMEM;
    cfg.stream = stream;
    // (with fixed scratch the launches stay ordinary ones: a graph captured from them has no
    // programmatic edges)
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = after_previous_kernel();
    cfg.attrs = attr;
    cfg.numAttrs = RAWX ? 1 : 2;
    // one resident pair per two SMs (queried once per process), no more than units
    static std::atomic<int> resident{0};
    int pairs = resident.load(std::memory_order_relaxed);
    if (pairs == 0) {
        cfg.gridDim = dim3(2 * E_MAX_PAIRS, 1, 1);
        e = cudaOccupancyMaxActiveClusters(&pairs, output_error_chain_kernel<KP1, RAWX>, &cfg);
        if (e != cudaSuccess) return cuda_status(e, "cudaOccupancyMaxActiveClusters");
        pairs = std::max(1, std::min(pairs, E_MAX_PAIRS));
        resident.store(pairs, std::memory_order_relaxed);
    }
    // the schedule with the least work on the busiest pair (see the top) within the scratch given;
    // on ties the larger gang, contiguous runs only where they are better
    int gang = 1, parts = 1;
    long long best = -1;
    for (int g = 1; g <= E_MAX_GANG && g <= n_rt && g <= pairs; g *= 2) {
        const long long gangs = std::min<long long>(pairs / g, tiles);
        const long long cost = ((tiles + gangs - 1) / gangs) *
                               ((long long)((n_rt + g - 1) / g) * n_ks + E_TILE_COST +
                                (g > 1 ? E_PART_COST : 0));
        if (g > 1 && chain_scratch_bytes(tiles, g) > part_bytes) break;
        if (best < 0 || cost <= best) {
            best = cost;
            gang = g;
            parts = g;
        }
    }
    const long long units = (long long)tiles * n_rt;
    const long long runs = std::min<long long>(pairs, units);        // pairs with a run of their own
    const long long most = (units + runs - 1) / runs, least = units / runs;
    const long long split = std::min<long long>(n_rt, (n_rt + 2 * least - 2) / least);   // of a tile
    const long long over = std::min<long long>(most, (most + 2LL * n_rt - 2) / n_rt);    // tiles of a run
    const double reread = (double)C * d * (4 + G::K) > 64e6 ? 1.06 : 1.0;   // W and codes beyond L2
    if (split <= E_MAX_GANG && chain_scratch_bytes(tiles, (int)split) <= part_bytes &&
        reread * (double)(most * n_ks + over * (E_TILE_COST + E_PART_COST)) < (double)best) {
        gang = 0;
        parts = (int)split;
    }
    pairs = gang > 0 ? (int)std::min<long long>(pairs / gang, tiles) * gang : (int)runs;
    cfg.gridDim = dim3((unsigned)(2 * pairs), 1, 1);
    ChainScratch sp;
    sp.count = static_cast<unsigned *>(part);
    sp.slot = reinterpret_cast<double *>(static_cast<char *>(part) + chain_count_bytes(tiles));
    sp.parts = parts;
    WaitCtl wc;
    const mpq_status wst = wait_ctl(&wc);
    if (wst != MPQ_OK) return wst;
    e = cudaLaunchKernelEx(&cfg, output_error_chain_kernel<KP1, RAWX>, X, W, codes, scales, C, N, d,
                           xrange, vrange, err, tiles, gang, nearest, sp, wc, tmX, tmW, tmQ);
    return cuda_status(e, "output-error kernel launch");
}

}  // namespace

int chain_tiles(int C, int k_max)
{
    const int ch = E_VEC / (k_max + 2);
    return (int)((C + 2LL * ch - 1) / (2 * ch));
}

size_t chain_count_bytes(int tiles) { return ((size_t)tiles * 8 + 255) / 256 * 256; }

size_t chain_scratch_bytes(int tiles, int gang)
{
    return chain_count_bytes(tiles) + (gang > 1 ? (size_t)tiles * gang * 2 * E_VEC * 8 : 0);
}

int chain_max_gang(int N) { return N <= E_M ? 1 : E_MAX_GANG; }

mpq_status launch_output_error_chain(const float *X, int N, const float *W, const int8_t *codes,
                                     const float *scales, int C, int d, int k_max, float *err,
                                     const unsigned *xrange, const unsigned *vrange,
                                     bool nearest, const uint16_t *xs, const PadRows &pad, void *part,
                                     size_t part_bytes, cudaStream_t stream)
{
    switch (k_max) {
#define MPQ_CASE(n)                                                                               \
    case n:                                                                                       \
        return xs ? launch_chain<n + 1, false>(X, xs, N, W, codes, scales, C, d, err, xrange,     \
                                               vrange, nearest, pad, part, part_bytes, stream)    \
                  : launch_chain<n + 1, true>(X, X, N, W, codes, scales, C, d, err, xrange,       \
                                              vrange, nearest, pad, part, part_bytes, stream);
        MPQ_CASE(1) MPQ_CASE(2) MPQ_CASE(3) MPQ_CASE(4) MPQ_CASE(5) MPQ_CASE(6) MPQ_CASE(7)
        MPQ_CASE(8) MPQ_CASE(9) MPQ_CASE(10) MPQ_CASE(11) MPQ_CASE(12) MPQ_CASE(13) MPQ_CASE(14)
        MPQ_CASE(15) MPQ_CASE(16)
#undef MPQ_CASE
    }
    set_error("k_max = %d unsupported", k_max);
    return MPQ_ERR_UNSUPPORTED;
}

}  // namespace mpq
