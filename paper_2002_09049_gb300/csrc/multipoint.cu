// Integer inference with multipoint weights (Sec. 3.4, Eq. 13):
//   Y[k][t] = sat32( floor( sum_{i<n_k} A_{k,i} (q_{k,i} . x_t) / 2^p ) ),  A_{k,i} = rint(2^p s_{k,i}),
// in the paper's three steps: integer dot products of every point's codes with the integer input
// (step 1), multiplication by the 32-bit coefficients and summation (step 2), and the shift by p
// (step 3).
//
// Packing (offline, mpq_pack_points).  Each channel's n_k code rows become consecutive rows of one
// operand: channels are grouped by R = the power of two >= n_k (a channel with no point gets one
// zero row), and every 128-row tile holds 128/R channels of one group, so a channel's rows are R
// aligned TMEM lanes of one warp.  Rows past n_k and empty slots are zero with coefficient 0.  The
// codes are stored as bf16 (every int8 value is exact), rows padded to a multiple of 64 elements.
//
// Step 1 on the tensor cores.  tcgen05.mma kind::f16 with bf16 operands: the codes (TMA straight
// into 128-byte-swizzled K-major tiles) against the input rows (int8 by TMA into a raw ring, turned
// into bf16 exactly by eight producer warps through the fp32 exponent bias).  Products are exact
// and every partial sum is an integer of magnitude below 2^24 when d * Qmax * 128 < 2^24, so the
// fp32 accumulator holds the exact dot products (checked on the host; other layers take
// multipoint_mma_kernel, whose warps each accumulate an eighth of a row exactly in fp32 and add the
// parts as integers).  A unit of work is two 128-row tiles against 256
// inputs, K chunks of 64, by a CTA pair (cta_group::2: each CTA holds one row tile and half of the
// inputs, and gets its row tile's outputs for all of them); resident pairs take units a grid apart
// (inputs fastest, so the pairs that share row tiles run together and read their codes from L2).
// Two accumulators of 256 TMEM columns alternate: the epilogue of one unit runs under the MMAs of
// the next.  Shared-memory bandwidth bounds a chunk, not the MMAs' 512 cycles: per CTA and chunk
// the codes take 128 wavefronts in and 128 out, the inputs 64 in, 64 read, 128 written as bf16 and
// 128 read: 640 in all (one CTA alone with 256 inputs: 1,024, and 1,300 cycles measured; the pair:
// 830, of which the hand-offs between its warps are about a half).
// Raw input tiles have a ring of their own (handed back as soon as the producers have read them);
// a codes tile and a bf16 input tile share a slot, freed by one commit.  Two groups of four producer warps take
// alternate chunks.
// Steps 2 and 3 in the epilogue: each lane turns its accumulator into an integer, multiplies by its
// row's coefficient in 64 bits, the R lanes of a channel add with warp shuffles, and the first lane
// shifts (arithmetic: floor), saturates and writes 32 consecutive outputs.  Every wait is bounded.
// Asymmetric sets (a centre B_k, Eq. 1): the producers also sum each input row's int8 values while
// they convert it, and the first lane adds A_B,k (sum_j x_tj), A_B,k = rint(2^p B_k), before the
// shift.
//
// A few inputs, rows that TMA cannot address (d not a multiple of 16, unaligned input) and layers
// beyond the exactness bound take multipoint_mma_kernel: one CTA per 16 or 32 packed rows, its eight
// warps splitting the K range, code rows and inputs straight from global memory into the fragments
// of warp-level bf16 MMAs.  A handful of inputs leaves nothing to do but read the codes, and the
// 256-input tiles of the kernel above leave most SMs without a row tile (4096 x 4096 at 1.25
// points a channel is 42 row tiles).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "mpq_internal.cuh"
#include "sm100.cuh"
#include "tf32_operands.cuh"
#include "waits.cuh"

MPQ_CHECKED_UNIT("multipoint.cu");

namespace mpq {
namespace {

using namespace sm100;

constexpr int L_M = 128;                        // packed rows per tile (TMEM lanes)
constexpr int L_N = 256;                        // inputs per tile (UMMA N)
constexpr int L_KC = 64;                        // bf16 per K chunk = one 128-byte swizzle row
constexpr int L_A_BYTES = L_M * L_KC * 2;       // 16 KB codes tile
constexpr int L_IN = L_N / 2;                   // inputs a CTA of the pair converts
constexpr int L_B_BYTES = L_IN * L_KC * 2;      // 16 KB input tile (bf16)
constexpr int L_RAW_BYTES = L_IN * L_KC;        // 8 KB input tile (int8, as loaded)

// Rings: operand slots (a codes tile by TMA and a bf16 input tile by the producers, freed together
// by the MMAs) and raw int8 input tiles (TMA, freed as soon as the producers have read them).
constexpr int L_SLOTS = 5, L_R_SLOTS = 6;
constexpr int L_OFF_B = L_SLOTS * L_A_BYTES;
constexpr int L_OFF_RAW = L_OFF_B + L_SLOTS * L_B_BYTES;
constexpr int L_OFF_OUT = L_OFF_RAW + L_R_SLOTS * L_RAW_BYTES;
constexpr int L_OUT_COLS = 8;                   // output columns a warp transposes at a time
constexpr int L_PROD_WARPS = 8;
constexpr int L_GROUP_WARPS = 4;                // producer warps of a chunk
constexpr int L_GROUPS = L_PROD_WARPS / L_GROUP_WARPS;
constexpr int L_GROUP_THREADS = L_GROUP_WARPS * 32;
constexpr int L_EPI_WARP0 = L_PROD_WARPS;       // warps 8..15: TMEM lane quarter warp % 4, column half
constexpr int L_EPI_WARPS = 8;
constexpr int L_MMA_WARP = L_EPI_WARP0 + L_EPI_WARPS;
constexpr int L_TMA_A_WARP = L_MMA_WARP + 1;    // codes tiles
constexpr int L_TMA_X_WARP = L_TMA_A_WARP + 1;  // raw input tiles
constexpr int L_THREADS = (L_TMA_X_WARP + 1) * 32;   // 608
constexpr int L_BYTES = L_OFF_OUT + L_EPI_WARPS * 32 * (L_OUT_COLS + 1) * 4;

struct LinCtrl {
    uint64_t a_full[L_SLOTS];         // this CTA's codes tile has landed
    uint64_t full[L_SLOTS];           // even CTA: both CTAs' producers (inputs written, codes landed)
    uint64_t empty[L_SLOTS];          // both CTAs: the MMAs reading a slot completed
    uint64_t r_full[L_R_SLOTS];       // this CTA's raw input tile has landed
    uint64_t r_empty[L_R_SLOTS];      // this CTA's producers read a raw input slot
    uint64_t acc_full[2];             // both CTAs: a unit's MMAs completed
    uint64_t acc_empty[2];            // even CTA: both CTAs' epilogues are done with a unit
    uint64_t done;                    // even CTA: every MMA completed
    uint64_t xs_ready[2];             // both CTAs' producers stored a unit's input-row sums here
    uint64_t xs_empty[2];             // both CTAs' epilogues are done with a unit's sums
    uint32_t tmem_base;
    int abort;
    int xsum[2][L_GROUPS][L_N];       // sum_j x_tj of a unit's inputs, by producer group (centred)
    int kch[L_EPI_WARPS][32];         // per epilogue warp: the channel of each lane's row (-1: none)
};
constexpr int L_CTRL_BYTES = (sizeof(LinCtrl) + 1023) / 1024 * 1024;
constexpr int L_SMEM = 1024 + L_CTRL_BYTES + L_BYTES;

// Row r of a packed buffer: (channel, point) or channel -1 / point -1 for padding.
struct PackView {
    int *coef;
    int *chan;
    int *point;
    int *tile_R;
    int *center;                  // A_B of each channel, or null
    __nv_bfloat16 *codes;
    int *flag;
};

PackView view(const mpq_packed_layout *L, void *packed)
{
    unsigned char *b = static_cast<unsigned char *>(packed);
    PackView v;
    v.coef = reinterpret_cast<int *>(b + L->off_coef);
    v.chan = reinterpret_cast<int *>(b + L->off_chan);
    v.point = reinterpret_cast<int *>(b + L->off_point);
    v.tile_R = reinterpret_cast<int *>(b + L->off_tile);
    v.center = L->centered ? reinterpret_cast<int *>(b + L->off_center) : nullptr;
    v.codes = reinterpret_cast<__nv_bfloat16 *>(b + L->off_codes);
    v.flag = reinterpret_cast<int *>(b);   // header word 0: coefficient overflow
    return v;
}

// rint(2^p v) (ties to even) as a 32-bit coefficient; sets *flag when it does not fit (NaN included).
__device__ __forceinline__ int fixed_coeff(float v, int p, int *flag)
{
    const double x = nearbyint(ldexp((double)v, p));
    if (fabs(x) < 2147483648.0) return (int)x;
    atomicExch(flag, 1);
    return 0;
}

// A_B = rint(2^p B_k) of every channel.
__global__ void pack_center_kernel(const float *__restrict__ center, int C, int p, PackView v)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < C) v.center[k] = fixed_coeff(center[k], p, v.flag);
}

// A = rint(2^p s) (ties to even) and the bf16 codes of every packed row.
__global__ void pack_kernel(const int8_t *__restrict__ codes, const float *__restrict__ scales,
                            int C, int d, int d_pad, int k_max, int p, int rows, PackView v)
{
    const int r = blockIdx.x;
    const int k = v.chan[r], i = v.point[r];
    const bool live = k >= 0 && i >= 0 && MPQ_IN(k, C) && MPQ_IN(i, k_max);
    if (threadIdx.x == 0) v.coef[r] = live ? fixed_coeff(scales[(size_t)k * k_max + i], p, v.flag) : 0;
    const int8_t *q = live ? codes + (size_t)i * C * d + (size_t)k * d : nullptr;
    for (int j = threadIdx.x; j < d_pad; j += blockDim.x)
        v.codes[(size_t)r * d_pad + j] = __float2bfloat16_rn(live && j < d ? (float)q[j] : 0.0f);
}

// Four int8 (a word) as bf16 pairs, exact: 0x4300 | (v & 0x7F) is 128 + (v & 0x7F), and 0x4300 |
// (v & 0x80) is 128, or 256 for a negative v.
__device__ __forceinline__ void bf16x4_from_int8(uint32_t v, uint32_t &lo, uint32_t &hi)
{
    auto pair = [](uint32_t h) -> uint32_t {
        const uint32_t a = h & 0x437F437Fu, b = h & 0x43804380u;
        const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162 *>(&a),
                                         *reinterpret_cast<const __nv_bfloat162 *>(&b));
        return *reinterpret_cast<const uint32_t *>(&d);
    };
    lo = pair(__byte_perm(v, 0x43434343u, 0x4140u));
    hi = pair(__byte_perm(v, 0x43434343u, 0x4342u));
}

// A role's place in a ring of N slots: slot and phase parity, `step` slots further at a time.
template <int N>
struct RingAt {
    int slot = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ explicit RingAt(int first = 0) : slot(first) {}
    __device__ __forceinline__ void advance(int step = 1)
    {
        slot += step;
        if (slot >= N) {
            slot -= N;
            ph ^= 1u;
        }
    }
};

// Work: (pair of row tiles, input tile) units, and after the first `full` of them parts of L_N / cut
// inputs of the rest (lin_schedule).
struct LinWork {
    long long full, units;   // whole units, and units in all
    int cut, n_in;           // parts of each of the rest; input tiles
    struct Unit {
        int tile, n0, width; // pair of row tiles, first input, inputs
    };
    __device__ __forceinline__ Unit at(long long u) const
    {
        long long v = u;
        int part = 0, width = L_N;
        if (u >= full) {
            v = full + (u - full) / cut;
            part = (int)((u - full) % cut);
            width = L_N / cut;
        }
        return {(int)(v / n_in), (int)(v % n_in) * L_N + part * width, width};
    }
};

__global__ void __launch_bounds__(L_THREADS, 1)
multipoint_linear_kernel(int T, int C, int tiles, const LinWork work, int n_kc, int p,
                         const int *__restrict__ coef, const int *__restrict__ chan,
                         const int *__restrict__ tile_R, const int *__restrict__ center_coef,
                         int32_t *__restrict__ Y, const WaitCtl wc,
                         const __grid_constant__ CUtensorMap tmA,
                         const __grid_constant__ CUtensorMap tmX)
{
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw_u32 = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw_u32 & 1023u)) & 1023u;
    LinCtrl &ctl = *reinterpret_cast<LinCtrl *>(smem_raw + pad);
    unsigned char *ring = smem_raw + pad + L_CTRL_BYTES;
    const uint32_t a_u32 = raw_u32 + pad + L_CTRL_BYTES;
    const uint32_t b_u32 = a_u32 + L_OFF_B, x_u32 = a_u32 + L_OFF_RAW;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = (int)cluster_ctarank();   // 0: even CTA (issues the MMAs), 1: its peer
    // this pair's units pair0 + i n_pairs; this CTA has row tile 2 tile + half of each
    const int pair0 = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
    const long long mine = (work.units - pair0 + n_pairs - 1) / n_pairs;
    auto width_of = [&](long long i) {   // inputs of this pair's unit i
        return pair0 + i * n_pairs >= work.full ? L_N / work.cut : L_N;
    };
    const long long chunks = mine * n_kc;
    if (!MPQ_CHECK_SMEM_END((size_t)pad + L_CTRL_BYTES + (size_t)L_BYTES)) return;

    if (threadIdx.x == 0) {
        for (int i = 0; i < L_SLOTS; ++i) {
            mbar_init(&ctl.a_full[i], 1);
            mbar_init(&ctl.full[i], 2 * L_GROUP_WARPS);
            mbar_init(&ctl.empty[i], 1);
        }
        for (int i = 0; i < L_R_SLOTS; ++i) {
            mbar_init(&ctl.r_full[i], 1);
            mbar_init(&ctl.r_empty[i], L_GROUP_WARPS);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&ctl.acc_full[i], 1);
            mbar_init(&ctl.acc_empty[i], 2 * L_EPI_WARPS);
            mbar_init(&ctl.xs_ready[i], 2 * L_PROD_WARPS);
            mbar_init(&ctl.xs_empty[i], 2 * L_EPI_WARPS);
        }
        mbar_init(&ctl.done, 1);
        ctl.abort = 0;
        fence_barrier_init();
    }
    if (warp == L_MMA_WARP) {
        tmem_alloc_pair(&ctl.tmem_base, 2 * L_N);
        tc_fence_before();
    }
    cluster_sync();   // barriers of both CTAs initialised, TMEM allocated
    tc_fence_after();
    const uint32_t tmem = ctl.tmem_base;
    volatile int *abort_flag = &ctl.abort;

    const bool centered = center_coef != nullptr;
    if (warp < L_PROD_WARPS) {
        // ---------------------------------------------------------------- producers: int8 -> bf16
        // group `grp` takes chunks grp, grp + 2, .. of the CTA's whole sequence
        constexpr int ITEMS = L_IN * (L_KC / 16) / L_GROUP_THREADS;
        const int grp = warp / L_GROUP_WARPS, pt = threadIdx.x % L_GROUP_THREADS;
        int xs[ITEMS];   // this thread's 16-byte share of each input row's sum
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) xs[it] = 0;
        bool run = true;
        RingAt<L_R_SLOTS> ra(grp);
        RingAt<L_SLOTS> at(grp);
        int kc = grp;   // chunk of the unit
        for (long long u = 0; u < mine && run; ++u, kc -= n_kc) {
            const int rows = width_of(u) / 2;   // input rows of this CTA, 32 an item
            for (; kc < n_kc; kc += L_GROUPS) {
                const int rs = ra.slot, sl = at.slot;
                // (a fresh barrier's wait for the phase before its first returns at once)
                bool ok = mbar_wait(&ctl.r_full[rs], ra.ph, wc.budget) &&
                          mbar_wait_cluster(&ctl.empty[sl], at.ph ^ 1u, wc.budget);
                if (!ok) {
                    *abort_flag = 1;
                    note_timeout(wc, MPQ_TIMEOUT_INFERENCE);
                }
                if (__any_sync(0xffffffffu, !ok || *abort_flag)) {   // warp-uniform
                    run = false;
                    break;
                }
                // 16 input bytes (one input row, 16 K elements) per item, 4 items per thread: all
                // reads first, then the raw slot goes back to the TMA thread
                float4 raw[ITEMS];
#pragma unroll
                for (int it = 0; it < ITEMS; ++it)
                    if (it * 32 < rows)
                        raw[it] = ld_shared_v4(x_u32 + rs * L_RAW_BYTES +
                                               (uint32_t)(pt + it * L_GROUP_THREADS) * 16u);
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl.r_empty[rs]);
                const uint32_t bb = b_u32 + sl * L_B_BYTES;
#pragma unroll
                for (int it = 0; it < ITEMS; ++it) {
                    if (it * 32 >= rows) break;
                    const int q = pt + it * L_GROUP_THREADS;
                    const int row = q >> 2, c16 = q & 3;
                    const uint32_t w[4] = {__float_as_uint(raw[it].x), __float_as_uint(raw[it].y),
                                           __float_as_uint(raw[it].z), __float_as_uint(raw[it].w)};
                    if (centered) {   // signed bytes summed exactly (|sum| <= 128 d)
#pragma unroll
                        for (int i = 0; i < 4; ++i) xs[it] = __dp4a((int)w[i], 0x01010101, xs[it]);
                    }
                    uint32_t o[8];
#pragma unroll
                    for (int i = 0; i < 4; ++i) bf16x4_from_int8(w[i], o[2 * i], o[2 * i + 1]);
                    st_shared_v4(bb + sw128_offset(row, 2 * c16),
                                 make_float4(__uint_as_float(o[0]), __uint_as_float(o[1]),
                                             __uint_as_float(o[2]), __uint_as_float(o[3])));
                    st_shared_v4(bb + sw128_offset(row, 2 * c16 + 1),
                                 make_float4(__uint_as_float(o[4]), __uint_as_float(o[5]),
                                             __uint_as_float(o[6]), __uint_as_float(o[7])));
                }
                fence_proxy_async_smem();
                // the chunk's codes tile has landed too before the slot is reported full
                ok = mbar_wait(&ctl.a_full[sl], at.ph, wc.budget);
                if (!ok) {
                    *abort_flag = 1;
                    note_timeout(wc, MPQ_TIMEOUT_INFERENCE);
                }
                if (__any_sync(0xffffffffu, !ok || *abort_flag)) {
                    run = false;
                    break;
                }
                if (lane == 0) mbar_arrive_cluster(&ctl.full[sl], 0);
                ra.advance(L_GROUPS);
                at.advance(L_GROUPS);
            }
            if (centered && run) {
                // both epilogues are done with the sums of two units ago; the 4 threads of an input
                // row (lanes 4m..4m+3) hold its 4 column shares, which both CTAs need
                const int b = (int)(u & 1);
                bool ok = u < 2 || mbar_wait_cluster(&ctl.xs_empty[b], (uint32_t)(u / 2 - 1) & 1u,
                                                     wc.budget);
                if (!ok) {
                    *abort_flag = 1;
                    note_timeout(wc, MPQ_TIMEOUT_INFERENCE);
                }
                run = !__any_sync(0xffffffffu, !ok || *abort_flag);
#pragma unroll
                for (int it = 0; it < ITEMS; ++it) {
                    int v = xs[it];
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    const int row = (pt + it * L_GROUP_THREADS) >> 2;
                    int *at = &ctl.xsum[b][grp][(half * rows + row) % L_N];
                    if (run && (lane & 3) == 0 && row < rows) {
                        st_dsmem_u32(at, 0, (uint32_t)v);
                        st_dsmem_u32(at, 1, (uint32_t)v);
                    }
                    xs[it] = 0;
                }
                fence_cluster();   // the warp's stores, then one arrival for it
                __syncwarp();
                if (lane == 0 && run) {
                    mbar_arrive_release_cluster(&ctl.xs_ready[b], 0);
                    mbar_arrive_release_cluster(&ctl.xs_ready[b], 1);
                }
            }
        }
    } else if (warp < L_MMA_WARP) {
        // ---------------------------------------------------------------- epilogue
        const int ew = warp - L_EPI_WARP0, q = ew & 3, h = ew >> 2;
        int (*out)[L_OUT_COLS + 1] =
            reinterpret_cast<int (*)[L_OUT_COLS + 1]>(ring + L_OFF_OUT) + ew * 32;
        const bool wide = (T & 3) == 0 && ((uintptr_t)Y & 15) == 0;   // 16-byte stores
        for (long long i = 0; i < mine; ++i) {
            const LinWork::Unit un = work.at(pair0 + i * (long long)n_pairs);
            const int hw = un.width / 2;      // columns of a half
            const int tile = un.tile * 2 + half, n0 = un.n0 + h * hw;
            const int b = (int)(i & 1);
            const bool real = tile < tiles;   // (an odd last tile's pair has no second one)
            const int R = real ? tile_R[tile] : 1;
            const int r = q * 32 + lane;
            const int k = real ? chan[(size_t)tile * L_M + r] : -1;
            const long long a = real ? coef[(size_t)tile * L_M + r] : 0;
            const long long ab =
                centered && k >= 0 && MPQ_IN(k, C) ? (long long)center_coef[k] : 0;
            bool ok = mbar_wait_cluster(&ctl.acc_full[b], (uint32_t)(i / 2) & 1u, wc.budget);
            if (ok && centered)
                ok = mbar_wait_cluster(&ctl.xs_ready[b], (uint32_t)(i / 2) & 1u, wc.budget);
            if (!ok) {
                *abort_flag = 1;
                note_timeout(wc, MPQ_TIMEOUT_INFERENCE);
            }
            if (__any_sync(0xffffffffu, !ok || *abort_flag)) break;   // warp-uniform
            tc_fence_after();
            const uint32_t lane_base =
                tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * L_N + h * hw);
            // the rows this warp writes: one per channel (its first lane), -1 for none
            const int kw = (lane & (R - 1)) == 0 ? k : -1;
            ctl.kch[ew][lane] = kw;
            __syncwarp();
#pragma unroll 1
            for (int cb = 0; real && cb < hw / 16 && n0 + cb * 16 < T; ++cb) {
                float v[16];
                tmem_ld_32x32b_x16(lane_base + (uint32_t)(cb * 16), v);
                long long sum[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) sum[j] = a * (long long)__float2int_rz(v[j]);
                for (int o = 1; o < R; o <<= 1) {   // the channel's R lanes (R-aligned)
#pragma unroll
                    for (int j = 0; j < 16; ++j) sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], o);
                }
                if (centered) {   // the row sums first: no shared-memory store comes before them
                    const int *xa = ctl.xsum[b][0] + h * hw + cb * 16;
                    const int *xb = ctl.xsum[b][1] + h * hw + cb * 16;
#pragma unroll
                    for (int j = 0; j < 16; ++j) sum[j] += ab * (long long)(xa[j] + xb[j]);
                }
                int zr[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    long long z = sum[j] >> p;   // arithmetic shift: floor division by 2^p
                    z = z > 2147483647LL ? 2147483647LL : (z < -2147483648LL ? -2147483648LL : z);
                    zr[j] = (int)z;
                }
                const int t0 = n0 + cb * 16;
                if (wide) {
                    // each channel's lane stores its 16 consecutive outputs itself: no exchange
                    // (and no waits on one) between the accumulator and memory
                    if (kw >= 0 && MPQ_IN(kw, C)) {
                        int32_t *y = Y + (size_t)kw * T + t0;
#pragma unroll
                        for (int j = 0; j < 16; j += 4)
                            if (t0 + j < T)
                                *reinterpret_cast<int4 *>(y + j) =
                                    make_int4(zr[j], zr[j + 1], zr[j + 2], zr[j + 3]);
                    }
                    continue;
                }
#pragma unroll
                for (int c0 = 0; c0 < 16; c0 += L_OUT_COLS) {
#pragma unroll
                    for (int j = 0; j < L_OUT_COLS; ++j) out[lane][j] = zr[c0 + j];
                    __syncwarp();
                    // four rows' 8 consecutive outputs per store (32-byte sectors); every
                    // shared-memory read is issued before the first store
                    const int t = t0 + c0 + (lane & 7);
                    int kv[8], ov[8];
#pragma unroll
                    for (int L = 0; L < 8; ++L) {
                        kv[L] = ctl.kch[ew][L * 4 + (lane >> 3)];
                        ov[L] = out[L * 4 + (lane >> 3)][lane & 7];
                    }
                    __syncwarp();
                    if (t < T) {
#pragma unroll
                        for (int L = 0; L < 8; ++L)
                            if (kv[L] >= 0 && MPQ_IN(kv[L], C)) Y[(size_t)kv[L] * T + t] = ov[L];
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive_cluster(&ctl.acc_empty[b], 0);
                if (centered) {
                    mbar_arrive_cluster(&ctl.xs_empty[b], 0);
                    mbar_arrive_cluster(&ctl.xs_empty[b], 1);
                }
            }
        }
    } else if (warp == L_MMA_WARP) {
        // ---------------------------------------------------------------- MMA issuer
        if (lane == 0 && half == 0) {
            uint32_t idesc = idesc_bf16(2 * L_M, width_of(0));
            long long i = 0;
            int kc = 0;
            RingAt<2> acc;
            RingAt<L_SLOTS> at;
            for (long long c = 0; c < chunks && !*abort_flag; ++c) {
                const int sl = at.slot, b = acc.slot;
                bool ok = true;
                if (kc == 0)   // the epilogues have read this accumulator
                    ok = mbar_wait_cluster(&ctl.acc_empty[b], acc.ph ^ 1u, wc.budget);
                if (ok) ok = mbar_wait_cluster(&ctl.full[sl], at.ph, wc.budget);
                if (!ok) {
                    *abort_flag = 1;
                    note_timeout(wc, MPQ_TIMEOUT_INFERENCE);
                    break;
                }
                tc_fence_after();
                const uint64_t bd = smem_desc_sw128(b_u32 + sl * L_B_BYTES);
                const uint64_t ad = smem_desc_sw128(a_u32 + sl * L_A_BYTES);
#pragma unroll
                for (int kk = 0; kk < L_KC / 16; ++kk) {
                    const uint64_t o = (uint64_t)(kk * 2);   // 32 bytes, in 16 B units
                    mma_f16_pair(tmem + (uint32_t)(b * L_N), ad + o, bd + o, idesc,
                             (kc > 0 || kk > 0) ? 1u : 0u);
                }
                mma_commit_pair(&ctl.empty[sl], 3);
                if (++kc == n_kc) {
                    mma_commit_pair(&ctl.acc_full[b], 3);
                    kc = 0;
                    acc.advance();
                    idesc = idesc_bf16(2 * L_M, width_of(++i));
                }
                at.advance();
            }
            // every MMA issued above completes before tensor memory is released
            mma_commit_pair(&ctl.done, 1);
            drain_wait_cluster(&ctl.done, 0, wc, MPQ_TIMEOUT_INFERENCE);
        }
        __syncwarp();
    } else if (warp == L_TMA_A_WARP) {
        // ---------------------------------------------------------------- TMA: codes tiles
        if (lane == 0) {
            prefetch_tensormap(&tmA);
            long long issued = 0;
            long long u = pair0;
            int kc = 0, tile = work.at(u).tile * 2 + half;
            RingAt<L_SLOTS> aa;
            for (long long c = 0; c < chunks; ++c) {
                const int as = aa.slot;
                if (!mbar_wait_cluster(&ctl.empty[as], aa.ph ^ 1u, wc.budget)) {
                    *abort_flag = 1;
                    note_timeout(wc, MPQ_TIMEOUT_INFERENCE);
                }
                if (*abort_flag) break;
                // 16-byte aligned tile copies (bf16 codes: x a multiple of 8)
                if (!MPQ_CHECK(((kc * L_KC) & 7) == 0 && ((a_u32 + as * L_A_BYTES) & 1023u) == 0u)) {
                    *abort_flag = 1;
                    break;
                }
                mbar_arrive_expect_tx(&ctl.a_full[as], (uint32_t)L_A_BYTES);
                tma_load_2d(a_u32 + as * L_A_BYTES, &tmA, kc * L_KC, tile * L_M, &ctl.a_full[as]);
                issued = c + 1;
                aa.advance();
                if (++kc == n_kc) {
                    kc = 0;
                    u += n_pairs;
                    tile = work.at(u).tile * 2 + half;
                }
            }
            // no copy may land after the CTA is gone
            for (long long c = issued - L_SLOTS > 0 ? issued - L_SLOTS : 0; c < issued; ++c)
                drain_wait(&ctl.a_full[c % L_SLOTS], (uint32_t)(c / L_SLOTS) & 1u, wc,
                           MPQ_TIMEOUT_INFERENCE);
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- TMA: raw input tiles
        if (lane == 0) {
            prefetch_tensormap(&tmX);
            long long issued = 0, u = pair0;
            auto row0 = [&](long long v) {   // this CTA's first input row (a box holds a whole unit's)
                const LinWork::Unit un = work.at(v);
                return un.n0 + half * (un.width / 2);
            };
            int kc = 0, n0 = row0(u);
            RingAt<L_R_SLOTS> ra;
            for (long long c = 0; c < chunks; ++c) {
                const int rs = ra.slot;
                if (!mbar_wait(&ctl.r_empty[rs], ra.ph ^ 1u, wc.budget)) {
                    *abort_flag = 1;
                    note_timeout(wc, MPQ_TIMEOUT_INFERENCE);
                }
                if (*abort_flag) break;
                // 16-byte aligned tile copies (int8 inputs: x a multiple of 16)
                if (!MPQ_CHECK(((kc * L_KC) & 15) == 0 && ((x_u32 + rs * L_RAW_BYTES) & 127u) == 0u)) {
                    *abort_flag = 1;
                    break;
                }
                mbar_arrive_expect_tx(&ctl.r_full[rs], (uint32_t)L_RAW_BYTES);
                tma_load_2d(x_u32 + rs * L_RAW_BYTES, &tmX, kc * L_KC, n0, &ctl.r_full[rs]);
                issued = c + 1;
                ra.advance();
                if (++kc == n_kc) {
                    kc = 0;
                    u += n_pairs;
                    n0 = row0(u);
                }
            }
            for (long long c = issued - L_R_SLOTS > 0 ? issued - L_R_SLOTS : 0; c < issued; ++c)
                drain_wait(&ctl.r_full[c % L_R_SLOTS], (uint32_t)(c / L_R_SLOTS) & 1u, wc,
                           MPQ_TIMEOUT_INFERENCE);
        }
        __syncwarp();
    }

    cluster_sync();   // nothing of the pair's is in flight (every MMA was drained above)
    if (warp == L_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, 2 * L_N);
    }
}

// ---- a few inputs, or rows and layers the kernel above cannot take ----------------------------
constexpr int S_WARPS = 8;
// a warp accumulates at most an eighth of the longest row in fp32: 1,024 x 127 x 128 < 2^24, exact
static_assert((MPQ_MAX_DIM / S_WARPS) * 127LL * 128 < (1LL << 24), "exact fp32 sums");

// 8 inputs from byte p on, of which `avail` (> 0) are the row's: 0 past them.  Aligned: p is a
// multiple of 8 and so is the row.  Else the aligned words that hold them, shifted together (a
// word is read only where it holds one of them).
template <bool ALIGNED>
__device__ __forceinline__ uint2 load_int8x8(const int8_t *p, int avail)
{
    if constexpr (ALIGNED) return __ldg(reinterpret_cast<const uint2 *>(p));
    const uintptr_t a = reinterpret_cast<uintptr_t>(p), end = a + min(avail, 8);
    const uint32_t *w = reinterpret_cast<const uint32_t *>(a & ~(uintptr_t)3);
    const int sh = (int)(a & 3) * 8;
    const uint32_t w0 = __ldg(w);
    const uint32_t w1 = reinterpret_cast<uintptr_t>(w + 1) < end ? __ldg(w + 1) : 0u;
    const uint32_t w2 = reinterpret_cast<uintptr_t>(w + 2) < end ? __ldg(w + 2) : 0u;
    uint2 v = make_uint2(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh));
    if (avail < 8) {
        if (avail < 4) v.x &= (1u << (8 * avail)) - 1u;
        v.y = avail <= 4 ? 0u : v.y & ((1u << (8 * (avail - 4))) - 1u);
    }
    return v;
}

__device__ __forceinline__ void mma_bf16_16x8x16(float (&c)[4], uint32_t a0, uint32_t a1,
                                                 uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// 16 MT packed rows x 8 NT inputs per CTA.  Lane (g, t) = (lane / 4, lane % 4) of a warp holds 8
// consecutive K elements of code rows g and g + 8 and of input g: the MMAs' K index is a
// permutation of the elements, the same for both operands (32 elements are two MMAs).
template <int MT, int NT, bool ALIGNED>
__global__ void __launch_bounds__(S_WARPS * 32, MT * NT <= 4 ? 3 : 2)
multipoint_mma_kernel(const int8_t *__restrict__ X, int T, int C, int d, int d_pad, int n_blocks,
                      int p, const int *__restrict__ coef, const int *__restrict__ chan,
                      const __nv_bfloat16 *__restrict__ codes, const int *__restrict__ tile_R,
                      const int *__restrict__ center_coef, int32_t *__restrict__ Y)
{
    constexpr int ROWS = 16 * MT, INS = 8 * NT;
    extern __shared__ int red[];                     // [S_WARPS][ROWS][INS]
    __shared__ int xsum[S_WARPS][INS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    // input blocks vary fastest: the CTAs that share code rows run together
    const int row0 = (int)(blockIdx.x / (unsigned)n_blocks) * ROWS;
    const int n0 = (int)(blockIdx.x % (unsigned)n_blocks) * INS;
    const int n_kc = d_pad / L_KC;
    const bool centered = center_coef != nullptr;
    if (!MPQ_CHECK_SMEM_END(sizeof(int) * S_WARPS * ROWS * INS)) return;

    float acc[MT][NT][4];
    int xs[NT];
#pragma unroll
    for (int n = 0; n < NT; ++n) {
        xs[n] = 0;
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.0f;
    }
    const __nv_bfloat16 *qrow = codes + (size_t)(row0 + g) * d_pad;
#pragma unroll(MT * NT == 1 ? 4 : (MT * NT == 2 ? 2 : 1))
    for (int kc = warp; kc < n_kc; kc += S_WARPS) {
        uint4 a[2][MT][2];
        uint2 x[2][NT];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = kc * L_KC + h * 32 + 8 * t;
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    a[h][m][r] = __ldg(reinterpret_cast<const uint4 *>(
                        qrow + (size_t)(m * 16 + r * 8) * d_pad + k));
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                const int in = n0 + n * 8 + g;
                x[h][n] = make_uint2(0u, 0u);
                if (in < T && k < d) x[h][n] = load_int8x8<ALIGNED>(X + (size_t)in * d + k, d - k);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                uint32_t b0, b1, b2, b3;
                bf16x4_from_int8(x[h][n].x, b0, b1);
                bf16x4_from_int8(x[h][n].y, b2, b3);
                if (centered)   // signed bytes summed exactly
                    xs[n] = __dp4a((int)x[h][n].y, 0x01010101, __dp4a((int)x[h][n].x, 0x01010101, xs[n]));
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const uint4 u = a[h][m][0], v = a[h][m][1];
                    mma_bf16_16x8x16(acc[m][n], u.x, v.x, u.y, v.y, b0, b1);
                    mma_bf16_16x8x16(acc[m][n], u.z, v.z, u.w, v.w, b2, b3);
                }
            }
    }
    int *mine = red + (size_t)warp * ROWS * INS;
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                mine[(m * 16 + g + (e >> 1) * 8) * INS + n * 8 + 2 * t + (e & 1)] =
                    __float2int_rz(acc[m][n][e]);
    if (centered) {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            int v = xs[n];
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if (t == 0) xsum[warp][n * 8 + g] = v;
        }
    }
    __syncthreads();
    // steps 2 and 3: a thread per (channel, input)
    const int R = tile_R[row0 / L_M];   // divides 16: a channel's rows are in one CTA
    for (int i = threadIdx.x; i < ROWS / R * INS; i += S_WARPS * 32) {
        const int row = i / INS * R, n = i % INS;
        const int k = chan[row0 + row];
        if (k < 0 || n0 + n >= T || !MPQ_IN(k, C)) continue;
        long long sum = 0;
        for (int j = 0; j < R; ++j) {
            int dot = 0;   // below 2^27
#pragma unroll
            for (int w = 0; w < S_WARPS; ++w) dot += red[((size_t)w * ROWS + row + j) * INS + n];
            sum += (long long)coef[row0 + row + j] * (long long)dot;
        }
        if (centered) {
            long long v = 0;
            for (int w = 0; w < S_WARPS; ++w) v += xsum[w][n];
            sum += (long long)center_coef[k] * v;
        }
        long long z = sum >> p;   // arithmetic shift: floor division by 2^p
        z = z > 2147483647LL ? 2147483647LL : (z < -2147483648LL ? -2147483648LL : z);
        Y[(size_t)k * T + n0 + n] = (int32_t)z;
    }
}

// Which kernel takes a layer the tensor-memory kernel can take: the one whose modelled time is less,
// in microseconds, fitted to both on layers of 64 x 576 to 11008 x 4096 with 1 to 2,048 inputs
// (within some 15 %).  Here: waves of resident blocks, each a fixed cost and one per K chunk; there:
// a fixed cost and lin_schedule's time of a chunk over the rounds.  4096 x 4096 at 8 / 64 / 128 / 256 /
// 2,048 inputs: 7.4 / 25.6 / 38.7 / 66.5 / 485 us here, 32.9 / 34.7 / 37.0 / 34.5 / 98 there.
struct LinSchedule {
    long long full, units;
    int cut;
    double chunk_us;   // modelled time of a K chunk, over the rounds
};

// The last round of units leaves pairs idle: what is beyond whole rounds is cut into 1, 2 or 4 parts
// by its inputs, whichever takes the least.  A chunk of a half or quarter takes 0.36 and 0.35 us: its
// codes tile and hand-overs stay (a smaller box for its inputs changes nothing).  4096 x 4096 at 256 /
// 1,024 / 2,048 inputs (21, 84, 168 units on 76 pairs) 39.4 / 72.6 / 105 -> 34.5 / 65 / 98 us, 11008 x
// 4096 at 512 73.5 -> 67.8.
LinSchedule lin_schedule(long long units, long long pairs)
{
    const double part_us[3] = {0.45, 0.36, 0.35};
    const long long rest = units % pairs;
    LinSchedule s = {units, units, 1, part_us[0] * (double)((units + pairs - 1) / pairs)};
    for (int i = 1; i < 3 && rest > 0; ++i) {
        const int cut = 1 << i;
        const double t = part_us[0] * (double)(units / pairs) +
                         part_us[i] * (double)((rest * cut + pairs - 1) / pairs);
        if (t < s.chunk_us) s = {units - rest, units - rest + rest * cut, cut, t};
    }
    return s;
}

bool few_inputs(const mpq_packed_layout *L, int T)
{
    const double n_kc = L->d_pad / L_KC, sms = sm_count();
    double blocks, per_sm, wave;
    if (T <= 32) {
        blocks = L->rows / 16;
        per_sm = 3.0;
        wave = T <= 8 ? 2.0 + 0.12 * n_kc : (T <= 16 ? 2.0 + 0.15 * n_kc : 3.0 + 0.21 * n_kc);
    } else {
        blocks = L->rows / 32 * floor((T + 31.0) / 32);
        per_sm = 2.0;
        wave = 4.5 + 0.15 * n_kc;
    }
    const long long units = (L->tiles + 1LL) / 2 * (((long long)T + L_N - 1) / L_N);
    const double here = ceil(blocks / (per_sm * sms)) * wave;
    const double there = 10.0 + n_kc * lin_schedule(units, std::max(1, sm_count() / 2)).chunk_us;
    return here <= there;
}

template <int MT, int NT>
mpq_status launch_mma(const int8_t *X, int T, const mpq_packed_layout *L, const PackView &v,
                      int32_t *Y, cudaStream_t stream)
{
    const bool aligned = L->d % 8 == 0 && (uintptr_t)X % 8 == 0;
    auto kernel = aligned ? multipoint_mma_kernel<MT, NT, true> : multipoint_mma_kernel<MT, NT, false>;
    const int smem = (int)sizeof(int) * S_WARPS * 16 * MT * 8 * NT;
    static std::atomic<int> limit[2][kMaxDevices];
    const cudaError_t e = allow_smem(reinterpret_cast<const void *>(kernel), limit[aligned], smem);
    if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute");
    const long long n_blocks = ((long long)T + 8 * NT - 1) / (8 * NT);
    const long long blocks = n_blocks * (L->rows / (16 * MT));
    if (blocks > 0x7FFFFFFFLL) {
        set_error("multipoint linear: %lld blocks", blocks);
        return MPQ_ERR_UNSUPPORTED;
    }
    kernel<<<(unsigned)blocks, S_WARPS * 32, smem, stream>>>(X, T, L->C, L->d, L->d_pad, (int)n_blocks,
                                                             L->p, v.coef, v.chan, v.codes, v.tile_R,
                                                             v.center, Y);
    return cuda_status(cudaGetLastError(), "multipoint linear kernel launch");
}

PFN_cuTensorMapEncodeTiled_v12000 lin_map_encoder()
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

int pow2_at_least(int n)
{
    int r = 1;
    while (r < n) r <<= 1;
    return r;
}

}  // namespace

mpq_status make_pack_layout(const int *npoints, int C, int d, int k_max, int bits, int p,
                            int centered, mpq_packed_layout *L)
{
    memset(L, 0, sizeof(*L));
    L->C = C;
    L->d = d;
    L->k_max = k_max;
    L->bits = bits;
    L->p = p;
    L->centered = centered;
    L->d_pad = (d + L_KC - 1) / L_KC * L_KC;
    long long tiles = 0;
    for (int R = 1; R <= MPQ_MAX_POINTS; R <<= 1) {
        long long n = 0;
        for (int k = 0; k < C; ++k) {
            int nk = npoints[k] < 0 ? 0 : (npoints[k] > k_max ? k_max : npoints[k]);
            if (pow2_at_least(nk < 1 ? 1 : nk) == R) ++n;
        }
        tiles += (n + (L_M / R) - 1) / (L_M / R);
    }
    if (tiles * L_M > (1LL << 30)) {
        set_error("packed layer too large");
        return MPQ_ERR_UNSUPPORTED;
    }
    L->tiles = (int)tiles;
    L->rows = (int)(tiles * L_M);
    size_t off = 64;
    L->off_coef = off;
    off += (size_t)L->rows * 4;
    L->off_chan = off;
    off += (size_t)L->rows * 4;
    L->off_point = off;
    off += (size_t)L->rows * 4;
    L->off_tile = off;
    off += (size_t)L->tiles * 4;
    L->off_center = off;
    off += centered ? (size_t)C * 4 : 0;
    off = (off + 1023) / 1024 * 1024;
    L->off_codes = off;
    off += (size_t)L->rows * L->d_pad * 2;
    L->bytes = off;
    return MPQ_OK;
}

mpq_status launch_pack(const int8_t *codes, const float *scales, const float *center,
                       const int *npoints, const mpq_packed_layout *L, void *packed,
                       cudaStream_t stream)
{
    const int C = L->C, rows = L->rows;
    std::vector<int> chan((size_t)rows, -1), point((size_t)rows, -1), tR((size_t)L->tiles, 1);
    int t = 0;
    for (int R = 1; R <= MPQ_MAX_POINTS; R <<= 1) {
        int slot = 0, per = L_M / R;
        for (int k = 0; k < C; ++k) {
            int nk = npoints[k] < 0 ? 0 : (npoints[k] > L->k_max ? L->k_max : npoints[k]);
            if (pow2_at_least(nk < 1 ? 1 : nk) != R) continue;
            if (slot == per) {
                slot = 0;
                ++t;
            }
            tR[(size_t)t] = R;
            for (int i = 0; i < R; ++i) {
                const size_t r = (size_t)t * L_M + (size_t)slot * R + i;
                chan[r] = (i == 0 || i < nk) ? k : -1;   // the first row carries the channel
                point[r] = i < nk ? i : -1;
            }
            ++slot;
        }
        if (slot > 0) ++t;
    }
    if (t != L->tiles) {
        set_error("npoints differ from the ones the layout was made for");
        return MPQ_ERR_INVALID_ARG;
    }
    PackView v = view(L, packed);
    cudaError_t e = cudaMemsetAsync(packed, 0, 64, stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(v.chan, chan.data(), (size_t)rows * 4, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(v.point, point.data(), (size_t)rows * 4, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(v.tile_R, tR.data(), (size_t)L->tiles * 4, cudaMemcpyHostToDevice,
                            stream);
    if (e != cudaSuccess) return cuda_status(e, "packing copies");
    if (rows > 0) {
        pack_kernel<<<rows, 256, 0, stream>>>(codes, scales, C, L->d, L->d_pad, L->k_max, L->p, rows,
                                              v);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_status(e, "pack kernel launch");
    }
    if (L->centered) {
        pack_center_kernel<<<(C + 255) / 256, 256, 0, stream>>>(center, C, L->p, v);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_status(e, "pack center kernel launch");
    }
    int flag = 0;
    e = cudaMemcpyAsync(&flag, v.flag, sizeof(int), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);   // host arrays above must outlive the copies
    if (e != cudaSuccess) return cuda_status(e, "packing");
    if (flag) {
        set_error("a coefficient rint(2^p * s) or rint(2^p * B) does not fit 32 bits (p = %d)", L->p);
        return MPQ_ERR_UNSUPPORTED;
    }
    return MPQ_OK;
}

mpq_status launch_multipoint_linear(const int8_t *X, int T, const mpq_packed_layout *L,
                                    const void *packed, int32_t *Y, cudaStream_t stream)
{
    PackView v = view(L, const_cast<void *>(packed));
    const int d = L->d, qmax = (1 << (L->bits - 1)) - 1;
    const bool exact = (double)d * qmax * 128.0 < 16777216.0;
    const bool tma = exact && d % 16 == 0 && (uintptr_t)X % 16 == 0 && L->rows > 0;
    if (tma && !few_inputs(L, T)) {
        PFN_cuTensorMapEncodeTiled_v12000 enc = lin_map_encoder();
        CUtensorMap tmA, tmX;
        memset(&tmA, 0, sizeof(tmA));
        memset(&tmX, 0, sizeof(tmX));
        const cuuint64_t da[2] = {(cuuint64_t)L->d_pad, (cuuint64_t)L->rows};
        const cuuint64_t sa[1] = {(cuuint64_t)L->d_pad * 2};
        const cuuint32_t ba[2] = {L_KC, L_M};
        const cuuint64_t dx[2] = {(cuuint64_t)d, (cuuint64_t)T};
        const cuuint64_t sx[1] = {(cuuint64_t)d};
        const cuuint32_t bx[2] = {L_KC, L_IN};
        const cuuint32_t es[2] = {1, 1};
        if (!enc ||
            enc(&tmA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, v.codes, da, sa, ba, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
            enc(&tmX, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t *>(X), dx, sx, bx, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            set_error("multipoint linear: tensor map encoding failed");
            return MPQ_ERR_CUDA;
        }
        const long long n_in = ((long long)T + L_N - 1) / L_N;
        const long long units = (L->tiles + 1LL) / 2 * n_in;
        if ((long long)L_SMEM > max_smem_optin()) {
            set_error("multipoint linear needs %d bytes of shared memory", L_SMEM);
            return MPQ_ERR_UNSUPPORTED;
        }
        static std::atomic<int> limit[kMaxDevices];
        const cudaError_t e =
            allow_smem(reinterpret_cast<const void *>(multipoint_linear_kernel), limit, L_SMEM);
        if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute");
        WaitCtl wc;
        const mpq_status wst = wait_ctl(&wc);
        if (wst != MPQ_OK) return wst;
        cudaLaunchConfig_t cfg = {};
        cfg.blockDim = dim3(L_THREADS, 1, 1);
        cfg.dynamicSmemBytes = (size_t)L_SMEM;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        // one resident pair per two SMs, no more than units
        const long long resident = std::max(1, sm_count() / 2);
        const LinSchedule sch = lin_schedule(units, resident);
        const LinWork work = {sch.full, sch.units, sch.cut, (int)n_in};
        const long long pairs = std::min<long long>(resident, sch.units);
        cfg.gridDim = dim3((unsigned)(2 * pairs), 1, 1);
        const cudaError_t el =
            cudaLaunchKernelEx(&cfg, multipoint_linear_kernel, T, L->C, L->tiles, work,
                               L->d_pad / L_KC, L->p, (const int *)v.coef, (const int *)v.chan,
                               (const int *)v.tile_R, (const int *)v.center, Y, wc, tmA, tmX);
        if (el != cudaSuccess) return cuda_status(el, "multipoint linear kernel launch");
        return cuda_status(cudaGetLastError(), "multipoint linear kernel launch");
    }
    if (L->rows == 0) return MPQ_OK;
    if (T <= 8) return launch_mma<1, 1>(X, T, L, v, Y, stream);
    if (T <= 16) return launch_mma<1, 2>(X, T, L, v, Y, stream);
    if (T <= 32) return launch_mma<1, 4>(X, T, L, v, Y, stream);
    return launch_mma<2, 4>(X, T, L, v, Y, stream);
}

}  // namespace mpq
