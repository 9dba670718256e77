// The clipping search's output errors (Sec. 3.3, Eq. 12) on the tensor cores:
//   err[k][c] = (1/N) sum_t (x_t . r_{k,c})^2,  r_{k,c} = w_k - s_{k,c} q_{k,c},
// and the split of X into fp16 planes that the output error of the greedy points uses too.
//
// A CTA-pair contraction Y = R X^T: M = 256 residual vectors (128 per CTA) by N = 256 calibration
// rows per pair tile, each operand scaled by a power of two and split into fp16 hi/lo halves,
// Y = hi*hi + hi*lo + lo*hi on kind::f16 with fp32 accumulation restarted every 256 elements of d,
// the segments added into fp32 running sums, err = mean of Y^2 with the scales undone exactly.
// (The candidates of a channel share no chain of points, and w - s q from products with w and q
// would cancel, so the residuals themselves are the operands.)
//
// * X is scaled and split once per call (f16_split_kernel) into fp16 hi and lo planes in global
//   memory ([2][N][d]), and clip_planes_kernel writes every candidate's residual as such planes;
//   tile copies put each 64-element step straight into the operand tiles (128-byte swizzle).
// * Work advances in steps of 64 elements (one 128-byte row of fp16 per operand row).
// * Resident pairs take units (vector tile, part of its row tiles) in turn, so that pairs at work at
//   the same time share vector tiles (from L2) and none has more than one unit above the mean
//   (20000 vectors, N = 2048: 9 row tiles on the busiest pair; whole vector tiles to clusters of four
//   pairs: 10; 1000 x 2048, N = 2048, 20 candidates 424 -> 343 us with one commit a step for both
//   operands).  A vector tile's parts are summed through global scratch, by the last to
//   arrive, in order.
// * Two accumulators in tensor memory (columns [0, 256) and [256, 512)) take alternate segments,
//   and the running sums live in the epilogue warps' registers (one TMEM lane x 128 columns per
//   thread; setmaxnreg moves registers from warpgroups 0-1 to the epilogue's), so the MMA thread
//   starts the next segment in the other accumulator while the epilogue folds the last one.
// * The tile copies are issued by one epilogue warp, which is idle between its folds.
//
// Warps: 0 relays that a stage's tiles have landed, 7 the MMA issuer (lane 0 of the even CTA),
// 8-15 the epilogue (lane quarter warp % 4, column half; warp 15 also issues this CTA's tile
// copies).  Every wait is bounded; on a timeout the kernel records MPQ_TIMEOUT_CLIP, waits for what
// it issued, and the outputs read NaN.
#include <cuda.h>
#include <cuda_fp16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <atomic>

#include "mpq_internal.cuh"
#include "pair_common.cuh"
#include "slow_channels.cuh"
#include "rounding.cuh"
#include "sm100.cuh"
#include "tf32_operands.cuh"
#include "waits.cuh"

MPQ_CHECKED_UNIT("output_error_f16.cu");

namespace mpq {
namespace {

using namespace sm100;

constexpr int F_VEC = 128;                 // residual vectors per CTA (TMEM lanes)
constexpr int F_ROWS = 128;                // calibration rows per CTA
constexpr int F_N = 2 * F_ROWS;            // rows per pair row tile (UMMA N)
constexpr int F_KS = 64;                   // elements per step: one 128-byte fp16 row
constexpr int F_STAGES = 3;                // operand stages (an A and a B tile set each)
constexpr int F_SEG = 4;                   // steps per accumulation segment (256 elements)
constexpr int F_MMA_WARP = 7;              // MMA issuer
constexpr int F_EPI_WARP0 = 8;             // a multiple of 4: warp % 4 is the TMEM lane quarter
constexpr int F_EPI_WARPS = 8;
constexpr int F_COPY_WARP = 15;            // an epilogue warp that also issues the tile copies
constexpr int F_THREADS = 512;
// registers per thread after setmaxnreg: warpgroups 0-1 (relay, MMA issuer) and 2-3
// (epilogue); together they use exactly what the launch holds (512 threads x 128)
constexpr int F_REGS_LOW = 88;
constexpr int F_REGS_HIGH = 168;
static_assert(256 * F_REGS_LOW + 256 * F_REGS_HIGH == F_THREADS * 128, "register split");
constexpr int F_TILE = 128 * 128;          // 16 KB: 128 rows of 128 bytes (128-byte swizzle)
constexpr int F_SET = 2 * F_TILE;          // hi and lo tiles of one operand stage
constexpr uint32_t F_TMEM_COLS = 512;
constexpr int F_SMEM_LIMIT = 232448;       // opt-in shared memory per CTA on sm_100 parts

struct F16Ctrl {
    uint64_t full[F_STAGES];   // even CTA: both CTAs' relays (A and B landed)
    uint64_t empty[F_STAGES];  // both CTAs: pair MMA commit (stage free)
    uint64_t landed[F_STAGES]; // this CTA's A and B tile copies
    uint64_t segfull[2];       // both CTAs: pair MMA commit, per accumulator
    uint64_t segempty[2];      // even CTA: both CTAs' epilogue warps, per accumulator
    uint64_t done;             // even CTA: every MMA complete
    uint32_t tmem_base;
    int abort;
    int last[2];               // this CTA was the last to leave a tile's sums (alternate units)
    double part[2][F_VEC];     // the upper column half's sums over y^2 (alternate units)
    int xexp;
};
constexpr int F_CTRL_BYTES = (sizeof(F16Ctrl) + 1023) / 1024 * 1024;
constexpr int F_SMEM = 1024 + F_CTRL_BYTES + F_STAGES * 2 * F_SET;
static_assert(F_SMEM <= F_SMEM_LIMIT, "clipping search: shared memory");

// Partial sums of a vector tile's parts, in global scratch, by tile and CTA of the pair: how many
// have arrived (zeroed before the launch), and 2 F_VEC sums per part.
struct ClipScratch {
    unsigned *count;   // [tiles][2]
    double *slot;      // [tiles][parts][2][F_VEC]
};

// C residual vectors, given as fp16 hi/lo planes (tmA: [2][C][d], clip_planes_kernel); vrange: the
// bound on each vector's elements that set its operand scale; xrange[0]: max|X|, both as float
// bits; tmX: the split X planes [2][N][d] fp16.  parts: of a vector tile's row tiles, each one unit.
__global__ void __launch_bounds__(F_THREADS, 1)
clip_error_kernel(int C, int N, int d, const unsigned *__restrict__ xrange,
                  const unsigned *__restrict__ vrange, float *__restrict__ err, int parts,
                  const ClipScratch scratch, const WaitCtl wc,
                  const __grid_constant__ CUtensorMap tmX,
                  const __grid_constant__ CUtensorMap tmA)
{
    constexpr int NS = F_STAGES, SEG = F_SEG;
    constexpr unsigned KBIT = MPQ_TIMEOUT_CLIP;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw_u32 = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw_u32 & 1023u)) & 1023u;
    F16Ctrl &ctl = *reinterpret_cast<F16Ctrl *>(smem_raw + pad);
    const uint32_t a_u32 = raw_u32 + pad + F_CTRL_BYTES;   // stages of an A and a B set

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = (int)cluster_ctarank();         // 0: even CTA (issues the MMAs), 1: its peer
    const uint16_t pair_mask = 3u;
    const int n_rt = (N + F_N - 1) / F_N;
    const int n_ks = (d + F_KS - 1) / F_KS;          // steps per row tile
    const int nseg = (n_ks + SEG - 1) / SEG;
    // this pair's units: every n_pairs-th of (vector tile, part of its row tiles)
    const int pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
    const int units = (C + 2 * F_VEC - 1) / (2 * F_VEC) * parts;
    auto vec0 = [&](int u) { return (u / parts * 2 + half) * F_VEC; };   // this CTA's first vector
    auto rt_lo = [&](int u) { return (int)((long long)n_rt * (u % parts) / parts); };
    auto rt_hi = [&](int u) { return (int)((long long)n_rt * (u % parts + 1) / parts); };
    long long total = 0;                             // steps
    for (int u = pair; u < units; u += n_pairs) total += (long long)(rt_hi(u) - rt_lo(u)) * n_ks;
    // control block and operand tiles within the launch's shared memory (the same in every CTA, so
    // the whole cluster leaves together)
    if (!MPQ_CHECK_SMEM_END((size_t)pad + F_CTRL_BYTES + (size_t)NS * 2 * F_SET)) return;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(&ctl.full[s], 2);
            mbar_init(&ctl.empty[s], 1);
            mbar_init(&ctl.landed[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&ctl.segfull[b], 1);
            mbar_init(&ctl.segempty[b], 2 * F_EPI_WARPS);
        }
        mbar_init(&ctl.done, 1);
        ctl.abort = 0;
        fence_barrier_init();
    }
    if (warp == F_MMA_WARP) {
        tmem_alloc_pair(&ctl.tmem_base, F_TMEM_COLS);
        tc_fence_before();
    }
    griddep_wait();                     // nothing above reads global memory
    if (threadIdx.x == 0) ctl.xexp = f16_scale_exp(__uint_as_float(ld_after_wait(xrange)));
    cluster_sync();                     // barriers of both CTAs initialised, TMEM allocated
    tc_fence_after();
    const uint32_t tmem = ctl.tmem_base;
    volatile int *abort_flag = &ctl.abort;

    // one setmaxnreg per warpgroup: 0-1 (relay, MMA issuer) give registers to 2-3 (epilogue)
    if (warp < F_EPI_WARP0) {
        setmaxnreg_dec<F_REGS_LOW>();
        if (warp == 0) {
            // ------------------------------------------------------------ relay
            // a step's A and B tiles of this CTA have landed: report the stage full
            int s = 0;
            uint32_t ph = 0;
            for (long long it = 0; it < total; ++it) {
                const bool ok = mbar_wait(&ctl.landed[s], ph, wc.budget);
                if (!ok) {
                    *abort_flag = 1;
                    note_timeout(wc, KBIT);
                }
                if (__any_sync(0xffffffffu, !ok || *abort_flag)) break;   // warp-uniform
                if (lane == 0) mbar_arrive_cluster(&ctl.full[s], 0);
                if (++s == NS) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        } else if (warp == F_MMA_WARP && half == 0 && lane == 0) {
            // ------------------------------------------------------------ MMA issuer (even CTA)
            constexpr uint32_t idesc = idesc_f16(2 * F_VEC, F_N);
            bool ok = true;
            // step it = (row tile, step ks), stage s, segment g (accumulator g & 1)
            int ks = 0, s = 0, sk = 0;
            unsigned g = 0;
            uint32_t ph = 0;
            for (long long it = 0; it < total && ok && !*abort_flag; ++it) {
                const bool seg_start = sk == 0;
                const uint32_t b = g & 1u;
                if (seg_start) {
                    // this accumulator's previous segment has been folded by both epilogues
                    if (!mbar_wait_cluster(&ctl.segempty[b], ((g >> 1) & 1u) ^ 1u, wc.budget)) {
                        note_timeout(wc, KBIT);
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                }
                if (!mbar_wait_cluster(&ctl.full[s], ph, wc.budget)) {
                    note_timeout(wc, KBIT);
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t aset = a_u32 + s * 2 * F_SET, bset = aset + F_SET;
                const uint64_t ah = smem_desc_sw128(aset), al = smem_desc_sw128(aset + F_TILE);
                const uint64_t bh = smem_desc_sw128(bset), bl = smem_desc_sw128(bset + F_TILE);
                const uint32_t dt = tmem + b * (F_TMEM_COLS / 2);
                // 64 fp16 elements = four K = 16 steps, 32 bytes apart in the 128-byte rows
                // (16-byte units); per K step the passes lo*hi, hi*lo, hi*hi
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint64_t o = (uint64_t)(kk * 2);
                    mma_f16_pair(dt, al + o, bh + o, idesc, (seg_start && kk == 0) ? 0u : 1u);
                    mma_f16_pair(dt, ah + o, bl + o, idesc, 1u);
                    mma_f16_pair(dt, ah + o, bh + o, idesc, 1u);
                }
                mma_commit_pair(&ctl.empty[s], pair_mask);
                ++ks;
                if (++sk == SEG || ks == n_ks) {
                    mma_commit_pair(&ctl.segfull[b], pair_mask);
                    sk = 0;
                    ++g;
                }
                if (ks == n_ks) ks = 0;
                if (++s == NS) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            if (!ok) *abort_flag = 1;
            // drain: every MMA issued above completes before tensor memory is released
            mma_commit_pair(&ctl.done, (uint16_t)1u);
            drain_wait_cluster(&ctl.done, 0, wc, KBIT);
        }
        __syncwarp();
    } else {
        setmaxnreg_inc<F_REGS_HIGH>();
        // ---------------------------------------------------------------- epilogue
        // lane quarter q (the TMEM lanes this warp may access) and column half h; the running sums
        // of this thread's TMEM lane over the half's 128 columns stay in registers
        const int ew = warp - F_EPI_WARP0, q = ew & 3, h = ew >> 2;
        const int m = q * 32 + lane;                 // this thread's vector of the CTA's
        const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * (F_N / 2));
        float sums[F_N / 2];
        // Warp F_COPY_WARP also issues the CTA's tile copies, step by step: A and B tiles of step f
        // once the MMAs of the step that held their stage have completed.  It goes on copying until
        // the next segment has ended, then folds it like the other epilogue warps (a segment ends
        // every SEG steps, and its fold is needed only SEG steps later, when its accumulator is
        // taken again).
        const bool copier = warp == F_COPY_WARP && wc.withhold == 0;
        long long next = 0, issued = 0;
        int cks = 0, cu = pair, crt = rt_lo(pair), cs = 0;   // step, unit, row tile, stage to copy
        uint32_t cph = 1;
        if (copier && lane == 0) {
            prefetch_tensormap(&tmX);
            prefetch_tensormap(&tmA);
        }
        unsigned g = 0;             // segment
        int un = 0;                 // units done
        bool stop = false;          // given up: no more waits, sums are NaN (warp-uniform)
        for (int u = pair; u < units; u += n_pairs, ++un) {
            double acc = 0.0;
            for (int rt = rt_lo(u); rt < rt_hi(u) && !stop; ++rt) {
                // a row tile's sums start from zero (0 + v = v, up to the sign of a zero, which the
                // squares below do not see)
#pragma unroll
                for (int i = 0; i < F_N / 2; ++i) sums[i] = 0.0f;
                for (int sg = 0; sg < nseg; ++sg, ++g) {
                    const uint32_t b = g & 1u, par = (g >> 1) & 1u;
                    bool ok = true;
                    if (copier) {
                        while (next < total) {
                            if (lane == 0) {
                                const int x = cks * F_KS;
                                const uint32_t adst = a_u32 + cs * 2 * F_SET;
                                // a tile copy starts 16-byte aligned (fp16 elements) into a
                                // 1024-byte aligned destination (128-byte swizzle), or is not
                                // issued and the launch ends through the bounded waits
                                ok = MPQ_CHECK((x & 7) == 0 && (adst & 1023u) == 0u && x < d);
                                if (ok && next >= NS)
                                    ok = mbar_wait_cluster(&ctl.empty[cs], cph, wc.budget);
                                if (ok) {
                                    mbar_arrive_expect_tx(&ctl.landed[cs], 4 * F_TILE);
                                    tma_load_3d(adst, &tmA, x, vec0(cu), 0, &ctl.landed[cs]);
                                    tma_load_3d(adst + F_SET, &tmX, x, crt * F_N + half * F_ROWS, 0,
                                                &ctl.landed[cs]);
                                    issued = next + 1;
                                }
                            }
                            ++next;
                            if (++cks == n_ks) {
                                cks = 0;
                                if (++crt == rt_hi(cu) && (cu += n_pairs) < units) crt = rt_lo(cu);
                            }
                            if (++cs == NS) {
                                cs = 0;
                                cph ^= 1u;
                            }
                            ok = __shfl_sync(0xffffffffu, ok, 0);
                            if (!ok) break;
                            // stop copying once segment g has ended
                            const bool ended = mbar_test_cluster(&ctl.segfull[b], par);
                            if (__shfl_sync(0xffffffffu, ended, 0)) break;
                        }
                    }
                    ok = ok && mbar_wait_cluster(&ctl.segfull[b], par, wc.budget);
                    if (!ok) {
                        *abort_flag = 1;
                        note_timeout(wc, KBIT);
                    }
                    stop = __any_sync(0xffffffffu, !ok || *abort_flag);
                    if (stop) break;
                    // fold segment g (accumulator b) into the sums
                    tc_fence_after();
#pragma unroll
                    for (int cb = 0; cb < F_N / 64; ++cb) {
                        float v[32];
                        tmem_ld_32x32b_x32(lane_base + b * (F_TMEM_COLS / 2) + (uint32_t)(cb * 32), v);
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            sums[cb * 32 + i] = __fadd_rn(v[i], sums[cb * 32 + i]);
                    }
                    // the accumulator is free again (the loads have completed)
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(&ctl.segempty[b], 0);
                }
                if (stop) break;
#pragma unroll
                for (int cb = 0; cb < F_N / 64; ++cb) {
                    float p = 0.0f;
#pragma unroll
                    for (int i = 0; i < 32; ++i) p = fmaf(sums[cb * 32 + i], sums[cb * 32 + i], p);
                    acc += (double)p;
                }
            }
            // ---- the end of a unit, reached by every epilogue warp also when it has given up
            const int ub = un & 1, tile = u / parts;
            if (h == 1) ctl.part[ub][m] = acc;
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (h == 0) {
                double s = acc + ctl.part[ub][m];
                if (*abort_flag) s = (double)NAN;
                bool write = true;
                if (parts > 1) {   // this part's sums into scratch; the last one adds them in order
                    double *slots = scratch.slot + ((size_t)tile * parts * 2 + half) * F_VEC + m;
                    slots[(size_t)(u - tile * parts) * 2 * F_VEC] = s;
                    __threadfence();
                    asm volatile("bar.sync 2, 128;" ::: "memory");
                    if (m == 0)
                        ctl.last[ub] = atomicAdd(scratch.count + 2 * (size_t)tile + half, 1u) ==
                                       (unsigned)(parts - 1);
                    asm volatile("bar.sync 2, 128;" ::: "memory");
                    write = ctl.last[ub] != 0;
                    if (write) {
                        __threadfence();
                        s = 0.0;
                        for (int p = 0; p < parts; ++p) s += __ldcg(slots + (size_t)p * 2 * F_VEC);
                    }
                }
                const int v = vec0(u) + m;
                if (write && v < C && MPQ_IN(v, C)) {
                    // exact: undo the operand scales
                    const int e = ctl.xexp + f16_scale_exp(__uint_as_float(ld_after_wait(vrange + v)));
                    err[v] = (float)(s / (double)N * pow2d(-2 * e));
                }
            }
        }
        // no copy lands after the CTA is gone: the last copy of every stage
        if (copier && lane == 0) {
            for (long long f = issued - NS > 0 ? issued - NS : 0; f < issued; ++f)
                drain_wait(&ctl.landed[f % NS], (uint32_t)(f / NS) & 1u, wc, KBIT);
        }
        __syncwarp();
    }

    cluster_sync();   // nothing of the pair's is in flight
    if (warp == F_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, F_TMEM_COLS);
    }
}

// The slow channels of the output error that this split is for (none for the clipping search), by the
// blocks from `first` on: a block looks at channels a grid of them apart, a lane each (every warp at
// all of them: where there are none that is over in a latency or two, before the split is), and its
// warps take the errors of the slow ones in turn.
__device__ __forceinline__ void split_slow_channels(const SlowLayer &l, int first)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int step = (int)gridDim.x - first;
    for (int k0 = (int)blockIdx.x - first; k0 < l.C; k0 += 32 * step) {
        const long long k = k0 + (long long)lane * step;
        unsigned slow = __ballot_sync(0xffffffffu, k < l.C && is_slow(l, (int)k));
        for (; slow; slow &= slow - 1)
            for (int n = warp; n <= l.K; n += S_WARPS)
                slow_error(l, k0 + (__ffs(slow) - 1) * step, n, lane);
    }
}

// X * 2^e split into fp16 hi and lo planes ([2][N][d]: hi at 0, lo at N d) by the first `blocks` blocks,
// 8 elements a thread per step, e from max|X| (xrange[0]) as the contraction's operand scale.
template <bool SLOW>
__global__ void __launch_bounds__(256, SLOW ? 4 : 1)
f16_split_kernel(const float4 *__restrict__ X, long long n8, const unsigned *__restrict__ xrange,
                 uint4 *__restrict__ hi, uint4 *__restrict__ lo, int blocks,
                 const __grid_constant__ SlowLayer slow)
{
    griddep_launch();
    griddep_wait();
    if (SLOW && (int)blockIdx.x >= blocks) {
        split_slow_channels(slow, blocks);
        return;
    }
    const float xs = pow2f(f16_scale_exp(__uint_as_float(ld_after_wait(xrange))));
    const long long stride = (long long)blocks * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n8; i += stride) {
        const float4 a = __ldg(X + 2 * i), b = __ldg(X + 2 * i + 1);
        uint4 H, L;
        split_f16x2(__fmul_rn(a.x, xs), __fmul_rn(a.y, xs), H.x, L.x);
        split_f16x2(__fmul_rn(a.z, xs), __fmul_rn(a.w, xs), H.y, L.y);
        split_f16x2(__fmul_rn(b.x, xs), __fmul_rn(b.y, xs), H.z, L.z);
        split_f16x2(__fmul_rn(b.z, xs), __fmul_rn(b.w, xs), H.w, L.w);
        hi[i] = H;
        lo[i] = L;
    }
}

// The same for rows of any length and alignment, into rows of dp elements (zeros from d on).
template <bool SLOW>
__global__ void __launch_bounds__(256, SLOW ? 4 : 1)
f16_split_rows_kernel(const float *__restrict__ X, int N, int d, int dp,
                      const unsigned *__restrict__ xrange, uint4 *__restrict__ hi,
                      uint4 *__restrict__ lo, int blocks,
                      const __grid_constant__ SlowLayer slow)
{
    griddep_launch();
    griddep_wait();
    if (SLOW && (int)blockIdx.x >= blocks) {
        split_slow_channels(slow, blocks);
        return;
    }
    const float xs = pow2f(f16_scale_exp(__uint_as_float(ld_after_wait(xrange))));
    const int d8 = dp / 8;
    const long long n8 = (long long)N * d8, stride = (long long)blocks * blockDim.x;
    const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long dt = stride / d8;               // rows and items that a stride advances
    const int dj = (int)(stride - dt * d8);
    long long t = i0 / d8;
    int j = (int)(i0 - t * d8);
    for (long long i = i0; i < n8; i += stride) {
        const float *x = X + t * d + 8 * j;
        const int left = d - 8 * j;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = e < left ? __fmul_rn(__ldg(x + e), xs) : 0.0f;
        uint4 H, L;
        split_f16x2(v[0], v[1], H.x, L.x);
        split_f16x2(v[2], v[3], H.y, L.y);
        split_f16x2(v[4], v[5], H.z, L.z);
        split_f16x2(v[6], v[7], H.w, L.w);
        hi[i] = H;
        lo[i] = L;
        t += dt;
        j += dj;
        if (j >= d8) {
            j -= d8;
            ++t;
        }
    }
}

// Clipping search (Eq. 12): the residual r = w - s q of channel c0 + v / n_cand under candidate
// v mod n_cand (s = K / Qmax, the codes q of Eq. 8 with the sign of w, q = 0 where s is 0 or NaN),
// scaled by 2^e and split into fp16 hi/lo planes ([2][M][d] as hi and lo).  A CTA takes vectors a
// grid apart, 8 elements a thread per step: one vector each would make CTAs that live for a few loads,
// and each of them pays for the dependent launch's instructions (65,536 vectors of 64 elements, 32
// candidates, N = 128, the whole call: 104 us, 73 without those instructions, 58 so; 20,000 of 2,048
// the same either way).  e comes from a bound on the vector's elements,
// max(min(max|w|, s/2), max|w| - Qmax s): an element with code 0 keeps r = w, one with a nearest
// nonzero code |r| <= s/2, a clamped one |r| = |w| - Qmax s (a residual a rounding above the bound
// still fits fp16, whose range reaches 2^16); kept in vrange[v] (float bits) for the contraction.
// (With max|w| below s/2, as for a small channel under a layer-wide K, every code is 0 and the
// bound is max|r| itself.)
__global__ void __launch_bounds__(128)
clip_planes_kernel(const float *__restrict__ W, int d, const float *__restrict__ clip,
                   const float *__restrict__ chmax, int c0, int n_cand, int qmax, int M,
                   uint4 *__restrict__ hi, uint4 *__restrict__ lo, unsigned *__restrict__ vrange)
{
    griddep_launch();
    griddep_wait();
    const int d8 = d / 8;
    const float qmaxf = (float)qmax, qlim = qmaxf + 1.0f;
    const float tband = 0.5f - MPQ_FAST_REL * (qlim + 1.0f);
    for (int v = blockIdx.x; v < M; v += gridDim.x) {
        const long long k = c0 + v / n_cand;
        // clip row of channel k, candidate v mod n_cand: index c0 n_cand + v
        const float sv = __fdiv_rn(__ldg(clip + (long long)c0 * n_cand + v), qmaxf);
        // (the fast codes' bound holds for normal reciprocals: other scales take the division)
        const bool normal = sv > 0x1p-120f && sv < 0x1p120f;
        const float inv = normal ? __frcp_rn(sv) : 0.0f;
        const float m = __ldg(chmax + k);
        const float bound = fmaxf(fminf(m, __fmul_rn(0.5f, sv)), __fmaf_rn(-qmaxf, sv, m));
        const float vf = pow2f(f16_scale_exp(bound));
        if (threadIdx.x == 0) vrange[v] = __float_as_uint(bound);
        const float4 *w4 = reinterpret_cast<const float4 *>(W + k * d);
        const long long row = (long long)v * d8;
        for (int j = threadIdx.x; j < d8; j += blockDim.x) {
            const float4 a = __ldg(w4 + 2 * j), b = __ldg(w4 + 2 * j + 1);
            const float w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
            float q[8];
            bool unsure = !normal;
#pragma unroll
            for (int e = 0; e < 8; ++e) q[e] = code_signed_fast(w[e], inv, qmaxf, qlim, tband, unsure);
            if (unsure) {
#pragma unroll
                for (int e = 0; e < 8; ++e) q[e] = code_signed_exact(w[e], sv, qmaxf);
            }
            uint32_t h[4], l[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                split_f16x2(__fmul_rn(__fmaf_rn(-sv, q[2 * e], w[2 * e]), vf),
                            __fmul_rn(__fmaf_rn(-sv, q[2 * e + 1], w[2 * e + 1]), vf), h[e], l[e]);
            hi[row + j] = make_uint4(h[0], h[1], h[2], h[3]);
            lo[row + j] = make_uint4(l[0], l[1], l[2], l[3]);
        }
    }
}

int clip_tiles(int vectors) { return (vectors + 2 * F_VEC - 1) / (2 * F_VEC); }

// Parts of a vector tile's row tiles, each one unit: those with the least modelled time on the busiest
// pair, in twentieths of a step of 64 elements -- a row tile costs its steps (a twentieth more where
// the planes of the vector tiles at work do not stay in L2 from one row tile to the next: 1746 x 1920,
// N = 2020, 32 candidates 820 us whole, 790 in 3 parts, as many row tiles a pair), the end of a unit
// two (its sums, which nothing of the pair overlaps), leaving them to another pair half a step more.
// Fewer parts on ties; at most about 16 units a pair (the scratch of their sums stays below about 5 MB),
// never more than row tiles.  Single row tiles throughout cost short rows dearly: 2048 x 64, N = 2048,
// 20 candidates 139 us in 8 parts, 89 whole; 1000 x 2048 338 us in 8 parts, 540 whole.  Fitted to 126
// layers of 64 to 2,048 channels, 64 to 2,048 elements and 500 to 2,048 rows (within 2 % on average).
int clip_parts(int tiles, int N, int d)
{
    const long long n_rt = (N + (long long)F_N - 1) / F_N, n_ks = (d + F_KS - 1) / F_KS;
    const long long pairs = std::max(1, sm_count() / 2);
    const long long per = std::min(n_rt, std::max(1LL, tiles * n_rt / (16 * pairs)));
    const long long most = (n_rt + per - 1) / per;
    long long best = -1;
    int parts = 1;
    for (long long p = 1; p <= most; ++p) {
        const long long units = (tiles * p + pairs - 1) / pairs;        // of the busiest pair
        const bool reread = std::min((long long)tiles, pairs / p) * 1024 * d > 100000000;
        const long long cost = (units * n_rt + p - 1) / p * n_ks * (reread ? 21 : 20) +
                               units * (p > 1 ? 50 : 40);
        if (best < 0 || cost < best) {
            best = cost;
            parts = (int)p;
        }
    }
    return parts;
}

size_t clip_slot_bytes(int tiles, int N, int d)
{
    const int parts = clip_parts(tiles, N, d);
    return parts > 1 ? (size_t)tiles * parts * 2 * F_VEC * sizeof(double) : 0;
}

// The contraction over the residual planes A of C vectors, X already split into xs; count, slot:
// ClipScratch of clip_tiles(C) tiles.
mpq_status launch_clip_error(const void *A, int N, int C, int d, float *err,
                             const unsigned *xrange, const unsigned *vrange, const uint16_t *xs,
                             unsigned *count, double *slot, cudaStream_t stream)
{
    const int tiles = clip_tiles(C), parts = clip_parts(tiles, N, d);

    CUtensorMap tmX, tmA;
    memset(&tmX, 0, sizeof(tmX));
    memset(&tmA, 0, sizeof(tmA));
    const cuuint64_t dx[3] = {(cuuint64_t)d, (cuuint64_t)N, 2};
    const cuuint64_t sx[2] = {(cuuint64_t)d * 2, (cuuint64_t)N * d * 2};
    const cuuint32_t bx[3] = {F_KS, F_ROWS, 2};
    const cuuint64_t da[3] = {(cuuint64_t)d, (cuuint64_t)C, 2};
    const cuuint64_t sa[2] = {(cuuint64_t)d * 2, (cuuint64_t)C * d * 2};
    const cuuint32_t ba[3] = {F_KS, F_VEC, 2};
    if (!encode_tile_map(&tmX, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, xs, dx, sx, bx,
                         CU_TENSOR_MAP_SWIZZLE_128B) ||
        !encode_tile_map(&tmA, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, A, da, sa, ba,
                         CU_TENSOR_MAP_SWIZZLE_128B)) {
        set_error("clipping search: tensor map encoding failed");
        return MPQ_ERR_CUDA;
    }
    if ((long long)F_SMEM > max_smem_optin()) {
        set_error("clipping search needs %d bytes of shared memory", F_SMEM);
        return MPQ_ERR_UNSUPPORTED;
    }
    static std::atomic<int> limit[kMaxDevices];
    cudaError_t e = allow_smem(reinterpret_cast<const void *>(clip_error_kernel), limit, F_SMEM);
    if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute");

    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(F_THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)F_SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = after_previous_kernel();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    // one resident pair per two SMs (queried once per process), no more than units
    static std::atomic<int> resident{0};
    int pairs = resident.load(std::memory_order_relaxed);
    if (pairs == 0) {
        cfg.gridDim = dim3((unsigned)(sm_count() / 2 * 2), 1, 1);
        e = cudaOccupancyMaxActiveClusters(&pairs, clip_error_kernel, &cfg);
        if (e != cudaSuccess) return cuda_status(e, "cudaOccupancyMaxActiveClusters");
        pairs = std::max(1, pairs);
        resident.store(pairs, std::memory_order_relaxed);
    }
    pairs = std::min(pairs, tiles * parts);
    cfg.gridDim = dim3((unsigned)(2 * pairs), 1, 1);
    const ClipScratch scratch = {count, slot};
    WaitCtl wc;
    mpq_status wst = wait_ctl(&wc);
    if (wst != MPQ_OK) return wst;
    e = cudaLaunchKernelEx(&cfg, clip_error_kernel, C, N, d, xrange, vrange, err, parts, scratch, wc,
                           tmX, tmA);
    return cuda_status(e, "clipping-search kernel launch");
}

}  // namespace

// X split into the fp16 planes xs ([2][N][dp]) and the slow channels' errors on `stream`.
cudaError_t launch_x_split(const float *X, int N, int d, const unsigned *xrange, uint16_t *xs,
                           const SlowLayer &slow, cudaStream_t stream)
{
    const int dp = (d + 15) / 16 * 16;
    const long long n8 = (long long)N * dp / 8;
    const int sb = (int)std::max(1LL, std::min<long long>((n8 + 255) / 256, 4LL * sm_count()));
    cudaLaunchAttribute attr[1] = {after_previous_kernel()};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(sb + std::min(slow.C, sm_count())), 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    uint4 *hi = reinterpret_cast<uint4 *>(xs), *lo = reinterpret_cast<uint4 *>(xs + (size_t)N * dp);
    if (d != dp || ((uintptr_t)X & 15) != 0)
        return cudaLaunchKernelEx(&cfg, slow.C ? f16_split_rows_kernel<true> : f16_split_rows_kernel<false>,
                                  X, N, d, dp, xrange, hi, lo, sb, slow);
    return cudaLaunchKernelEx(&cfg, slow.C ? f16_split_kernel<true> : f16_split_kernel<false>,
                              reinterpret_cast<const float4 *>(X), n8, xrange, hi, lo, sb, slow);
}

// Channels per chunk of residual planes: whole channels, at most 4 GiB of planes at a time.
static int clip_chunk_channels(int C, int d, int n_cand)
{
    return (int)std::min<long long>(C, std::max(1LL, (1LL << 32) / (4LL * d * n_cand)));
}

// The X range word, X's planes, the residual planes of one chunk, their bounds, the partial sums of
// one chunk, the arrival counters of every chunk.
struct ClipLayout {
    int cc, n_count;          // channels of a chunk, counters
    size_t xs, planes, vrange, slot, count, bytes;
};

static ClipLayout clip_layout(int C, int N, int d, int n_cand)
{
    ClipLayout l;
    l.cc = clip_chunk_channels(C, d, n_cand);
    const int chunks = (C + l.cc - 1) / l.cc;
    const int last = (C - (chunks - 1) * l.cc) * n_cand, m_max = l.cc * n_cand;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    l.xs = 256;
    l.planes = l.xs + (size_t)N * d * 4;
    l.vrange = l.planes + (size_t)m_max * d * 4;
    l.slot = up(l.vrange + (size_t)m_max * 4);
    l.count = l.slot + std::max(chunks > 1 ? clip_slot_bytes(clip_tiles(m_max), N, d) : 0,
                                clip_slot_bytes(clip_tiles(last), N, d));
    l.n_count = 2 * ((chunks - 1) * clip_tiles(m_max) + clip_tiles(last));
    l.bytes = up(l.count + (size_t)l.n_count * 4);
    return l;
}

size_t clip_f16_scratch_bytes(int C, int N, int d, int n_cand)
{
    return clip_layout(C, N, d, n_cand).bytes;
}

mpq_status launch_clip_f16(const float *X, int N, const float *W, const float *clip,
                           const float *chmax, int C, int d, int qmax, int n_cand, float *err,
                           void *scratch, cudaStream_t stream)
{
    const ClipLayout l = clip_layout(C, N, d, n_cand);
    const int cc = l.cc;
    char *p = static_cast<char *>(scratch);
    unsigned *xrange = reinterpret_cast<unsigned *>(p);
    uint16_t *xs = reinterpret_cast<uint16_t *>(p + l.xs);
    uint16_t *planes = reinterpret_cast<uint16_t *>(p + l.planes);
    unsigned *vrange = reinterpret_cast<unsigned *>(p + l.vrange);
    double *slot = reinterpret_cast<double *>(p + l.slot);
    unsigned *count = reinterpret_cast<unsigned *>(p + l.count);
    mpq_status st = launch_x_range(X, N, d, xrange, count, l.n_count, stream);
    if (st != MPQ_OK) return st;
    cudaError_t e = launch_x_split(X, N, d, xrange, xs, SlowLayer{}, stream);
    if (e != cudaSuccess) return cuda_status(e, "X split kernel launch");
    for (int c0 = 0; c0 < C && st == MPQ_OK; c0 += cc) {
        const int cn = std::min(cc, C - c0);
        const int M = cn * n_cand;
        const int threads = std::min(128, (d / 8 + 31) / 32 * 32);
        uint4 *hi = reinterpret_cast<uint4 *>(planes);
        cudaLaunchAttribute attr[1] = {after_previous_kernel()};
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)std::min(M, 32 * sm_count()), 1, 1);
        cfg.blockDim = dim3((unsigned)threads, 1, 1);
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, clip_planes_kernel, W, d, clip, chmax, c0, n_cand, qmax, M, hi,
                               hi + (size_t)M * (d / 8), vrange);
        st = cuda_status(e, "clip residual planes kernel launch");
        if (st == MPQ_OK)
            st = launch_clip_error(planes, N, M, d, err + (size_t)c0 * n_cand, xrange, vrange, xs,
                                   count, slot, stream);
        count += 2 * clip_tiles(M);
    }
    return st;
}

}  // namespace mpq
