// Algorithm 1 with the adaptive grid of Eq. 10 (Definition 1), for channels of any length.
//
// Step i of channel k: Delta = the minimal gap of r_i (Definition 1, pairs of distinct
// magnitudes), gamma = min(Delta / Qmax, eta) (eta when r_i has one distinct magnitude), and the
// grid search of a over I = [0, 2 Qmax ||r_i||] with step gamma: a_m = m gamma, m = 1..M,
// M = floor(2 Qmax ||r_i|| / gamma), each taken as the fp32 point scale s_m = fl(a_m / Qmax)
// (s q = a [r/a]_Q, Eq. 1).  Codes q = clamp(rint(fl(r / s)), -Qmax, Qmax) (Eq. 8), the objective
// ||r - s q||^2 (Eq. 9), its first minimiser over m, r <- fmaf(-s, q, r) (Eq. 7).
//
// The grid is not enumerated (Definition 1 makes it 1e8..1e10 points long on real channels).
// Every element's code magnitude is a non-increasing step function of the scale, so for each
// element a = |r_j| and level L the set of fp32 scales where the code is at least L is
// {s <= tau_{j,L}}, with tau the largest such fp32 value (found with the correctly rounded
// division itself).  Sorted, the thresholds cut the scale axis into pieces with constant codes,
// on which the objective is the quadratic R2 - 2 s P + s^2 N (P = sum a_j c_j exact in 64-bit
// fixed point, N = sum c_j^2 exact).  An fp32 screen bounds every piece's minimum from below; the
// pieces whose bound can reach the best exact value are settled in double at their grid points
// next to the quadratic's minimiser (grid indices found by bisection on the exact s_m).  Equal
// values go to the smaller scale, i.e. the first m.  The decision is the exact minimiser of the
// objective; the oracle's double sum of squares differs from it only by rounding, so the two can
// differ only at a near tie.
//
// Few pieces can hold the minimum, so few thresholds are sorted.  Rows with more thresholds than
// the sort list holds first count them in buckets of the scale's leading bits (128 or 256 per
// octave) in shared memory, P and N exact per bucket: the suffix sums give each bucket's codes at
// its upper edge (P_hi, N_hi), and since a threshold's element and level satisfy
// a / (2L - 1) = tau / 2, on the bucket [lo, hi)
//   D(s) >= min_s (s^2 N_hi - 2 s P_hi) - (N_lo - N_hi) hi (hi - lo).
// Only the thresholds of buckets whose bound can reach the best value found at a bucket's edge
// (moved to the nearest grid point) are sorted.  On c2's 64 x 576 layer that is a few hundred of
// 4,032.  Lists that overflow (equal magnitudes by the thousand, extreme tails) sort all
// thresholds in global scratch instead (adaptive_search_all).
//
// ||r||^2 (for M and the squared-norm output) is the double sum in index order, exactly as the
// definition, by a warp of its own (ad_ordered_sum) while the others sort the magnitudes
// (Definition 1's minimal gap) and count thresholds, none of which needs it.  One CTA per channel
// at a time (persistent over the layer).
//
// The kernel is bound by latency, of double operations above all (a dependent addition takes some
// 85 cycles here, a division about ten times that): the norm's additions run as integers, 32 at a
// time, grid points are found by a warp at once, and the point scales take a division only where a
// product with 1/Qmax leaves their fp32 rounding open.  64 x 576, 4 bits, 4 points: 462 us with all
// thresholds sorted in global memory and a norm of dependent double additions, 150 now (of a step's
// 67 thousand cycles: magnitudes 9, counting 5, bucket sums 5, the norm's last 7, screen and list
// 16, settling 24).
#include <float.h>
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "mpq_internal.cuh"

MPQ_CHECKED_UNIT("adaptive.cu");

namespace mpq {
namespace {

constexpr int AW = 16;                 // worker warps per CTA
constexpr int AT = AW * 32;
constexpr int A_THREADS = AT + 32;     // and the warp that sums ||r||^2
constexpr int A_CTAS_PER_SM = 2;
constexpr int A_MAX_EVENTS = 1 << 16;  // d * Qmax (the thresholds of one step)

// ---- the definition's scalar arithmetic -------------------------------------------------------
__device__ __forceinline__ int ad_code_mag(float a, float s, int qmax)
{
    if (s == 0.0f) return 0;
    return (int)fminf(rintf(__fdiv_rn(a, s)), (float)qmax);
}

// the grid's point scale s_m = fl32(fl64(m gamma) / Qmax), each operation rounded once.  inv =
// fl64(1 / Qmax): the product with it is within 2^-51 of the quotient, so it rounds to the same
// fp32 value unless it lies within 16 double steps of the middle of two (or fp32's exponent range
// ends), where the division decides.
__device__ __forceinline__ float ad_scale(long long m, double gamma, int qmax, double inv)
{
    const double y = __dmul_rn((double)m, gamma);
    const double v = __dmul_rn(y, inv);
    const unsigned low = (unsigned)__double_as_longlong(v) & 0x1FFFFFFFu;   // below fp32's mantissa
    if (low - (0x10000000u - 16u) > 32u && v > 1e-36 && v < 1e38) return __double2float_rn(v);
    return __double2float_rn(__ddiv_rn(y, (double)qmax));
}

// code magnitude >= L (1 <= L <= Qmax) at scale s: rint(fl(a/s)) >= L
__device__ __forceinline__ bool ad_held(float a, float s, int L)
{
    return s > 0.0f && rintf(__fdiv_rn(a, s)) >= (float)L;
}

// tau_{a,L}: the largest fp32 scale with code >= L, 0 if no positive scale has it.  fl(a/s) is
// non-increasing in s, so the set is a prefix of the positive floats; the start a / (L - 1/2) is
// within a few ulps of its end.  Each loop is bounded (64 steps; the start is never that far off).
__device__ __forceinline__ float ad_threshold(float a, int L)
{
    float s = __fdiv_rn(a, (float)L - 0.5f);
    if (!(s < FLT_MAX)) s = FLT_MAX;
    if (ad_held(a, s, L)) {
        for (int it = 0; it < 64 && s < FLT_MAX; ++it) {
            const float u = nextafterf(s, FLT_MAX);
            if (!ad_held(a, u, L)) break;
            s = u;
        }
        return s;
    }
    for (int it = 0; it < 64; ++it) {
        s = nextafterf(s, 0.0f);
        if (s == 0.0f || ad_held(a, s, L)) return s;
    }
    return s;
}

// Smallest m in [lo, M] with s_m >= f (an fp32 value); M + 1 if none.  s_m = fl32(y_m) is
// non-decreasing in m and reaches f once y_m passes the midpoint between f's predecessor and f,
// which y_m = m gamma / Qmax (1 + O(2^-52)) crosses within a couple of indices of
// midpoint * Qmax / gamma: the answer is bracketed there by two exact s_m and bisected (about
// five exact scales in all); a failed bracket falls back to bisecting [lo, M].
__device__ long long ad_first_m_ge(float f, long long lo, long long M, double gamma, int qmax,
                                  double inv)
{
    auto ok = [&](long long m) { return ad_scale(m, gamma, qmax, inv) >= f; };
    if (lo > M) return M + 1;
    if (ok(lo)) return lo;
    if (!ok(M)) return M + 1;
    long long a = lo, b = M;   // ok(a) false, ok(b) true
    const double h = 0.5 * ((double)nextafterf(f, 0.0f) + (double)f);   // exact
    const double est = __dmul_rn(h, __ddiv_rn((double)qmax, gamma));
    if (est > (double)lo && est < (double)M) {
        const long long c = (long long)est;
        const long long a2 = c - 2 > lo ? c - 2 : lo;
        const long long b2 = c + 3 < M ? c + 3 : M;
        if (!ok(a2) && ok(b2)) {
            a = a2;
            b = b2;
        }
    }
    for (int it = 0; it < 80 && b - a > 1; ++it) {
        const long long mid = a + (b - a) / 2;
        if (ok(mid)) b = mid; else a = mid;
    }
    return b;
}

// the smallest fp32 value >= x, and the one after the fp32 value x
__device__ __forceinline__ float ad_ceil_f(double x)
{
    float f = __double2float_rn(x);
    if ((double)f < x) f = nextafterf(f, INFINITY);
    return f;
}
__device__ __forceinline__ float ad_next_f(float x) { return nextafterf(x, INFINITY); }

// ---- building blocks of the AT worker threads ------------------------------------------------
// the workers' barrier, and the two hand-offs with the norm warp (named barriers)
__device__ __forceinline__ void ad_sync() { asm volatile("bar.sync 1, %0;" ::"n"(AT) : "memory"); }
__device__ __forceinline__ void ad_bar_arrive(int id)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(A_THREADS) : "memory");
}
__device__ __forceinline__ void ad_bar_sync(int id)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(A_THREADS) : "memory");
}

// The strides j, j/2, .., 1 (j <= 32) of a bitonic merge of size k over 64 values held by a warp, two
// per lane (i0 = the first's index, the second's 32 above).
template <typename T>
__device__ __forceinline__ void ad_merge64(T &a0, T &a1, int i0, int k, int j)
{
    auto order = [](T &x, T &y, bool up) {
        if ((x > y) == up) {
            const T z = x;
            x = y;
            y = z;
        }
    };
    if (j == 32) {
        order(a0, a1, (i0 & k) == 0);
        j = 16;
    }
    const int lane = threadIdx.x & 31;
    const bool up0 = (i0 & k) == 0, up1 = ((i0 + 32) & k) == 0;
    for (; j > 0; j >>= 1) {
        const T b0 = __shfl_xor_sync(0xffffffffu, a0, j), b1 = __shfl_xor_sync(0xffffffffu, a1, j);
        const bool low = (lane & j) == 0;
        a0 = ((a0 > b0) == (low == up0)) ? b0 : a0;
        a1 = ((a1 > b1) == (low == up1)) ? b1 : a1;
    }
}

// Sorts n values ascending in shared memory (n a power of two, at least 64; padded by the caller):
// a bitonic network, its strides up to 32 in a warp's registers.
template <typename T>
__device__ __forceinline__ void ad_bitonic(T *a, int n)
{
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    ad_sync();
    for (int c = w; c < n / 64; c += AW) {
        const int i0 = c * 64 + lane;
        T a0 = a[i0], a1 = a[i0 + 32];
        for (int k = 2; k <= 64; k <<= 1) ad_merge64(a0, a1, i0, k, k >> 1);
        a[i0] = a0;
        a[i0 + 32] = a1;
    }
    ad_sync();
    for (int k = 128; k <= n; k <<= 1) {
        for (int j = k >> 1; j >= 64; j >>= 1) {
            for (int p = t; p < n / 2; p += AT) {
                const int i = ((p & ~(j - 1)) << 1) | (p & (j - 1));
                const T x = a[i], y = a[i + j];
                if ((x > y) == ((i & k) == 0)) {
                    a[i] = y;
                    a[i + j] = x;
                }
            }
            ad_sync();
        }
        for (int c = w; c < n / 64; c += AW) {
            const int i0 = c * 64 + lane;
            T a0 = a[i0], a1 = a[i0 + 32];
            ad_merge64(a0, a1, i0, k, 32);
            a[i0] = a0;
            a[i0 + 32] = a1;
        }
        ad_sync();
    }
}

struct ASort {
    unsigned hist[AW][256];   // per-warp digit counts, then scatter offsets
    unsigned wsum[AW];
    unsigned keys_or, keys_and;
};

// exclusive prefix over the 256 digit totals (threads 0..255 each hold one), through wsum
__device__ __forceinline__ unsigned ad_scan256(unsigned v, ASort &st)
{
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (t < 256 && lane == 31) st.wsum[w] = x;
    ad_sync();
    unsigned base = 0;
    if (t < 256)
        for (int i = 0; i < w; ++i) base += st.wsum[i];
    ad_sync();
    return base + x - v;
}

// Sorts n (key, val) pairs ascending by key: stable LSD radix sort, 8-bit digits, ping-pong between
// a and b; digits on which every key agrees are skipped.  Each warp owns a contiguous segment and
// ranks equal digits inside a 32-element tile with __match_any_sync, so the order is stable.
// Returns the buffer that holds the result.
__device__ uint2 *ad_sort(uint2 *a, uint2 *b, int n, ASort &st)
{
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (t == 0) {
        st.keys_or = 0u;
        st.keys_and = 0xffffffffu;
    }
    ad_sync();
    unsigned o = 0u, an = 0xffffffffu;
    for (int i = t; i < n; i += AT) {
        const unsigned k = a[i].x;
        o |= k;
        an &= k;
    }
    atomicOr(&st.keys_or, o);
    atomicAnd(&st.keys_and, an);
    ad_sync();
    const unsigned diff = st.keys_or ^ st.keys_and;
    const int seg = ((n + AW - 1) / AW + 31) / 32 * 32;
    const int w0 = min(n, w * seg), w1 = min(n, w * seg + seg);
    const unsigned lt = (1u << lane) - 1u;
    for (int shift = 0; shift < 32; shift += 8) {
        if (((diff >> shift) & 255u) == 0u) continue;   // uniform across the CTA
        for (int i = t; i < AW * 256; i += AT) (&st.hist[0][0])[i] = 0u;
        ad_sync();
        for (int t0 = w0; t0 < w1; t0 += 32) {
            const int i = t0 + lane;
            const unsigned dg = i < w1 ? (a[i].x >> shift) & 255u : 256u;
            const unsigned m = __match_any_sync(0xffffffffu, dg);
            if (dg < 256u && (m & lt) == 0u) st.hist[w][dg] += __popc(m);
            __syncwarp();
        }
        ad_sync();
        unsigned tot = 0;
        if (t < 256)
            for (int ww = 0; ww < AW; ++ww) tot += st.hist[ww][t];
        const unsigned base = ad_scan256(tot, st);
        if (t < 256) {
            unsigned run = base;
            for (int ww = 0; ww < AW; ++ww) {
                const unsigned c = st.hist[ww][t];
                st.hist[ww][t] = run;
                run += c;
            }
        }
        ad_sync();
        for (int t0 = w0; t0 < w1; t0 += 32) {
            const int i = t0 + lane;
            uint2 e = make_uint2(0u, 0u);
            if (i < w1) e = a[i];
            const unsigned dg = i < w1 ? (e.x >> shift) & 255u : 256u;
            const unsigned m = __match_any_sync(0xffffffffu, dg);
            if (dg < 256u && MPQ_IN(st.hist[w][dg] + __popc(m & lt), n))
                b[st.hist[w][dg] + __popc(m & lt)] = e;
            __syncwarp();
            if (dg < 256u && (m & lt) == 0u) st.hist[w][dg] += __popc(m);
            __syncwarp();
        }
        ad_sync();
        uint2 *x = a;
        a = b;
        b = x;
    }
    return a;
}

// Order-preserving image of a double (total order on non-NaN values).
__device__ __forceinline__ unsigned long long ad_ordered(double x)
{
    const unsigned long long v = (unsigned long long)__double_as_longlong(x);
    return (v >> 63) ? ~v : (v | 0x8000000000000000ull);
}

__device__ __forceinline__ unsigned ad_ordered_f(float x)
{
    const unsigned v = __float_as_uint(x);
    return (v >> 31) ? ~v : (v | 0x80000000u);
}


// |r| as a 64-bit fixed-point integer a * 2^S from its fp32 bits (exact whenever a * 2^S is an
// integer: for every element that can take a nonzero code; smaller ones truncate, and their code
// is 0 at every positive grid scale on which P is used).
__device__ __forceinline__ long long ad_fixed(float a, int S)
{
    const uint32_t bits = __float_as_uint(a);
    const int E = (int)(bits >> 23);
    const long long Mt = (long long)((bits & 0x7FFFFFu) | (E ? 0x800000u : 0u));
    const int sh = (E ? E : 1) - 150 + S;
    if (sh >= 0) return Mt << sh;
    return sh > -40 ? (Mt >> -sh) : 0;
}

// Decision value D(s) = s (s N - 2 P) = ||r - s q||^2 - ||r||^2, P = Pfix 2^-S, in double.
__device__ __forceinline__ double ad_decision(float s, long long Pfix, long long N, double down)
{
    const double sd = (double)s;
    return __dmul_rn(sd, __fma_rn(sd, (double)N, -2.0 * ((double)Pfix * down)));
}

constexpr int A_LIST = 512;   // candidate pieces settled by the whole CTA
constexpr int A_KEYS = 2048;  // thresholds sorted in shared memory (in the radix sort's counters)
constexpr int A_BUCKETS = 2048;
constexpr int A_ALL = 512;    // rows with fewer thresholds sort them all
constexpr int A_QMAX = (1 << (MPQ_MAX_BITS - 1)) - 1;
static_assert(sizeof(unsigned) * AW * 256 >= sizeof(unsigned long long) * A_KEYS, "sort list");

struct APiece {
    float lo, hi;
    long long P, N;
};

struct AShared {
    ASort sort;                 // its counters also hold the sort list
    APiece list[A_LIST];
    APiece best;                // the piece with the smallest lower bound
    int nlist;
    int finite;
    double r2;                  // ||r||^2, double, index order
    double gamma, ratio;        // gamma, fl64(Qmax / gamma)
    long long M, mpos;
    unsigned long long gap;     // Definition 1: bits of the smallest half-gap (non-negative double)
    unsigned long long lbkey;   // (ordered fp32 lower bound, piece) of the best piece
    unsigned long long ubkey;   // (ordered fp32 value, bucket) of the best bucket edge
    unsigned long long dkey;    // ordered D of the best settled grid point
    unsigned skey;              // its scale's bits, among equal D
    double U;                   // best exact D of the first settled piece
    int state;                  // 0 search, 1 scale 0 (null point or no positive grid scale), 2 dead
    int nev;                    // candidate thresholds of the step
    int nall;                   // adaptive_search_all's count: nev still decides the branch to it
    float spos, slast;
    float amax[AW];             // max |r| per warp
    float gsmall[AW];
    long long part[AW][2];
};

// The (P, N) prefix of this thread's block of sorted events, by a block exclusive scan.
__device__ __forceinline__ void ad_block_prefix(long long &p, long long &n, AShared &sh)
{
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    long long xp = p, xn = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long yp = __shfl_up_sync(0xffffffffu, xp, o);
        const long long yn = __shfl_up_sync(0xffffffffu, xn, o);
        if (lane >= o) {
            xp += yp;
            xn += yn;
        }
    }
    if (lane == 31) {
        sh.part[w][0] = xp;
        sh.part[w][1] = xn;
    }
    ad_sync();
    long long bp = 0, bn = 0;
    for (int i = 0; i < w; ++i) {
        bp += sh.part[i][0];
        bn += sh.part[i][1];
    }
    ad_sync();
    p = bp + xp - p;
    n = bn + xn - n;
}

// The smallest objective over the grid points of one piece (lo, hi] with constant (P, N): the
// grid points on either side of the quadratic's minimiser P / N, clipped to the piece.  Returns
// false when no grid point falls inside.
__device__ bool ad_settle_piece(float lo, float hi, long long Pfix, long long N, double down,
                                double gamma, int qmax, double inv, long long mpos, long long M,
                                double &D, float &s)
{
    const long long m1 = ad_first_m_ge(ad_next_f(lo), mpos, M, gamma, qmax, inv);
    if (m1 > M) return false;
    const long long m2 = ad_first_m_ge(ad_next_f(hi), m1, M, gamma, qmax, inv) - 1;
    if (m1 > m2) return false;
    if (N == 0) {   // every code 0: D = 0 on the whole piece, its smallest scale first
        D = 0.0;
        s = ad_scale(m1, gamma, qmax, inv);
        return true;
    }
    const double sbar = __ddiv_rn((double)Pfix * down, (double)N);
    long long mb = ad_first_m_ge(ad_ceil_f(sbar), m1, m2, gamma, qmax, inv);
    if (mb > m2) mb = m2;
    const long long ma = mb > m1 ? mb - 1 : m1;
    const float sa = ad_scale(ma, gamma, qmax, inv), sb = ad_scale(mb, gamma, qmax, inv);
    const double Da = ad_decision(sa, Pfix, N, down), Db = ad_decision(sb, Pfix, N, down);
    if (Db < Da) {
        D = Db;
        s = sb;
    } else {
        D = Da;
        s = sa;
    }
    return true;
}

// The same by a whole warp (arguments uniform, the result in every lane): the grid points next to
// the minimiser straddle the first fp32 value f at or above it (or the piece's nearer end), whose
// grid index is estimated to within two; 32 indices around the estimate are evaluated at once.
__device__ bool ad_settle_warp(float lo, float hi, long long Pfix, long long N, double down,
                               double gamma, int qmax, double inv, double ratio, long long mpos,
                               long long M, double &D, float &s)
{
    const int lane = threadIdx.x & 31;
    float f = ad_next_f(lo);
    if (N != 0) {
        const double sbar = __ddiv_rn((double)Pfix * down, (double)N);
        if (sbar > (double)hi) f = ad_next_f(hi);
        else if (sbar > (double)lo) f = ad_ceil_f(sbar);
    }
    // s_m reaches f where m gamma / Qmax passes the middle of f and its predecessor
    const double h = 0.5 * ((double)nextafterf(f, 0.0f) + (double)f);
    const double est = fmin(fmax(__dmul_rn(h, ratio), (double)mpos), (double)M);
    const long long m = (long long)est + lane - 15;
    const bool valid = m >= mpos && m <= M;
    float sm = valid ? ad_scale(m, gamma, qmax, inv) : 0.0f;
    unsigned ge = __ballot_sync(0xffffffffu, valid && sm >= f);
    unsigned lt = __ballot_sync(0xffffffffu, valid && sm < f);
    if ((ge == 0u && (long long)est + 16 < M) || (lt == 0u && (long long)est - 15 > mpos)) {
        // (never seen: the estimate was farther off) lanes 0 and 1 take the two neighbours
        const long long mb = ad_first_m_ge(f, mpos, M, gamma, qmax, inv);
        const long long mm = mb - 1 + lane;
        const bool ok = lane < 2 && mm >= mpos && mm <= M;
        sm = ok ? ad_scale(mm, gamma, qmax, inv) : 0.0f;
        lt = __ballot_sync(0xffffffffu, ok && lane == 0);
        ge = __ballot_sync(0xffffffffu, ok && lane == 1);
    }
    const float sb = __shfl_sync(0xffffffffu, sm, ge ? __ffs(ge) - 1 : 0);
    const float sa = __shfl_sync(0xffffffffu, sm, lt ? 31 - __clz(lt) : 0);
    const bool has_b = ge != 0u && sb > lo && sb <= hi, has_a = lt != 0u && sa > lo && sa <= hi;
    if (!has_a && !has_b) return false;
    if (N == 0) {   // every code 0: D = 0 on the whole piece, its smallest scale first (f's)
        D = 0.0;
        s = has_b ? sb : sa;
        return true;
    }
    const double Da = has_a ? ad_decision(sa, Pfix, N, down) : INFINITY;
    const double Db = has_b ? ad_decision(sb, Pfix, N, down) : INFINITY;
    D = Db < Da ? Db : Da;
    s = Db < Da ? sb : sa;
    return true;
}

// sum_j x_j^2 in double, in index order, one rounding per addition (the definition's ||r||^2: the
// squares of fp32 values are exact), by a warp.  While the sum's exponent stays the same, each
// addition adds a whole number of its last place: the square rounded to that place, or on a tie
// (the bits below are exactly half) to the even sum.  So 32 of them are one integer sum: the tied
// ones' parity comes from the odd additions since the tie before, after which the sum was even.
// Where the sum reaches the next exponent (or is still smaller than a square) that one addition is
// made in double and the rest start over.
__device__ __forceinline__ double ad_ordered_sum(const float *__restrict__ r, int d)
{
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    double sum = 0.0;
    float next = lane < d ? r[lane] : 0.0f;
    for (int j0 = 0; j0 < d; j0 += 32) {
        double x = (double)next;
        x = __dmul_rn(x, x);
        const int jn = j0 + 32 + lane;
        next = jn < d ? r[jn] : 0.0f;
        const long long xb = __double_as_longlong(x);
        const int xe = (int)(xb >> 52);
        const long long xm = xe ? (xb & 0xFFFFFFFFFFFFFll) | (1ll << 52) : 0;   // 0 only for x = 0
        unsigned left = __ballot_sync(0xffffffffu, xm != 0);
        while (left) {   // warp-uniform
            const long long sbits = __double_as_longlong(sum);
            const int se = (int)(sbits >> 52);
            const long long sm = (sbits & 0xFFFFFFFFFFFFFll) | (1ll << 52);
            const bool mine = (left >> lane) & 1u;
            const int k = se - xe;                 // bits of the square below the sum's last place
            const bool big = mine && k < 0;        // (sum = 0 too: its exponent field is 0)
            const int kk = min(max(k, 0), 62);
            const long long q = mine && !big ? xm >> kk : 0;
            const long long rem = xm & ((1ll << kk) - 1), half = kk ? 1ll << (kk - 1) : 0;
            const bool tie = mine && !big && kk > 0 && rem == half;
            long long c = q + (mine && !big && kk > 0 && rem > half ? 1 : 0);
            const unsigned ties = __ballot_sync(0xffffffffu, tie);
            if (ties) {
                const unsigned odd = __ballot_sync(0xffffffffu, !tie && (c & 1));
                if (tie) {
                    const unsigned before = ties & below;
                    const int last = 31 - __clz(before);   // -1: none
                    const unsigned since = before ? below & ~((2u << last) - 1u) : below;
                    const int par = __popc(odd & since) + (before ? 0 : (int)(sm & 1));
                    c = q + ((par + (int)(q & 1)) & 1);
                }
            }
            const unsigned bigs = __ballot_sync(0xffffffffu, big);
            int cross = bigs ? __ffs(bigs) - 1 : 32;   // the first addition to make in double
            if (lane >= cross) c = 0;
            // the sum of c (each below 2^53 + 1) as two 32-bit sums
            const long long add =
                ((long long)__reduce_add_sync(0xffffffffu, (unsigned)(c >> 27)) << 27) +
                (long long)__reduce_add_sync(0xffffffffu, (unsigned)c & 0x7FFFFFFu);
            long long total = sm + add;
            if (total >= (1ll << 53)) {
                long long pre = c;   // inclusive prefix
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const long long y = __shfl_up_sync(0xffffffffu, pre, o);
                    if (lane >= o) pre += y;
                }
                const unsigned over = __ballot_sync(0xffffffffu, sm + pre >= (1ll << 53));
                cross = __ffs(over) - 1;
                total = sm + __shfl_sync(0xffffffffu, pre - c, cross);
            }
            if (se) sum = __longlong_as_double(((long long)se << 52) | (total & 0xFFFFFFFFFFFFFll));
            if (cross == 32) break;
            sum = __dadd_rn(sum, __shfl_sync(0xffffffffu, x, cross));
            left &= cross == 31 ? 0u : ~((2u << cross) - 1u);
        }
    }
    return sum;
}

// fp32 lower bound of D' = D 2^-2e over the scales [lo, hi] of a piece (continuous, so it also
// bounds the piece's grid points), with a margin for the fp32 roundings (at most ~8 of 2^-24).
__device__ __forceinline__ float ad_piece_lb(float lo, float hi, float Pn, float N, int e)
{
    if (N == 0.0f) return 0.0f;
    const float l = ldexpf(lo, -e), h = ldexpf(hi, -e);
    const float sb = __fdiv_rn(Pn, N);
    constexpr float REL = 9.5367431640625e-07f;   // 2^-20
    if (sb >= l * (1.0f - REL) && sb <= h * (1.0f + REL)) return -(Pn * sb) * (1.0f + REL);
    const float dl = l * (l * N - 2.0f * Pn) - REL * l * (l * N + 2.0f * Pn);
    const float dh = h * (h * N - 2.0f * Pn) - REL * h * (h * N + 2.0f * Pn);
    return fminf(dl, dh);
}


// Everything a step's search needs, the same for every worker thread.
struct AStep {
    const float *r;        // the residual row, shared memory
    int d, qmax;
    int e, S;              // max |r| < 2^e; fixed point R = |r| 2^S
    double down;           // 2^-S
    float pscale;          // P 2^-S / 2^e for the fp32 screens
    double gamma, inv, ratio;   // gamma, fl64(1 / Qmax), fl64(Qmax / gamma)
    long long M, mpos;
    float spos, slast;     // the grid's first and last positive scales
};

// The exact minimiser among the pieces of the worker's own entries [x0, x1): piece(x, lo, hi, P, N)
// gives entry x's scales (lo, hi] and codes, false where it is empty.  Uf0: an upper bound of the
// minimum (D 2^-2e, fp32).  Returns the chosen scale.
template <typename Piece>
__device__ __forceinline__ float ad_search_pieces(const AStep &q, AShared &sh, int x0, int x1,
                                                  float Uf0, Piece piece)
{
    const int t = threadIdx.x;
    // screen: every piece's fp32 lower bound; the smallest one's piece is settled first
    unsigned long long mykey = ~0ull;
    for (int x = x0; x < x1; ++x) {
        float lo, hi;
        long long P, N;
        if (piece(x, lo, hi, P, N)) {
            const float lb = ad_piece_lb(lo, hi, (float)P * q.pscale, (float)N, q.e);
            const unsigned long long key =
                ((unsigned long long)ad_ordered_f(lb) << 32) | (unsigned)x;
            if (key < mykey) mykey = key;
        }
    }
    unsigned long long wkey = mykey;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wkey = min(wkey, __shfl_xor_sync(0xffffffffu, wkey, o));
    if ((t & 31) == 0) atomicMin(&sh.lbkey, wkey);
    ad_sync();
    if (mykey != ~0ull && mykey == sh.lbkey) {
        APiece pc;
        if (piece((int)(unsigned)mykey, pc.lo, pc.hi, pc.P, pc.N)) sh.best = pc;
    }
    ad_sync();
    if (t < 32 && sh.lbkey != ~0ull) {
        const APiece pc = sh.best;
        float sv;
        double D;
        if (ad_settle_warp(pc.lo, pc.hi, pc.P, pc.N, q.down, q.gamma, q.qmax, q.inv, q.ratio,
                           q.mpos, q.M, D, sv) &&
            t == 0)
            sh.U = fmin(sh.U, D);
    }
    ad_sync();
    // pieces whose lower bound can reach the best settled value: settle them all
    const double U = sh.U;
    float Uf = Uf0;
    if (U < INFINITY) {
        const float u = (float)ldexp(U, -2 * q.e);
        Uf = fminf(Uf, nextafterf(u, INFINITY) + fabsf(u) * 2.384185791015625e-07f);   // 2^-22
    }
    double bD = INFINITY;
    float bS = 0.0f;
    bool have = false;
    if (t == 0 && q.mpos > 1) {   // grid points of scale 0: every code 0, D = 0
        bD = 0.0;
        have = true;
    }
    auto take = [&](double D, float sv) {
        if (!have || D < bD || (D == bD && sv < bS)) {
            bD = D;
            bS = sv;
            have = true;
        }
    };
    for (int x = x0; x < x1; ++x) {
        float lo, hi;
        long long P, N;
        if (!piece(x, lo, hi, P, N)) continue;
        if (!(ad_piece_lb(lo, hi, (float)P * q.pscale, (float)N, q.e) <= Uf)) continue;
        // the piece's continuous minimum in double ends most of these (margin 2^-40 of its terms,
        // against the settled value's and this one's roundings of 2^-53 each)
        if (N != 0) {
            const double Pd = (double)P * q.down, Nd = (double)N;
            const double s0 = fmin(fmax(Pd / Nd, (double)lo), (double)hi);
            const double v = s0 * (s0 * Nd - 2.0 * Pd);
            if (v - s0 * (s0 * Nd + 2.0 * Pd) * 9.094947017729282e-13 > U) continue;
        }
        const int slot = atomicAdd(&sh.nlist, 1);
        if (slot < A_LIST) {
            sh.list[slot] = APiece{lo, hi, P, N};
        } else {   // beyond the list: settled by its own thread
            double D;
            float sv;
            if (ad_settle_piece(lo, hi, P, N, q.down, q.gamma, q.qmax, q.inv, q.mpos, q.M, D, sv))
                take(D, sv);
        }
    }
    ad_sync();
    for (int x = t >> 5; x < min(sh.nlist, A_LIST); x += AW) {   // a warp per queued piece
        const APiece pc = sh.list[x];
        double D;
        float sv;
        if (ad_settle_warp(pc.lo, pc.hi, pc.P, pc.N, q.down, q.gamma, q.qmax, q.inv, q.ratio,
                           q.mpos, q.M, D, sv))
            take(D, sv);
    }
    const unsigned long long dk = have ? ad_ordered(bD) : ~0ull;
    unsigned long long wdk = dk;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wdk = min(wdk, __shfl_xor_sync(0xffffffffu, wdk, o));
    if ((t & 31) == 0 && wdk != ~0ull) atomicMin(&sh.dkey, wdk);
    ad_sync();
    if (have && dk == sh.dkey) atomicMin(&sh.skey, __float_as_uint(bS));
    ad_sync();
    return sh.skey != ~0u ? __uint_as_float(sh.skey) : q.spos;
}

// Every threshold at or above the grid's first positive scale, sorted in global scratch (bufA,
// bufB: cap entries each): for rows whose candidate thresholds do not fit the sort list.  Workers
// enter one by one: a word that the branch to it reads (sh.nev) must not change here.
__device__ __noinline__ float adaptive_search_all(const AStep &q, AShared &sh, uint2 *bufA,
                                                  uint2 *bufB, int cap)
{
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const float *r = q.r;
    long long P0 = 0, N0 = 0;   // totals: P and N at spos (every kept threshold is held there)
    for (int j = t; j < q.d; j += AT) {
        const float a = fabsf(r[j]);
        if (a == 0.0f) continue;
        const long long R = ad_fixed(a, q.S);
        for (int L = 1; L <= q.qmax; ++L) {
            const float tau = ad_threshold(a, L);
            if (!(tau >= q.spos)) break;   // tau is non-increasing in L
            const int pos = atomicAdd(&sh.nall, 1);
            if (MPQ_IN(pos, cap))
                bufA[pos] = make_uint2(__float_as_uint(tau), ((unsigned)j << 8) | (unsigned)L);
            P0 += R;
            N0 += 2 * L - 1;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        P0 += __shfl_xor_sync(0xffffffffu, P0, o);
        N0 += __shfl_xor_sync(0xffffffffu, N0, o);
    }
    if (lane == 0) {
        sh.part[w][0] = P0;
        sh.part[w][1] = N0;
    }
    ad_sync();
    P0 = 0;
    N0 = 0;
    for (int x = 0; x < AW; ++x) {
        P0 += sh.part[x][0];
        N0 += sh.part[x][1];
    }
    ad_sync();
    int n = sh.nall;
    if (!MPQ_CHECK(n <= cap)) n = cap;
    const uint2 *ev = ad_sort(bufA, bufB, n, sh.sort);
    // pieces e = 0..n: scales (lo, hi] with the first e thresholds passed
    const int chunk = (n + 1 + AT - 1) / AT;
    const int e0 = min(n + 1, t * chunk), e1 = min(n + 1, e0 + chunk);
    long long cp = 0, cn = 0;
    auto passed = [&](int x) {
        const unsigned v = ev[x].y;
        if (!MPQ_IN(v >> 8, q.d)) return;
        cp += ad_fixed(fabsf(r[v >> 8]), q.S);
        cn += 2 * (int)(v & 255u) - 1;
    };
    for (int x = e0; x < min(e1, n); ++x) passed(x);
    ad_block_prefix(cp, cn, sh);   // the thresholds before e0
    const long long pre_p = cp, pre_n = cn;
    int at = e0;                   // cp, cn: the thresholds before entry `at`
    return ad_search_pieces(q, sh, e0, e1, INFINITY,
                            [&](int x, float &lo, float &hi, long long &P, long long &N) -> bool {
                                if (x < at) {
                                    at = e0;
                                    cp = pre_p;
                                    cn = pre_n;
                                }
                                for (; at < x; ++at) passed(at);
                                lo = x == 0 ? nextafterf(q.spos, 0.0f) : __uint_as_float(ev[x - 1].x);
                                hi = x == n ? q.slast : fminf(__uint_as_float(ev[x].x), q.slast);
                                P = P0 - cp;
                                N = N0 - cn;
                                return lo < hi;
                            });
}

// Dynamic shared memory: the residual row, then the magnitudes being sorted or the buckets.
__host__ __device__ __forceinline__ int ad_pow2(int n)
{
    int p = 64;
    while (p < n) p <<= 1;
    return p;
}

size_t adaptive_smem(int d)
{
    const size_t mag = (size_t)ad_pow2(d) * 4, hist = (size_t)A_BUCKETS * 12;
    return ((size_t)d * 4 + 15) / 16 * 16 + (mag > hist ? mag : hist);
}

__global__ void __launch_bounds__(A_THREADS, A_CTAS_PER_SM)
adaptive_kernel(const float *__restrict__ W, int C, int d, int qmax, int k_max, double eta,
                long long max_cand, int hbits, int8_t *__restrict__ codes,
                float *__restrict__ scales, float *__restrict__ resid_sq,
                long long *__restrict__ ncand, uint2 *__restrict__ scratch, int cap)
{
    extern __shared__ __align__(16) float r[];   // the residual row, d floats
    __shared__ AShared sh;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const bool worker = t < AT;
    uint2 *bufA = scratch + (size_t)blockIdx.x * 2 * cap;
    uint2 *bufB = bufA + cap;
    unsigned *mag = reinterpret_cast<unsigned *>(r + (d + 3) / 4 * 4);   // [ad_pow2(d)]
    unsigned *hLo = mag, *hHi = hLo + A_BUCKETS, *hN = hHi + A_BUCKETS;  // the same words, later
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(&sh.sort.hist[0][0]);
    const int dp = ad_pow2(d);
    const size_t plane = (size_t)C * d;
    const size_t n_codes = (size_t)k_max * plane, n_sc = (size_t)C * k_max;
    const size_t n_rs = (size_t)C * (k_max + 1);
    if (!MPQ_CHECK_SMEM_END(4 * (size_t)((d + 3) / 4 * 4) +
                            4 * (size_t)max(dp, 3 * A_BUCKETS)) ||
        !MPQ_CHECK(d <= cap))
        return;
    // buckets of 2^shift float steps: 8 octaves (256 per octave) below 2 max|r| reach scales of
    // max|r| / 128, 16 octaves (128 per octave) max|r| / 2^15; sets with larger codes take smaller
    // scales
    const int shift = 32 * qmax <= 256 ? 15 : 16;
    // short rows list every threshold (and one entry for the last piece) without counting
    const bool all_listed = (long long)d * qmax < A_ALL;
    const double inv = __ddiv_rn(1.0, (double)qmax);
    __shared__ float s_hinv[A_QMAX + 1];   // 1 / (L - 1/2)
    for (int L = t; L <= qmax; L += A_THREADS) s_hinv[L] = __frcp_rn((float)L - 0.5f);

    for (int k = blockIdx.x; k < C; k += gridDim.x) {
        if (t == 0) sh.finite = 1;
        __syncthreads();
        if (worker) {
            int fin = 1;
            float am = 0.0f;
            for (int j = t; j < d; j += AT) {
                const float v = MPQ_IN((size_t)k * d + j, plane) ? W[(size_t)k * d + j] : 0.0f;
                r[j] = v;
                mag[j] = __float_as_uint(fabsf(v));
                am = fmaxf(am, fabsf(v));
                fin &= isfinite(v);
            }
            for (int j = d + t; j < dp; j += AT) mag[j] = 0xFFFFFFFFu;
            if (!fin) atomicAnd(&sh.finite, 0);
            for (int o = 16; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
            if (lane == 0) sh.amax[w] = am;
        }
        for (int i = 0; i <= k_max; ++i) {
            __syncthreads();   // the residual row r_{i+1}, its magnitudes and their maximum
            const bool finite = sh.finite != 0;
            if (!worker) {
                // ---- the norm warp: ||r||^2 in index order, then the grid of Eq. 10
                const double r2 = ad_ordered_sum(r, d);
                if (lane == 0 && resid_sq && MPQ_IN((size_t)k * (k_max + 1) + i, n_rs))
                    resid_sq[(size_t)k * (k_max + 1) + i] = finite ? (float)r2 : NAN;
                if (i == k_max || !finite) break;
                ad_bar_sync(2);   // the minimal gap
                if (lane == 0) {
                    int state = 1;
                    long long M = 0;
                    if (r2 != 0.0) {   // (else a null point)
                        double g = __ddiv_rn(__longlong_as_double((long long)sh.gap), (double)qmax);
                        if (!(g < eta)) g = eta;
                        const double top = __dmul_rn(__dmul_rn(2.0, (double)qmax), __dsqrt_rn(r2));
                        const double mf = floor(__ddiv_rn(top, g));
                        sh.gamma = g;
                        sh.ratio = __ddiv_rn((double)qmax, g);
                        if (mf > (double)max_cand) {
                            state = 2;
                            M = -1;
                        } else {
                            M = (long long)mf;
                            if (M > 0) {
                                const long long mp = ad_first_m_ge(ad_next_f(0.0f), 1, M, g, qmax, inv);
                                sh.mpos = mp;
                                sh.U = mp > 1 ? 0.0 : INFINITY;
                                if (mp <= M) {
                                    state = 0;
                                    sh.spos = ad_scale(mp, g, qmax, inv);
                                    sh.slast = ad_scale(M, g, qmax, inv);
                                }
                            }
                        }
                    }
                    sh.M = M;
                    sh.state = state;
                }
                __syncwarp();
                ad_bar_sync(3);
                if (sh.state == 2) break;
                continue;
            }
            // ---- the workers
            if (i == k_max) break;
            if (finite) {
                if (t == 0) {
                    sh.gap = 0x7FF0000000000000ull;   // +inf
                    sh.lbkey = ~0ull;
                    sh.ubkey = ~0ull;
                    sh.dkey = ~0ull;
                    sh.skey = ~0u;
                    sh.nlist = 0;
                    sh.nev = 0;
                    sh.nall = 0;
                }
                float amax = 0.0f;
                for (int x = 0; x < AW; ++x) amax = fmaxf(amax, sh.amax[x]);
                // ---- Definition 1: the sorted magnitudes' smallest half-gap
                ad_bitonic(mag, dp);
                double gl = INFINITY;
                float gf = INFINITY;   // in fp32 first: double only where it can be the smallest
                for (int j = t + 1; j < d; j += AT) {
                    const unsigned a0 = mag[j - 1], a1 = mag[j];
                    if (a0 == a1) continue;
                    const float f = __fsub_rn(__uint_as_float(a1), __uint_as_float(a0));
                    if (f <= gf + gf * 2.384185791015625e-07f) {   // 2^-22
                        gl = fmin(gl, 0.5 * __dsub_rn((double)__uint_as_float(a1),
                                                      (double)__uint_as_float(a0)));
                        gf = fminf(gf, f);
                    }
                }
                unsigned long long gb = (unsigned long long)__double_as_longlong(gl);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) gb = min(gb, __shfl_xor_sync(0xffffffffu, gb, o));
                if (lane == 0) atomicMin(&sh.gap, gb);
                __syncwarp();
                ad_bar_arrive(2);
                ad_sync();   // the magnitudes are no longer read
                AStep q;
                q.r = r;
                q.d = d;
                q.qmax = qmax;
                frexpf(amax, &q.e);                 // max |r| < 2^e
                q.S = 62 - q.e - hbits;             // sum_j R_j c_j < 2^62
                q.down = __longlong_as_double((long long)(1023 - q.S) << 52);
                q.pscale = ldexpf(1.0f, hbits - 62);   // P 2^-S / 2^e
                // buckets: bucket b >= 1 (or any, if b0 = 0) holds the floats whose bits >> shift
                // are b0 + b, bucket 0 also everything below
                const unsigned top = min(__float_as_uint(amax) + 0x00800000u, 0x7F7FFFFFu) + 64u;
                const int b0 = max(0, (int)(top >> shift) + 1 - A_BUCKETS);
                auto bucket = [&](unsigned bits) -> int {
                    return all_listed ? 0 : max(0, min(A_BUCKETS - 1, (int)(bits >> shift) - b0));
                };
                const unsigned step_mask = (1u << shift) - 1u;
                // tau's bucket: from the reciprocal estimate unless that lies within 16 float
                // steps of a bucket's edge (it is within a few of tau)
                auto bucket_of = [&](float a, int L) -> int {
                    const unsigned est = __float_as_uint(__fmul_rn(a, s_hinv[L]));
                    const unsigned in = est & step_mask;
                    if (in - 16u < step_mask - 32u && est < 0x7F000000u) return bucket(est);
                    return bucket(__float_as_uint(ad_threshold(a, L)));
                };
                // f(j, L) for every (element, level), spread over the workers
                auto for_thresholds = [&](auto f) {
                    int L = 1, j = t;
                    for (int x = t; x < d * qmax; x += AT, j += AT) {
                        while (j >= d) {
                            j -= d;
                            ++L;
                        }
                        f(j, L);
                    }
                };
                if (!all_listed && amax > 0.0f) {
                    for (int x = t; x < 3 * A_BUCKETS; x += AT) hLo[x] = 0u;
                    ad_sync();
                    for_thresholds([&](int j, int L) {
                        const float a = fabsf(r[j]);
                        if (a == 0.0f) return;
                        const int b = bucket_of(a, L);
                        const unsigned long long R = (unsigned long long)ad_fixed(a, q.S);
                        const unsigned Rl = (unsigned)R;
                        const unsigned old = atomicAdd(&hLo[b], Rl);
                        atomicAdd(&hHi[b], (unsigned)(R >> 32) + (old + Rl < old ? 1u : 0u));
                        atomicAdd(&hN[b], (unsigned)(2 * L - 1));
                    });
                    ad_sync();
                    // suffix sums: bucket b <- P_hi, N_hi, the codes held above its upper edge;
                    // this worker's buckets, the last first
                    constexpr int PER = A_BUCKETS / AT;
                    const int bt = A_BUCKETS - 1 - t * PER;
                    long long cp = 0, cn = 0;
                    for (int x = 0; x < PER; ++x) {
                        cp += (long long)(((unsigned long long)hHi[bt - x] << 32) | hLo[bt - x]);
                        cn += hN[bt - x];
                    }
                    ad_block_prefix(cp, cn, sh);
                    unsigned long long ukey = ~0ull;
                    for (int x = 0; x < PER; ++x) {
                        const int b = bt - x;
                        const long long hp = (long long)(((unsigned long long)hHi[b] << 32) | hLo[b]);
                        const unsigned hn = hN[b];
                        hLo[b] = (unsigned)cp;
                        hHi[b] = (unsigned)((unsigned long long)cp >> 32);
                        hN[b] = (unsigned)cn;
                        cp += hp;
                        cn += hn;
                        // D at the bucket's lower edge, where its own codes are held too
                        if (b > 0) {
                            const float l = ldexpf(__uint_as_float((unsigned)(b0 + b) << shift), -q.e);
                            const float Pn = (float)cp * q.pscale;
                            const float D = l * (l * (float)cn - 2.0f * Pn);
                            ukey = min(ukey, ((unsigned long long)ad_ordered_f(D) << 32) | (unsigned)b);
                        }
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
                        ukey = min(ukey, __shfl_xor_sync(0xffffffffu, ukey, o));
                    if (lane == 0) atomicMin(&sh.ubkey, ukey);
                    // bucket 0 (scales below edge 1): no element gains more than a^2, nor more
                    // than 2 s Qmax a
                    const float e1 = __uint_as_float((unsigned)(b0 + 1) << shift);
                    float gs = 0.0f;
                    for (int j = t; j < d; j += AT) {
                        const float a = ldexpf(fabsf(r[j]), -q.e);
                        gs += fminf(a * a, 2.0f * ldexpf(e1, -q.e) * (float)qmax * a);
                    }
                    for (int o = 16; o > 0; o >>= 1) gs += __shfl_xor_sync(0xffffffffu, gs, o);
                    if (lane == 0) sh.gsmall[w] = gs;
                }
                ad_bar_sync(3);   // the grid (and the buckets' sums)
                if (sh.state == 0) {
                    q.gamma = sh.gamma;
                    q.inv = inv;
                    q.ratio = sh.ratio;
                    q.M = sh.M;
                    q.mpos = sh.mpos;
                    q.spos = sh.spos;
                    q.slast = sh.slast;
                    float sbest;
                    float Uf = INFINITY;
                    const float REL = 3.814697265625e-06f;   // 2^-18: the fp32 roundings below
                    if (!all_listed) {
                        // an upper bound: the best edge's codes at the grid point next to it (at
                        // most half a step and a rounding away; codes fixed there are no better
                        // than the nearest ones, up to the division's rounding)
                        const int be = (int)(unsigned)sh.ubkey;
                        const float s0 = __uint_as_float((unsigned)(b0 + be) << shift);
                        const float gstep = (float)(q.gamma / (double)qmax);
                        if (s0 >= q.spos && s0 >= 2.0f * gstep && s0 <= 0.5f * q.slast) {
                            const float l = ldexpf(s0, -q.e);
                            const float dl = ldexpf(gstep, -q.e) + l * 4.76837158203125e-07f;   // 2^-21
                            // the codes at the edge: the next lower bucket's P_hi, N_hi
                            const long long P = (long long)(((unsigned long long)hHi[be - 1] << 32) |
                                                            hLo[be - 1]);
                            const float Pn = (float)P * q.pscale, Nn = (float)hN[be - 1];
                            Uf = l * (l * Nn - 2.0f * Pn) + 2.0f * fabsf(l * Nn - Pn) * dl + Nn * dl * dl +
                                 REL * l * (l * Nn + 2.0f * Pn);
                        }
                        if (q.mpos > 1) Uf = fminf(Uf, 0.0f);
                        ad_sync();   // hN is marked below
                        // buckets that can reach it: their bit 31 of hN, and an entry at the end
                        // of each for its last piece
                        for (int b = t; b < A_BUCKETS; b += AT) {
                            const float lo = __uint_as_float((unsigned)(b0 + b) << shift);
                            const float hi = __uint_as_float((unsigned)(b0 + b + 1) << shift);
                            const long long P = (long long)(((unsigned long long)hHi[b] << 32) | hLo[b]);
                            const float Pn = (float)P * q.pscale, Nn = (float)(hN[b] & 0x7FFFFFFFu);
                            float lb;
                            if (b == 0) {
                                lb = 0.0f;
                                for (int x = 0; x < AW; ++x) lb -= sh.gsmall[x];
                                lb *= 1.0f + 1.9073486328125e-05f;   // 2^-16: d roundings at most
                                if (b0 == 0) lb = -INFINITY;
                            } else {
                                const long long below = hN[b - 1] & 0x7FFFFFFFu;
                                const float dN = (float)(below - (long long)(hN[b] & 0x7FFFFFFFu));
                                const float l = ldexpf(lo, -q.e), h = ldexpf(hi, -q.e);
                                lb = ad_piece_lb(lo, hi, Pn, Nn, q.e) -
                                     dN * h * (h * (1.0f + 9.5367431640625e-07f) - l) * (1.0f + REL) -
                                     REL * h * (h * Nn + 2.0f * Pn);
                            }
                            if (!(lb > Uf) && lo <= q.slast) {
                                atomicOr(&hN[b], 0x80000000u);
                                const int pos = atomicAdd(&sh.nev, 1);
                                // the bucket's last float (the top bucket's may pass fp32's range)
                                const unsigned last = min(((unsigned)(b0 + b + 1) << shift) - 1u, 0x7F7FFFFFu);
                                if (pos < A_KEYS) keys[pos] = ((unsigned long long)last << 32) | 0xFFFFFFFFull;
                            }
                        }
                        ad_sync();
                    } else if (t == 0) {
                        sh.nev = 1;
                        keys[0] = (0x7F7FFFFFull << 32) | 0xFFFFFFFFull;
                    }
                    if (all_listed) ad_sync();
                    for_thresholds([&](int j, int L) {
                        const float a = fabsf(r[j]);
                        if (a == 0.0f) return;
                        if (!all_listed && (int)hN[bucket_of(a, L)] >= 0) return;
                        const int pos = atomicAdd(&sh.nev, 1);
                        if (pos < A_KEYS)
                            keys[pos] = ((unsigned long long)__float_as_uint(ad_threshold(a, L)) << 32) |
                                        ((unsigned)j << 8) | (unsigned)L;
                    });
                    ad_sync();
                    const int n = sh.nev;
                    if (n > A_KEYS) {
                        sbest = adaptive_search_all(q, sh, bufA, bufB, cap);
                    } else {
                        const int np = ad_pow2(n);
                        for (int x = n + t; x < np; x += AT) keys[x] = ~0ull;
                        ad_bitonic(keys, np);
                        // entry x: the piece (the threshold before it in its bucket, tau_x]; its
                        // codes are the bucket's P_hi, N_hi and the bucket's thresholds from x on
                        const int chunk = (n + AT - 1) / AT;
                        const int x0 = min(n, t * chunk), x1 = min(n, x0 + chunk);
                        long long cp = 0, cn = 0;
                        auto entry = [&](int x, long long &R, int &c) {
                            const unsigned v = (unsigned)keys[x];
                            R = 0;
                            c = 0;
                            if (v != 0xFFFFFFFFu && MPQ_IN(v >> 8, d)) {
                                R = ad_fixed(fabsf(r[v >> 8]), q.S);
                                c = 2 * (int)(v & 255u) - 1;
                            }
                        };
                        for (int x = x0; x < x1; ++x) {
                            long long R;
                            int c;
                            entry(x, R, c);
                            cp += R;
                            cn += c;
                        }
                        ad_block_prefix(cp, cn, sh);   // the entries before x0
                        const long long pre_p = cp, pre_n = cn;
                        // each bucket's end: P_hi, N_hi plus the prefix there
                        for (int x = x0; x < x1; ++x) {
                            long long R;
                            int c;
                            entry(x, R, c);
                            if ((unsigned)keys[x] == 0xFFFFFFFFu) {
                                if (all_listed) {
                                    sh.part[0][0] = cp;
                                    sh.part[0][1] = cn;
                                } else {
                                    const int b = bucket((unsigned)(keys[x] >> 32));
                                    const long long P = (long long)(((unsigned long long)hHi[b] << 32) |
                                                                    hLo[b]) + cp;
                                    hLo[b] = (unsigned)P;
                                    hHi[b] = (unsigned)((unsigned long long)P >> 32);
                                    hN[b] = (hN[b] & 0x7FFFFFFFu) + (unsigned)cn;
                                }
                            }
                            cp += R;
                            cn += c;
                        }
                        ad_sync();
                        int at = x0;
                        cp = pre_p;
                        cn = pre_n;
                        sbest = ad_search_pieces(
                            q, sh, x0, x1, Uf,
                            [&](int x, float &lo, float &hi, long long &P, long long &N) -> bool {
                                if (x < at) {
                                    at = x0;
                                    cp = pre_p;
                                    cn = pre_n;
                                }
                                long long R;
                                int c;
                                for (; at < x; ++at) {
                                    entry(at, R, c);
                                    cp += R;
                                    cn += c;
                                }
                                const unsigned bits = (unsigned)(keys[x] >> 32);
                                const int b = bucket(bits);
                                const unsigned prev = x > 0 ? (unsigned)(keys[x - 1] >> 32) : 0u;
                                unsigned lob = x > 0 && bucket(prev) == b ? prev : 0u;
                                if (lob == 0u && !all_listed && b > 0)
                                    lob = ((unsigned)(b0 + b) << shift) - 1u;
                                lo = fmaxf(__uint_as_float(lob), nextafterf(q.spos, 0.0f));
                                hi = fminf(__uint_as_float(bits), q.slast);
                                if (all_listed) {
                                    P = sh.part[0][0] - cp;
                                    N = sh.part[0][1] - cn;
                                } else {
                                    P = (long long)(((unsigned long long)hHi[b] << 32) | hLo[b]) - cp;
                                    N = (long long)hN[b] - cn;
                                }
                                return lo < hi;
                            });
                    }
                    if (t == 0 && MPQ_IN((size_t)k * k_max + i, n_sc))
                        scales[(size_t)k * k_max + i] = sbest;
                    if (t == 0) sh.spos = sbest;
                } else if (t == 0 && sh.state == 1) {
                    // null point, no grid point, or only scale-0 grid points
                    if (MPQ_IN((size_t)k * k_max + i, n_sc)) scales[(size_t)k * k_max + i] = 0.0f;
                    sh.spos = 0.0f;
                }
                if (t == 0 && ncand && MPQ_IN((size_t)k * k_max + i, n_sc))
                    ncand[(size_t)k * k_max + i] = sh.M;
                ad_sync();   // buckets and list no longer read, the scale published
            }
            if (!finite || sh.state == 2) {
                // a non-finite channel, or a refused step: this and every later step NaN
                for (int ii = i; ii < k_max; ++ii) {
                    for (int j = t; j < d; j += AT) {
                        const size_t at = (size_t)ii * plane + (size_t)k * d + j;
                        if (MPQ_IN(at, n_codes)) codes[at] = 0;
                    }
                    if (t == 0 && MPQ_IN((size_t)k * k_max + ii, n_sc) &&
                        MPQ_IN((size_t)k * (k_max + 1) + ii + 1, n_rs)) {
                        scales[(size_t)k * k_max + ii] = NAN;
                        if (ncand && (ii > i || !finite)) ncand[(size_t)k * k_max + ii] = 0;
                        if (resid_sq) resid_sq[(size_t)k * (k_max + 1) + ii + 1] = NAN;
                    }
                }
                break;
            }
            // update (Eq. 7): codes at the chosen scale, r <- fmaf(-s, q, r)
            const float sbest = sh.spos;
            float am = 0.0f;
            for (int j = t; j < d; j += AT) {
                const float v = r[j];
                int qv = ad_code_mag(fabsf(v), sbest, qmax);
                qv = v < 0.0f ? -qv : qv;
                const size_t at = (size_t)i * plane + (size_t)k * d + j;
                if (MPQ_IN(at, n_codes)) codes[at] = (int8_t)qv;
                const float nv = __fmaf_rn(-sbest, (float)qv, v);
                r[j] = nv;
                mag[j] = __float_as_uint(fabsf(nv));
                am = fmaxf(am, fabsf(nv));
            }
            for (int j = d + t; j < dp; j += AT) mag[j] = 0xFFFFFFFFu;
            for (int o = 16; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
            if (lane == 0) sh.amax[w] = am;
        }
        __syncthreads();   // everyone is done with this channel
    }
}

int ad_ceil_log2(long long x)
{
    int b = 0;
    while ((1LL << b) < x) ++b;
    return b;
}

}  // namespace

mpq_status launch_adaptive(const float *W, int C, int d, int qmax, int k_max, double eta,
                           long long max_cand, int8_t *codes, float *scales, float *resid_sq,
                           long long *ncand, cudaStream_t stream)
{
    const long long ev = (long long)d * qmax;
    if (ev > A_MAX_EVENTS) {
        set_error("adaptive grid: d * Qmax = %lld exceeds %d thresholds per step", ev, A_MAX_EVENTS);
        return MPQ_ERR_UNSUPPORTED;
    }
    const int cap = (int)(ev > d ? ev : d);
    const int grid = (int)std::min<long long>(C, (long long)sm_count() * A_CTAS_PER_SM);
    const size_t smem = adaptive_smem(d);
    static std::atomic<int> limit[kMaxDevices];
    cudaError_t e = allow_smem(reinterpret_cast<const void *>(adaptive_kernel), limit, smem);
    if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute (adaptive grid)");
    uint2 *scratch = nullptr;
    const mpq_status st = pool_scratch(reinterpret_cast<void **>(&scratch),
                                       (size_t)grid * 2 * cap * sizeof(uint2), stream);
    if (st != MPQ_OK) return st;
    adaptive_kernel<<<grid, A_THREADS, smem, stream>>>(W, C, d, qmax, k_max, eta, max_cand,
                                                ad_ceil_log2(ev) + 1, codes, scales, resid_sq,
                                                ncand, scratch, cap);
    e = cudaGetLastError();
    const cudaError_t ef = cudaFreeAsync(scratch, stream);
    if (e == cudaSuccess) e = ef;
    return cuda_status(e, "adaptive-grid kernel launch");
}

}  // namespace mpq
