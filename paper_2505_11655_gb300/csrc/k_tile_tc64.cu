// Float64-accurate likelihood on the tensor cores (arXiv:2505.11655 Sec. II A,
// Eq. (def:lnL:Decomposed), time-marginalised).
//
// The float64 pipe of this part does about two operations a clock and SM, so the plain
// float64 kernel (k_lnl.cu) is bound by it: 6 operations a mode, bin and detector.  Here
// the mode sum, the interpolation and the log-sum-exp over the time bins run in fixed point
// instead, exactly or to float64's resolution of the largest |c| times the largest |Q|, and the
// float64 pipe is left with the per-sample geometry (overlaps that are too uneven for one scale
// take the plain kernel: uneven64 below):
//   * the coefficients c_k,lm of a sample (one power-of-two scale over its detectors and
//     modes) and Q (one scale) are rounded to 55-bit integers, each cut into kDig = 7
//     balanced base-256 digits d_0..d_6 (|d| <= 128, exact in float16);
//   * R[s, c] = Re sum_lm conj(c_lm) Q_lm on the Q grid is contracted digit by digit with
//     tcgen05 kind::f16 MMAs into one float32 accumulator per order o = i + j <= 6 of digit
//     products: an order holds at most 7 x 42 products below 2^14, so every partial sum is
//     an integer below 2^22 (order 6: 2^23) and exact.  Digit i of the coefficients meets
//     digits 0..6-i of Q in one MMA (N = 32 (7 - i) columns: the digits of 32 Q columns side by
//     side), so the accumulators of all orders are filled by 7 MMAs per 16 components.  The
//     orders beyond 6 are left out: below 2^-53 of max|c| max|Q|, as is the rounding of the
//     55-bit integers;
//   * the seven accumulators are drained from tensor memory and joined to one 64-bit integer
//     X = sum_o a_o 2^(40 - 8 o) (float additions of 1.5 2^23 turn them into integers);
//   * interpolation between neighbouring columns by a 64-bit high multiplication with the
//     node fraction (48 bits), sums over detectors in 64-bit integers;
//   * the log-sum-exp takes differences to the running maximum as integers and 2^-t from a
//     128-entry table and a short polynomial in 64-bit fixed point; sums with 2^-52
//     resolution.  A chunk's bins are summed by four threads relative to their common maximum, and
//     the chunks' sums merged in order.
// The template term is contracted the same way, W_k = Z_k T_k (the real quadratic form of
// k_tile_tc.cu), with one order more (it is the whole of a faint sample's value, and what the orders
// beyond 6 leave out does not average away in a quadratic form), and summed against the components
// in 128-bit integers.
//
// Tiles are 128 samples in the order of the sky sort.  A tile's window on the Q grid is as
// wide as its samples' delays need (no sub-groups: a chunk of 64 time bins walks the
// detector's window in blocks of 64 columns and every sample takes the bins whose nodes lie
// in the block).  The coefficients' digits (86 KB a detector at 21 modes) are written once per
// tile to a scratch in global memory (L2) and loaded into shared memory by bulk copies
// whenever the detector changes.  When a batch has few tiles its time bins are split over
// several blocks (units), and a second kernel merges the chunks' sums.  Every step of a
// sample's value is exact or done in a fixed order on the sample's own numbers, so it does
// not depend on the batch, the tile or the split.
//
// Measured (3 detectors, 21 modes, 16384 Hz, 1001 bins, 20011 prior samples): 20.3 ms for the
// plain float64 kernel (70% of the float64 issue rate), 1.25 to 1.29 ms here; 100,000 samples 98.5
// -> 4.0 ms; 64 samples of 2 detectors, 2 modes, 401 bins 116 -> 99 us.  Against
// 80-bit arithmetic (8 problems at 3 SNRs, 1000 prior samples each, relative norms) its per-bin values
// are closer than the plain kernel's (0.45 to 0.83 of its error), ln L is as close (geometric mean of
// the ratios 0.94; the template term alone 3.7e-16 to 5.9e-16 in both: the geometry's roundings).
// With orders to 6 and float64 sums the template term had up to 6.6e-16.  What bounds it now is
// instruction issue (43% of the slots: the joins of the accumulators, the gathers' 64-bit
// arithmetic) and the quarters' barriers; the tensor pipe is 26% busy, the float64 pipe 13%.
//
// All waits are bounded (1 s by the global timer), as in k_tile_tc.cu.
#include <algorithm>
#include <array>
#include <climits>
#include <cmath>
#include <cuda_fp16.h>
#include <type_traits>

#include "ile_kernels.h"
#include "tc_ptx.cuh"
#include "tile_plan.cuh"

namespace rift {

namespace {

constexpr int kDig = 7;             // base-256 digits of a 55-bit integer
constexpr int kS = 128;             // samples per tile (MMA M)
constexpr int kSub = 32;            // Q columns per MMA batch
constexpr int kBlk = 64;            // Q columns per gathered block (two batches)
constexpr int kConsumers = 512;
constexpr int kThreads = kConsumers + 64;
constexpr int kIssuer = kConsumers / 32, kStager = kIssuer + 1;
constexpr int kQ = kConsumers / kS;      // threads per sample
constexpr int kBpt = 16;                 // time bins per thread and chunk
constexpr int kChunk = kQ * kBpt;
constexpr int kOrders = kDig + 1;        // (the last of the template term only)
constexpr int kAccCols = kOrders * kSub; // tensor-memory columns of one set of accumulators
constexpr int kTable = kTc64Table;       // entries 2^-(i/128) of the exponential
constexpr int kFrac = 48;                // fraction bits of a Q position
constexpr int kPows = kMaxPow + 1;
constexpr uint64_t kWait = 1000000000ull;
constexpr int kRecords = 4096;           // (tile, chunk) pairs of a batch whose time bins are split
constexpr int kSumBits = 52;             // resolution of the log-sum-exp (at most 4000 terms <= 1)
constexpr size_t kMinSmem = 120 * 1024;  // one block per SM
constexpr int64_t kPlanFrom = 128;       // tiles from which a batch's units are planned,
constexpr double kPlanSpan = 12.0 * kSub;   // where the delays span this many columns
constexpr int kUnitsPerTile = 16;
constexpr float kUnitsPerBlock = 2.2f;
static_assert(kS == kPlanSamples, "tiles of the planning code");
static_assert(2 * kAccCols <= 512, "two sets of accumulators in tensor memory");
static_assert(kS * kMaxDet <= kConsumers, "one (sample, detector) item per consumer thread");

struct Layout64 {
    size_t a, b, r, pos, u0, sc, gid, bad, tbl, m2, lo, bar, tptr, end;
    size_t nv, e5, ps, pw, pe, F, Y, pend;   // prologue tables, aliased on a, b, r
    int kp;
};

__host__ __device__ inline size_t al64(size_t o, size_t a = 128) { return (o + a - 1) / a * a; }

__host__ __device__ inline Layout64 layout64(int K, int M, int n_t)
{
    Layout64 L;
    L.kp = (2 * M + 15) / 16 * 16;
    size_t o = 0;
    L.a = o;   o = al64(o + (size_t)kDig * kS * L.kp * 2);
    L.b = o;   o = al64(o + (size_t)2 * kDig * kSub * L.kp * 2);
    L.r = o;   o = al64(o + (size_t)(kBlk + 1) * kS * 8);
    size_t p = 0;   // sample-minor tables of the prologue
    L.nv = p;  p += (size_t)3 * kS * 8;
    L.e5 = p;  p += (size_t)5 * kS * 8;
    L.ps = p;  p += (size_t)3 * kS * 8;
    L.pw = p;  p += (size_t)2 * kPows * kS * 8;
    L.pe = p;  p += (size_t)(kMaxL + 1) * kS * 16;
    L.F = p;   p += (size_t)K * kS * 16;
    L.Y = p;   p += (size_t)M * kS * 16;
    L.pend = p;
    o = p > o ? al64(p) : o;
    L.pos = o;  o = al64(o + (size_t)n_t * 8, 16);
    L.u0 = o;   o = al64(o + (size_t)K * kS * 8, 16);
    L.sc = o;   o = al64(o + (size_t)kS * 4, 16);
    L.gid = o;  o = al64(o + (size_t)kS * 4, 16);
    L.bad = o;  o = al64(o + (size_t)kS * 4, 16);
    L.tbl = o;  o = al64(o + (size_t)kTable * 8, 16);
    L.m2 = o;   o = al64(o + (size_t)2 * kS * 8, 16);
    L.lo = o;   o = al64(o + (size_t)2 * kMaxDet * 8, 16);
    L.bar = o;  o = al64(o + (size_t)8 * 8, 16);
    L.tptr = o; o = al64(o + 16, 16);
    L.end = o;
    return L;
}

// bytes of one detector's coefficient digits, and of a block's scratch
__host__ __device__ inline size_t a_bytes(int kp) { return (size_t)kDig * kS * kp * 2; }

// Units (tile x part of the time bins) of a batch: parts chosen so that the units fill the
// blocks evenly, where the split's records fit.  A unit costs its prologue (about a fifth of
// a whole tile's work) plus its share of the bins.
__host__ __device__ inline int parts64(int64_t tiles, int grid, int n_chunks)
{
    int best = 1;
    float cost = 1e30f;
    for (int p = 1; p <= 16 && p <= n_chunks; ++p) {
        if (p > 1 && tiles * n_chunks > (int64_t)kRecords)
            break;
        const float c = (float)((tiles * p + grid - 1) / grid) * (0.2f + 1.0f / p);
        if (c < cost) {
            cost = c;
            best = p;
        }
    }
    return best;
}

// Samples per tile and parts of a batch whose units are not planned.  While every tile of a quarter of
// the lanes and every chunk of bins has a block of its own, the tiles are that small: a block's
// prologue is bound by the float64 pipe and takes a quarter of the time (us a call: 512 samples of 1
// detector, 1 mode, 101 bins 101 -> 90, 64 of 3, 21, 1001 276 -> 262; the plain kernel takes 77 and
// 757).
struct Cut64 {
    int samples, parts;
    int64_t tiles;
};

__host__ __device__ inline Cut64 cut64(int64_t n, int grid, int n_chunks)
{
    const int64_t small = (n + 31) / 32, tiles = (n + kS - 1) / kS;
    const int most = n_chunks < 16 ? n_chunks : 16;
    if (small * most <= grid)
        return {32, most, small};
    return {kS, parts64(tiles, grid, n_chunks), tiles};
}

// ---------------------------------------------------------------- digits

// Position of the leading bit: |x| < 2^e for every x with |x| <= m (0 for m = 0).
__device__ __forceinline__ int exp_above(double m)
{
    int e = 0;
    if (m > 0.0)
        frexp(m, &e);
    return e;
}

// x 2^e by a multiplication (float64 is slow on this part, and ldexp is several operations)
__device__ __forceinline__ double mul_pow2(double x, int e)
{
    if (e > 1000 || e < -1000)
        return ldexp(x, e);
    return x * __hiloint2double((1023 + e) << 20, 0);
}

// The seven digits of a 55-bit integer as float16 bit patterns: the integer plus a bias of
// 128 in each of its six low bytes has the biased digits as bytes (the top one in bits
// 48..56), and float16 1024 + b is the pattern 0x6400 | b.
__device__ __forceinline__ uint64_t digit_bytes(long long I) { return (uint64_t)I + 0x0080808080808080ull; }

__device__ __forceinline__ uint32_t digit_pair(uint64_t x, uint64_t y, int part)
{
    // bytes of x and y biased by 128 -> two float16 digits
    const int sh = 8 * (kDig - 1 - part);
    const uint32_t mask = part == 0 ? 0x1ffu : 0xffu;
    const uint32_t a = (uint32_t)(x >> sh) & mask, b = (uint32_t)(y >> sh) & mask;
    const uint32_t v = 0x64006400u | a | (b << 16);
    __half2 h;
    memcpy(&h, &v, 4);
    h = __hsub2(h, __floats2half2_rn(1152.f, 1152.f));
    uint32_t r;
    memcpy(&r, &h, 4);
    return r;
}

// Q columns that some sample's bins reach, per detector (the Q window may be wider; what lies in
// the rest of it is no scale of anything).
struct Reach {
    int lo[kMaxDet], hi[kMaxDet];
    double inv[kMaxDet];   // 1 / columns
};

Reach reach_of(const Problem &P)
{
    Reach r{};
    for (int k = 0; k < P.K; ++k) {
        double d2 = 0.0;
        for (int i = 0; i < 3; ++i)
            d2 += P.xfs[k][i] * P.xfs[k][i];
        const double d = std::sqrt(d2), last = P.ufs0[k] + (P.n_t - 1) * P.t_step * P.fs;
        r.lo[k] = (int)std::max(0.0, std::floor(P.ufs0[k] - d) - 1.0);
        r.hi[k] = (int)std::min((double)(P.n_q - 1), std::floor(last + d) + 2.0);
        r.inv[k] = 1.0 / (r.hi[k] - r.lo[k] + 1);
    }
    return r;
}

// One block per (detector, mode): the largest component and the mean square modulus over the
// reachable columns; the largest of all to out[0].
__global__ void __launch_bounds__(256) scale64_kernel(const double2 *__restrict__ Q, int M, int n_q, Reach reach,
                                                      unsigned long long *__restrict__ out, double2 *__restrict__ sizes)
{
    __shared__ unsigned long long ms[8];
    __shared__ double ss[8];
    const int k = blockIdx.x / M, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double2 *row = Q + (size_t)blockIdx.x * n_q;
    unsigned long long m = 0ull;   // non-negative doubles order as integers
    double s = 0.0;
    for (int c = reach.lo[k] + threadIdx.x; c <= reach.hi[k]; c += blockDim.x) {
        const double2 q = row[c];
        m = max(m, (unsigned long long)__double_as_longlong(fabs(q.x)));
        m = max(m, (unsigned long long)__double_as_longlong(fabs(q.y)));
        s = fma(q.x, q.x, fma(q.y, q.y, s));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    if (lane == 0) {
        ms[warp] = m;
        ss[warp] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
            m = max(m, ms[w]);
            s += ss[w];
        }
        sizes[blockIdx.x] = make_double2(__longlong_as_double((long long)m), s * reach.inv[k]);
        if (m)
            atomicMax(out, m);
    }
}

// Whether one scale serves: the largest component is at most kUneven times the rms of every
// detector's strongest mode, and of the strongest mode with m = 2 and with m = -2 (alone in a
// face-on or face-off sample).  An error in fixed point is 8e-17 of the largest |c| times the
// largest |Q|, whichever detectors and modes a sample's value is made of; the plain kernel's bins
// carry the rounding of their positions, 2.4e-14 of the local term at 16384 Hz, 300 times as much.
// (Of the synthetic problems at SNRs of 8 to 150 the most uneven has 33.)  Zero rows say nothing.
constexpr double kUneven = 256.0;

// by a warp (non-negative doubles as integers: comparisons of doubles take the slow float64 pipe)
__device__ bool uneven64(const Problem &P, const double2 *sizes)
{
    using Bits = unsigned long long;
    const int lane = threadIdx.x & 31;
    Bits top = 0, det[kMaxDet] = {}, pol[2] = {};
    for (int e = lane; e < P.K * P.M; e += 32) {
        const int k = e / P.M, s = P.mode_m[e - k * P.M];
        const Bits largest = (Bits)__double_as_longlong(sizes[e].x), square = (Bits)__double_as_longlong(sizes[e].y);
        top = max(top, largest);
#pragma unroll
        for (int i = 0; i < kMaxDet; ++i)
            det[i] = k == i ? max(det[i], square) : det[i];
        pol[0] = s == 2 ? max(pol[0], square) : pol[0];
        pol[1] = s == -2 ? max(pol[1], square) : pol[1];
    }
    auto most = [](Bits v) {
#pragma unroll
        for (int o = 16; o; o >>= 1)
            v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
        return v;
    };
    Bits least = ~0ull;
    auto take = [&](Bits v) {
        v = most(v);
        least = v ? min(least, v) : least;
    };
#pragma unroll
    for (int i = 0; i < kMaxDet; ++i)
        take(det[i]);
    take(pol[0]);
    take(pol[1]);
    const double t = __longlong_as_double((long long)most(top));
    return least != ~0ull && !(t * t <= kUneven * kUneven * __longlong_as_double((long long)least));
}

// Q digits: [K][kDig][groups][kp/8][8 columns][8 components]
__global__ void digits_q_kernel(const double2 *__restrict__ Q, int K, int M, int n_q, int groups, int kp, Reach reach,
                                const unsigned long long *__restrict__ qmax, __half *__restrict__ out)
{
    const int sq = 55 - exp_above(__longlong_as_double((long long)*qmax));
    const int64_t per_part = (int64_t)groups * kp * 8, total = (int64_t)K * per_part / 2;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t f = 2 * e;   // an even component and the odd one behind it: one mode
        const int k = (int)(f / per_part);
        const int64_t w = f - (int64_t)k * per_part;
        const int g = (int)(w / (kp * 8)), rem = (int)(w - (int64_t)g * kp * 8);
        const int kc = rem / 64, row = (rem / 8) % 8, m = (8 * kc + rem % 8) / 2, c = 8 * g + row;
        uint64_t x = digit_bytes(0), y = x;
        if (c >= reach.lo[k] && c <= reach.hi[k] && m < M) {
            const double2 q = Q[((int64_t)k * M + m) * n_q + c];
            x = digit_bytes(__double2ll_rn(ldexp(q.x, sq)));
            y = digit_bytes(__double2ll_rn(ldexp(q.y, sq)));
        }
        for (int p = 0; p < kDig; ++p)
            reinterpret_cast<uint32_t *>(out + ((int64_t)k * kDig + p) * per_part)[w / 2] = digit_pair(x, y, p);
    }
}

// Entry (r, c) of the real template matrix: z^T T z = c^H U c + Re(c^T V c) (see k_tile_tc.cu)
__device__ __forceinline__ double template_entry(const double2 *U, const double2 *V, int M, int r, int c)
{
    const double2 u = U[(size_t)(r >> 1) * M + (c >> 1)], v = V[(size_t)(r >> 1) * M + (c >> 1)];
    if (!(r & 1))
        return (c & 1) ? -u.y - v.y : u.x + v.x;
    return (c & 1) ? u.x - v.x : u.y - v.y;
}

// Template digits: [K][kDig][kBlk/8 groups][kp/8][8 columns of T][8 components]; exps[k]
// such that |T_k| < 2^exps[k].  One block per detector (the last one looks at the overlaps' sizes too).
__global__ void digits_t_kernel(Problem P, int kp, const double2 *__restrict__ sizes, __half *__restrict__ out,
                                int *__restrict__ exps, int *err)
{
    __shared__ unsigned long long mx;
    const int k = blockIdx.x, M = P.M, R2 = 2 * M;
    const double2 *U = P.U64 + (size_t)k * M * M, *V = P.V64 + (size_t)k * M * M;
    if (threadIdx.x == 0)
        mx = 0ull;
    if (k == P.K - 1 && threadIdx.x >= blockDim.x - 32 && uneven64(P, sizes) && (threadIdx.x & 31) == 0)
        atomicOr(err, kNoteUneven);
    __syncthreads();
    for (int e = threadIdx.x; e < R2 * R2; e += blockDim.x)
        atomicMax(&mx, (unsigned long long)__double_as_longlong(fabs(template_entry(U, V, M, e / R2, e % R2))));
    __syncthreads();
    const int et = exp_above(__longlong_as_double((long long)mx));
    if (threadIdx.x == 0)
        exps[k] = et;
    const int per_part = kBlk * kp;
    for (int f = 2 * threadIdx.x; f < per_part; f += 2 * blockDim.x) {
        const int g = f / (kp * 8), rem = f - g * kp * 8;
        const int kc = rem / 64, row = (rem / 8) % 8, c = 8 * kc + rem % 8, n = 8 * g + row;
        uint64_t x = digit_bytes(0), y = x;
        if (n < R2 && c < R2) {
            x = digit_bytes(__double2ll_rn(ldexp(template_entry(U, V, M, c, n), 55 - et)));
            y = digit_bytes(__double2ll_rn(ldexp(template_entry(U, V, M, c + 1, n), 55 - et)));
        }
        for (int p = 0; p < kDig; ++p)
            reinterpret_cast<uint32_t *>(out + ((size_t)k * kDig + p) * per_part)[f / 2] = digit_pair(x, y, p);
    }
}

// ---------------------------------------------------------------- fixed point

// 2^-t of t = T 2^-57 (0 <= t < 64) as E 2^-63 times 2^-n: table of 2^-(i/128), and with
// g = r ln 2 of the rest r < 2^-7 the nested series 1 - g (1 - g/2 (1 - g/3 (1 - g/4 + g^2/20 -
// g^3/120))) in 64-bit fixed point (the innermost factor needs 32 bits only).
__device__ __forceinline__ uint64_t exp2_neg(uint64_t T, const uint64_t *__restrict__ tbl, int &n)
{
    n = (int)(T >> 57);
    const uint64_t f = T & ((1ull << 57) - 1ull);
    const uint64_t G = __umul64hi((f & ((1ull << 50) - 1ull)) << 14, 0xB17217F7D1CF79ACull);   // g 2^71
    const uint32_t g32 = (uint32_t)(G >> 39), gh = (uint32_t)(G >> 32);
    const uint32_t gg = __umulhi(g32, g32);
    // (1 - g/4 + g^2/20 - g^3/120) / 3 in units 2^-32
    const uint32_t c3 = 0x55555555u - __umulhi(gh, 2796202u) + __umulhi(gg, 71582788u - __umulhi(g32, 11930465u));
    const uint64_t a3 = ~(((uint64_t)gh * c3) >> 7);        // 1 - g/3 (...), units 2^-64
    const uint64_t a2 = ~(__umul64hi(G, a3) >> 8);          // 1 - g/2 (...)
    const uint64_t p = ~(__umul64hi(G, a2) >> 7);           // 1 - g (...)
    return __umul64hi(tbl[f >> 50], p);
}

// Scaled differences of a sample: lin = X 2^L.
struct DiffScale {
    int sh;          // T = (D << sh) log2(e) 2^-1 with sh = L + 58 (D >> -sh when negative)
    uint64_t dmax;   // larger differences are e^-44 and below
    __device__ void set(int L)
    {
        sh = max(-63, min(63, L + 58));
        const int s = -L;
        dmax = s >= 58 ? ~0ull : s >= 0 ? 44ull << s : s > -6 ? 44ull >> -s : 0ull;
    }
    __device__ uint64_t exponent(uint64_t D) const
    {
        return __umul64hi(sh >= 0 ? D << sh : D >> -sh, 0xB8AA3B295C17F0BCull);
    }
};

__extension__ typedef __int128 wide128;

// Log-sum-exp over bins: sum of exp(lin - max) in units 2^-kSumBits, max as an integer.
struct Lse {
    long long m;
    uint64_t s;
};

// exp(-D 2^L) in units 2^-kSumBits
__device__ __forceinline__ uint64_t term64(const DiffScale &ds, uint64_t D, const uint64_t *tbl)
{
    if (D > ds.dmax)
        return 0ull;
    int n;
    const uint64_t e = exp2_neg(ds.exponent(D), tbl, n);
    return ((e >> (62 - kSumBits + min(n, kSumBits + 1))) + 1ull) >> 1;
}

__device__ __forceinline__ Lse merge64(const DiffScale &ds, Lse a, Lse b, const uint64_t *tbl)
{
    if (a.m < b.m) {
        const Lse t = a;
        a = b;
        b = t;
    }
    const uint64_t D = (uint64_t)a.m - (uint64_t)b.m;
    if (b.s != 0ull && D <= ds.dmax) {
        int n;
        const uint64_t e = exp2_neg(ds.exponent(D), tbl, n);
        a.s += ((__umul64hi(b.s, e) << 1) | ((b.s * e) >> 63)) >> n;
    }
    return a;
}

// A double and what it lacks.
struct Two {
    double hi, lo;
};

__device__ __forceinline__ Two two_sum(double a, double b)
{
    const double s = __dadd_rn(a, b), r = __dsub_rn(s, a);
    return {s, __dadd_rn(__dsub_rn(a, __dsub_rn(s, r)), __dsub_rn(b, r))};
}

// (v has fewer than 2^62)
__device__ __forceinline__ Two two_of(long long v)
{
    const double h = (double)v;
    return {h, (double)(v - (long long)h)};
}

// max 2^lexp - quad + ln(sum) - ln(n_t) with one rounding of its large terms
__device__ __forceinline__ double lse_value(Lse v, int lexp, double quad, float quad_lo, int n_t)
{
    const double sum = (double)v.s * (1.0 / (double)(1ull << kSumBits));
    const Two m = two_of(v.m), d = two_sum(mul_pow2(m.hi, lexp), -quad);
    const double rest = __dadd_rn(d.lo, __dsub_rn(mul_pow2(m.lo, lexp), (double)quad_lo));
    return __dadd_rn(d.hi, __dadd_rn(rest, __dsub_rn(log(sum), log((double)n_t))));
}

// What the combination needs of a sample beside its chunks' sums and its template term: the scale
// (|lexp| < 4400), the error flags and what the template term lacks.
__device__ __forceinline__ uint64_t pack_info(int lexp, int flags, float quad_lo)
{
    return (uint64_t)(uint16_t)(int16_t)lexp | ((uint64_t)(uint16_t)flags << 16) |
           ((uint64_t)__float_as_uint(quad_lo) << 32);
}

// one accumulator set joined to X (see the head of the file)
template <int kN> __device__ __forceinline__ long long join_orders(const uint32_t (&v)[kN][4], int i)
{
    constexpr float kMagic = 12582912.f;   // 1.5 2^23: float bits 0x4B400000 + integer
    constexpr uint64_t kB = 0x4B400000ull;
    constexpr uint64_t kBias = (kB << 40) + (kB << 32) + (kB << 24) + (kB << 16) + (kB << 8) + kB + kB;
    const uint32_t b0 = __float_as_uint(__uint_as_float(v[0][i]) + kMagic);
    const uint32_t b1 = __float_as_uint(__uint_as_float(v[1][i]) + kMagic);
    const uint32_t b2 = __float_as_uint(__uint_as_float(v[2][i]) + kMagic);
    const uint32_t b3 = __float_as_uint(__uint_as_float(v[3][i]) + kMagic);
    const uint32_t b4 = __float_as_uint(__uint_as_float(v[4][i]) + kMagic);
    const uint32_t b5 = __float_as_uint(__uint_as_float(v[5][i]) + kMagic);
    float last = __uint_as_float(v[6][i]);
    if (kN > kDig)
        last = fmaf(__uint_as_float(v[kN - 1][i]), 0x1p-8f, last);
    const uint32_t b6 = __float_as_uint(fmaf(last, 0x1p-8f, kMagic));
    uint64_t x = (uint64_t)b5 + b6 - kBias;
    x += (uint64_t)b4 * 256u;
    x += (uint64_t)b3 * 65536u;
    x += (uint64_t)b2 * 16777216u;
    x += (uint64_t)((b0 << 8) + b1) << 32;
    return (long long)x;
}

}  // namespace

bool lnl_tc64_fits(const Problem &P, int max_smem)
{
    // at most 42 components (order 5: 6 x 42 products of 2^14 stay below 2^22)
    return !P.dist_marg && 2 * P.M <= 42 && P.n_q < (1 << 14) && P.n_t <= 4000 &&
           layout64(P.K, P.M, P.n_t).end + 2048 <= (size_t)max_smem;
}

size_t tc64_q_halves(int K, int M, int groups)
{
    return (size_t)K * kDig * groups * ((2 * M + 15) / 16 * 16) * 8;
}

size_t tc64_t_halves(int K, int M) { return (size_t)K * kDig * kBlk * ((2 * M + 15) / 16 * 16); }

// records of the split: per (chunk, sample) the chunk's Lse, and per sample its template term
// and scale
static int64_t split_tiles(int64_t n_max, int n_t)
{
    const int64_t n_chunks = (n_t + kChunk - 1) / kChunk;
    return std::min<int64_t>((n_max + kS - 1) / kS, kRecords / n_chunks);
}

size_t tc64_record_bytes(int64_t n_max, int n_t)
{
    return (size_t)split_tiles(n_max, n_t) * kS * 16 * ((n_t + kChunk - 1) / kChunk + 1);
}

// (with records, a tile has at most as many units as chunks)
int64_t tc64_units_cap(int64_t n_max) { return (n_max + kS - 1) / kS + kRecords; }

size_t tc64_scratch_bytes(int K, int M, int64_t n_max, int sms)
{
    const int64_t tiles = (n_max + kS - 1) / kS, blocks = std::min<int64_t>(sms, 16 * tiles);
    return (size_t)blocks * K * a_bytes((2 * M + 15) / 16 * 16);
}

// 2^-(i/128) in units 2^-63 (constants: filled once)
static const long long *exp2_table()
{
    static const std::array<long long, kTable> table = [] {
        std::array<long long, kTable> t{};
        for (int i = 0; i < kTable; ++i)
            t[i] = (long long)(uint64_t)std::ldexp(std::exp2(-(long double)i / kTable), 63);
        return t;
    }();
    return table.data();
}

void tc64_positions(const rift_ile_config &cfg, long long *pos, long long *u0)
{
    // the step with 32 bits behind a position's last (long double is emulated on some hosts: three
    // operations a bin, with the table above, were 0.3 ms of every handle's creation)
    __extension__ typedef __int128 wide;
    constexpr int kGuard = 32;
    const long double range = (long double)cfg.t_hi_s - (long double)cfg.t_lo_s;
    const wide step = cfg.n_t > 1 ? (wide)std::ldexp(range * (long double)cfg.fs_hz / (cfg.n_t - 1), kFrac + kGuard) : 0;
    for (int j = 0; j < cfg.n_t; ++j)
        pos[j] = (long long)((j * step + ((wide)1 << (kGuard - 1))) >> kGuard);
    std::copy_n(exp2_table(), kTable, pos + cfg.n_t);
    for (int k = 0; k < cfg.n_det; ++k)
        u0[k] = std::llround(
            std::ldexp(((long double)cfg.t_lo_s - (long double)cfg.q_t0_s[k]) * (long double)cfg.fs_hz, kFrac));
}

size_t tc64_scale_words(int K, int M) { return 2 + 2 * (size_t)K * M; }

cudaError_t launch_prep_tc64(const Problem &P, unsigned long long *qmax, __half *q_dig, __half *t_dig, int *t_exp,
                             int *err, cudaStream_t st)
{
    const int kp = (2 * P.M + 15) / 16 * 16;
    cudaError_t e = cudaMemsetAsync(qmax, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess)
        return e;
    const Reach reach = reach_of(P);
    double2 *sizes = reinterpret_cast<double2 *>(qmax + 2);
    scale64_kernel<<<P.K * P.M, 256, 0, st>>>(P.Q64, P.M, P.n_q, reach, qmax, sizes);
    const int64_t tot = (int64_t)P.K * P.tc_groups * kp * 4;
    digits_q_kernel<<<(int)std::min<int64_t>((tot + 255) / 256, 2048), 256, 0, st>>>(
        P.Q64, P.K, P.M, P.n_q, P.tc_groups, kp, reach, qmax, q_dig);
    digits_t_kernel<<<P.K, 512, 0, st>>>(P, kp, sizes, t_dig, t_exp, err);
    return cudaGetLastError();
}

namespace {

// Samples of the launch: n, or the device's count, of which counts up to `skip` are left to the
// caller's other kernel.
__device__ __forceinline__ int64_t device_count(int64_t n, const uint32_t *n_dev, uint32_t skip)
{
    if (!n_dev)
        return n;
    const uint32_t c = *n_dev;
    return c <= skip ? 0 : min(n, (int64_t)c);
}

// Whether a batch's chunks have records (its time bins may then be split over blocks).
__host__ __device__ inline bool has_records(int64_t n_tiles, int n_chunks)
{
    return n_tiles * n_chunks <= (int64_t)kRecords;
}

// Units of a batch of kPlanFrom tiles or more: a tile's time is that of the columns its samples'
// delays span, three and more times the narrowest in thinly sampled parts of the sky, so a tile
// is cut into parts of its time bins by its width (about kUnitsPerBlock units a block; whole tiles
// where the batch has no records), and the costly units are taken first.  With every tile in two
// parts, in the sort's order, the SMs were idle for 28% of a 20,000-sample batch.  One warp per
// tile.
__global__ void __launch_bounds__(32 * kPlanWarps)
units64_kernel(PlanProblem P, const double *__restrict__ theta, const uint32_t *__restrict__ perm, int64_t n,
               const uint32_t *__restrict__ n_dev, uint32_t skip, int grid, unsigned long long *__restrict__ list,
               int64_t cap, int *__restrict__ counts)
{
    __shared__ int cols[kPlanWarps][kMaxDet][kPlanSamples];
    __shared__ PlanFiles<unsigned long long, kPlanWarps * kUnitsPerTile> files;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tile = (int64_t)blockIdx.x * kPlanWarps + warp;
    const int64_t n_use = device_count(n, n_dev, skip), n_tiles = (n_use + kS - 1) / kS;
    plan_reset(files);
    if (tile < n_tiles) {
        int lo, hi;
        plan_columns(P, theta, perm, tile, n_use, 0xffffffffll, cols[warp], lo, hi);
        // batches of a chunk's windows over those of a single sample
        const int n_chunks = (P.n_t + kChunk - 1) / kChunk;
        const int span = (int)(P.beta * (float)(kChunk - 1)) + 2;
        const int own = lane < P.K ? span / kSub + 1 : 0;
        const int all = lane < P.K ? (span + (lo <= hi ? hi - lo : 0)) / kSub + 1 : 0;
        const float r = (float)__reduce_add_sync(0xffffffffu, all) / (float)__reduce_add_sync(0xffffffffu, own);
        const bool split = has_records(n_tiles, n_chunks);
        const float k = split ? kUnitsPerBlock * (float)grid / (float)n_tiles : 1.f;
        const int parts = split ? max(1, min(min(n_chunks, kUnitsPerTile), (int)(r * k + 0.5f))) : 1;
        const float x = r * k / (float)parts;   // about 1 where the batch is split as it wants
        const int cls = split ? (x > 1.5f ? 0 : x > 1.1f ? 1 : x > 0.8f ? 2 : 3) : (x > 2.4f ? 0 : x > 1.7f ? 1 : x > 1.25f ? 2 : 3);
        if (lane < parts) {
            const int c0 = lane * n_chunks / parts, c1 = (lane + 1) * n_chunks / parts;
            plan_file(files, ((unsigned long long)tile << 16) | (unsigned)(c0 << 8) | (unsigned)c1, cls);
        }
    }
    plan_write(files, list, cap, counts);
}

// The value of sample i (index g) from its chunks' sums; `padded` samples a chunk.
__device__ __forceinline__ void merge_sample(const Lse *records, int64_t padded, int64_t i, int n_chunks, int n_t,
                                             const uint64_t *tbl, uint32_t g, double *__restrict__ lnL_tmarg,
                                             const double *__restrict__ lnpw, double *__restrict__ lnw, int *err)
{
    // (other blocks' writes: not through this SM's first-level cache)
    auto load = [&](int64_t at) {
        const longlong2 v = __ldcg(reinterpret_cast<const longlong2 *>(records + at));
        return Lse{v.x, (uint64_t)v.y};
    };
    const Lse info = load(n_chunks * padded + i);
    const int lexp = (int)(int16_t)info.s, flags = (int)(uint16_t)(info.s >> 16);
    double r = __longlong_as_double(0x7ff8000000000000LL);
    if (flags == 0) {
        DiffScale ds;
        ds.set(lexp);
        Lse run = load(i);
        for (int c = 1; c < n_chunks; ++c)
            run = merge64(ds, run, load(c * padded + i), tbl);
        r = lse_value(run, lexp, __longlong_as_double(info.m), __uint_as_float((uint32_t)(info.s >> 32)), n_t);
    }
    if (!isfinite(r))
        atomicOr(err, kErrNonFinite);
    lnL_tmarg[g] = r;
    if (lnw && lnpw)
        lnw[g] = r + lnpw[g];
}

__global__ void __launch_bounds__(kThreads, 1)
lnl_tc64_kernel(Problem P, Tc64 X, const double *__restrict__ theta, const uint32_t *__restrict__ perm, int64_t n,
                double *__restrict__ lnL_tmarg, double *__restrict__ lnL_t, const double *__restrict__ lnpw,
                double *__restrict__ lnw, int *err, int *unit_counter, const uint32_t *__restrict__ n_dev,
                uint32_t skip, int planned, int fused)
{
    extern __shared__ __align__(128) unsigned char sm[];
    const int K = P.K, M = P.M, NT = P.n_t;
    const Layout64 L = layout64(K, M, NT);
    const int kp = L.kp, kcs = kp / 8;
    __half *As = reinterpret_cast<__half *>(sm + L.a);              // [kDig][kS x kp]
    __half *Bs = reinterpret_cast<__half *>(sm + L.b);              // [2][kDig][kSub x kp]
    long long *Rs = reinterpret_cast<long long *>(sm + L.r);        // [1 + kBlk][kS]; row 0 the previous block's last
    long long *pos = reinterpret_cast<long long *>(sm + L.pos);     // [NT] bin offset in Q samples, kFrac fraction bits
    long long *U0 = reinterpret_cast<long long *>(sm + L.u0);       // [K][kS] Q position of the first bin
    int *scs = reinterpret_cast<int *>(sm + L.sc);                  // [kS] c = I 2^-sc
    uint32_t *gid = reinterpret_cast<uint32_t *>(sm + L.gid);
    int *bad = reinterpret_cast<int *>(sm + L.bad);                 // [kS] error flags of the sample
    uint64_t *tbl = reinterpret_cast<uint64_t *>(sm + L.tbl);       // 2^-(i/128) 2^63
    unsigned long long *mF2 = reinterpret_cast<unsigned long long *>(sm + L.m2), *mY2 = mF2 + kS;
    long long *ulo = reinterpret_cast<long long *>(sm + L.lo), *uhi = ulo + kMaxDet;
    uint64_t *full = reinterpret_cast<uint64_t *>(sm + L.bar);      // [0,1] Q digits staged
    uint64_t *done = full + 2;                                      // [0,1] MMAs of a batch complete
    uint64_t *empty = full + 4;                                     // [0,1] accumulators drained
    uint64_t *fullA = full + 6;                                     // coefficient digits staged
    uint32_t *tptr = reinterpret_cast<uint32_t *>(sm + L.tptr);
    double *nv = reinterpret_cast<double *>(sm + L.nv), *e5 = reinterpret_cast<double *>(sm + L.e5);
    double *ps = reinterpret_cast<double *>(sm + L.ps), *pw = reinterpret_cast<double *>(sm + L.pw);
    double2 *pe = reinterpret_cast<double2 *>(sm + L.pe), *Fs = reinterpret_cast<double2 *>(sm + L.F);
    double2 *Ys = reinterpret_cast<double2 *>(sm + L.Y);
    __shared__ int unit_s, tile_s, chunks_s, abort_s, last_s;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool producer = warp >= kIssuer;
    const int64_t n_use = device_count(n, n_dev, skip);
    const int n_chunks = (NT + kChunk - 1) / kChunk, jnom = (NT + n_chunks - 1) / n_chunks;
    const Cut64 cut = planned ? Cut64{kS, 1, (n_use + kS - 1) / kS} : cut64(n_use, (int)gridDim.x, n_chunks);
    const int64_t n_tiles = cut.tiles;
    const int parts = cut.parts;
    const bool split = planned ? has_records(n_tiles, n_chunks) : parts > 1;
    const int sq = 55 - exp_above(__longlong_as_double((long long)*X.qmax));
    const uint32_t sub_bytes = (uint32_t)(kSub * kp * 2);           // one digit of a batch's columns
    const size_t ab = a_bytes(kp);
    __half *scratch = reinterpret_cast<__half *>(X.scratch + (size_t)blockIdx.x * K * ab);
    Lse *records = reinterpret_cast<Lse *>(X.records);
    const uint32_t sbo = (uint32_t)kcs * 128u;
    auto desc = [&](const void *p, uint32_t off) {
        return ((uint64_t)(((sbo >> 4) & 0x3FFFu) | (1u << 14)) << 32) |
               (((tc::smem_u32(p) + off) & 0x3FFFFu) >> 4) | ((uint64_t)(128u >> 4) << 16);
    };

    for (int j = tid; j < NT; j += kThreads)
        pos[j] = X.pos[j];
    for (int i = tid; i < kTable; i += kThreads)
        tbl[i] = (uint64_t)X.pos[NT + i];
    if (warp == 0)
        tc::tmem_alloc(tptr, 512);
    if (tid == 0) {
        for (int i = 0; i < 4; ++i)
            tc::mbar_init(full + i, 1);
        for (int i = 4; i < 6; ++i)
            tc::mbar_init(full + i, kConsumers / 32);
        tc::mbar_init(fullA, 1);
        tc::fence_mbar_init();
        abort_s = 0;
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tptr;
    // every role walks the same sequence of batches: g counts them (buffer g & 1, its
    // (g >> 1)-th use), ga the loads of coefficient digits
    uint32_t g = 0, ga = 0;
    bool first = true;

    for (;;) {
        // the shared memory that the next unit's copies overwrite was last touched by generic
        // accesses of this thread
        tc::fence_proxy_async_smem();
        if (tid == 0) {
            // the first unit by the block's index, the others from the counter
            // (no others where a launch merges for itself)
            unit_s = abort_s ? INT_MAX
                     : first ? (int)blockIdx.x
                     : fused ? INT_MAX
                             : (int)gridDim.x + atomicAdd(unit_counter, 1);
            first = false;
            tile_s = -1;
            unsigned long long w;
            if (planned) {
                if (!abort_s && plan_item(X.units, X.units_cap, X.unit_counts, unit_s, w)) {
                    tile_s = (int)(w >> 16);
                    chunks_s = (int)(w & 0xffffu);
                }
            } else if ((int64_t)unit_s < n_tiles * parts) {
                tile_s = unit_s / parts;
                const int part = unit_s - tile_s * parts;
                chunks_s = (int)((int64_t)part * n_chunks / parts) << 8 | (int)((int64_t)(part + 1) * n_chunks / parts);
            }
        }
        if (tid < K) {
            ulo[tid] = LLONG_MAX;
            uhi[tid] = LLONG_MIN;
        }
        if (tid < kS) {
            mF2[tid] = 0ull;
            mY2[tid] = 0ull;
            bad[tid] = 0;
        }
        __syncthreads();
        const int64_t tile = tile_s;
        if (tile < 0)
            break;
        const int ch0 = chunks_s >> 8, ch1 = chunks_s & 255;
        const int s_of = tid & (kS - 1), grp = tid >> 7;

        // ---------------- prologue A: trigonometry in float64, a quarter of it per thread
        if (!producer) {
            const int64_t si = tile * cut.samples + s_of;
            const uint32_t gi = s_of >= cut.samples || si >= n_use ? 0xffffffffu : perm ? perm[si] : (uint32_t)si;
            const double *th = theta + 6 * (int64_t)gi;
            const bool valid = gi != 0xffffffffu;
            if (grp == 0)
                gid[s_of] = gi;
            if (!__any_sync(0xffffffffu, valid)) {
                // a lane quarter without samples: its rows of every table are left as they are
            } else if (grp == 0) {
                const Sky sk = sky_of(valid ? th[0] : 0.0, valid ? th[1] : 0.0, P.gmst);
                nv[s_of] = sk.cd * sk.ch;
                nv[kS + s_of] = sk.cd * sk.sh;
                nv[2 * kS + s_of] = sk.sd;
                e5[s_of] = sk.cd;
                e5[kS + s_of] = sk.sd;
                e5[2 * kS + s_of] = sk.ch;
                e5[3 * kS + s_of] = sk.sh;
            } else if (grp == 1) {
                double s2, c2;
                sincos(2.0 * (valid ? th[2] : 0.0), &s2, &c2);
                ps[s_of] = c2;
                ps[kS + s_of] = s2;
                ps[2 * kS + s_of] = valid ? P.d_ref / th[5] : 0.0;
            } else if (grp == 2) {
                double sh, ch;
                sincos(0.5 * (valid ? th[4] : 0.0), &sh, &ch);
                double pc = 1.0, pp = 1.0;
                for (int q = 0; q < kPows; ++q) {
                    pw[q * kS + s_of] = pc;
                    pw[(kPows + q) * kS + s_of] = pp;
                    pc *= ch;
                    pp *= sh;
                }
            } else {
                // exp(-i j phi): the first two from the functions (2 phi is exact), the others from
                // the one two below, brought back to modulus one (the products' roundings add up in
                // the modulus, and twice that in the template term)
                const double phi = valid ? th[3] : 0.0;
                double2 e[2];
#pragma unroll 1
                for (int j = 1; j <= 2; ++j) {
                    double sp, cp;
                    sincos(j * phi, &sp, &cp);
                    pe[j * kS + s_of] = make_double2(cp, -sp);
                }
                pe[s_of] = make_double2(1.0, 0.0);
                e[1] = pe[kS + s_of];
                const double2 two = e[0] = pe[2 * kS + s_of];
#pragma unroll
                for (int j = 3; j <= kMaxL; ++j) {
                    const double2 x = e[j & 1];
                    const double t = x.x * two.x - x.y * two.y, u = x.x * two.y + x.y * two.x;
                    const double over = 0.5 * fma(t, t, fma(u, u, -1.0));
                    pe[j * kS + s_of] = e[j & 1] = make_double2(fma(-over, t, t), fma(-over, u, u));
                }
            }
        }
        __syncthreads();
        const bool live = !producer && __any_sync(0xffffffffu, gid[s_of] != 0xffffffffu);
        // ---------------- B: delays, x F_k, harmonics, and the largest |F|^2 and |Y|^2
        if (live) {
            if (tid < kS * K) {
                const int k = grp;
                const double n0 = nv[s_of], n1 = nv[kS + s_of], n2 = nv[2 * kS + s_of];
                const Sky sk{e5[s_of], e5[kS + s_of], e5[2 * kS + s_of], e5[3 * kS + s_of]};
                // the delay in Q samples; the first bin's position is added in fixed point, so that
                // its rounding, which every bin shares, is that of the delay alone
                const double u0 = fma(P.xfs[k][0], n0, fma(P.xfs[k][1], n1, P.xfs[k][2] * n2));
                const bool valid = gid[s_of] != 0xffffffffu, ok = isfinite(u0);
                if (valid && !ok)
                    atomicOr(bad + s_of, kErrRange | kErrNonFinite);
                const long long u = ok ? X.u0[k] + __double2ll_rn(u0 * (double)(1ll << kFrac)) : 0;
                U0[k * kS + s_of] = u;
                long long ulow = valid && ok ? u : LLONG_MAX, uhigh = valid && ok ? u : LLONG_MIN;
#pragma unroll
                for (int o = 16; o; o >>= 1) {
                    ulow = min(ulow, __shfl_xor_sync(0xffffffffu, ulow, o));
                    uhigh = max(uhigh, __shfl_xor_sync(0xffffffffu, uhigh, o));
                }
                if (lane == 0 && ulow != LLONG_MAX) {
                    atomicMin(ulo + k, ulow);
                    atomicMax(uhi + k, uhigh);
                }
                Cx<double> F = response<double>(P, k, sk, ps[s_of], ps[kS + s_of]);
                const double x = ps[2 * kS + s_of];
                F.re *= x;
                F.im *= x;
                Fs[k * kS + s_of] = make_double2(F.re, F.im);
                atomicMax(mF2 + s_of, (unsigned long long)__double_as_longlong(fma(F.re, F.re, F.im * F.im)));
            }
            for (int m = grp; m < M; m += kQ) {
                double d = 0.0;
                for (int t = 0; t < P.wn[m]; ++t)
                    d += P.wcoef[m][t] * pw[P.wpc[m][t] * kS + s_of] * pw[(kPows + P.wps[m][t]) * kS + s_of];
                const int mm = P.mode_m[m];
                const double2 e = pe[(mm < 0 ? -mm : mm) * kS + s_of];
                const double2 y = make_double2(d * e.x, d * (mm < 0 ? -e.y : e.y));
                Ys[m * kS + s_of] = y;
                atomicMax(mY2 + s_of, (unsigned long long)__double_as_longlong(d * d * fma(e.x, e.x, e.y * e.y)));
            }
        }
        __syncthreads();
        // ---------------- C: the sample's scale and the digits of its coefficients
        if (live) {
            const double f2 = __longlong_as_double((long long)mF2[s_of]), y2 = __longlong_as_double((long long)mY2[s_of]);
            int ef = 0, ey = 0;
            const bool zero = !(f2 > 0.0) || !(y2 > 0.0) || !isfinite(f2) || !isfinite(y2);
            if (!zero) {
                frexp(f2, &ef);
                frexp(y2, &ey);
            }
            // |c|^2 <= f2 y2 < 2^(ef + ey): |c| < 2^ceil((ef + ey) / 2)
            const int sc = zero ? 0 : 55 - ((ef + ey + 1) >> 1);
            if (grp == 0) {
                scs[s_of] = sc;
                if (gid[s_of] != 0xffffffffu && (!isfinite(f2) || !isfinite(y2)))
                    atomicOr(bad + s_of, kErrNonFinite);
            }
            for (int it = grp; it < K * kcs; it += kQ) {
                const int k = it / kcs, kc = it - k * kcs;
                double2 f = zero ? make_double2(0.0, 0.0) : Fs[k * kS + s_of];
                f.x = mul_pow2(f.x, sc);
                f.y = mul_pow2(f.y, sc);
                uint64_t d[8];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int m = 4 * kc + j;
                    long long cr = 0, ci = 0;
                    if (m < M && !zero) {
                        const double2 y = Ys[m * kS + s_of];
                        cr = __double2ll_rn(f.x * y.x - f.y * y.y);
                        ci = __double2ll_rn(f.x * y.y + f.y * y.x);
                    }
                    d[2 * j] = digit_bytes(cr);
                    d[2 * j + 1] = digit_bytes(ci);
                }
                __half *o = scratch + ((size_t)k * kDig * kS + (size_t)(s_of >> 3) * 8) * kp + kc * 64 + (s_of & 7) * 8;
#pragma unroll
                for (int p = 0; p < kDig; ++p)
                    *reinterpret_cast<uint4 *>(o + (size_t)p * kS * kp) =
                        make_uint4(digit_pair(d[0], d[1], p), digit_pair(d[2], d[3], p), digit_pair(d[4], d[5], p),
                                   digit_pair(d[6], d[7], p));
            }
            __threadfence();
        }
        // the tables (generic accesses) share their bytes with the targets of bulk copies, and
        // the scratch is read by them
        tc::fence_proxy_async();
        __syncthreads();

        const bool any = ulo[0] != LLONG_MAX;   // a sample with finite delays
        // first column (a multiple of 8) and batches of detector k's window for the bins [j0, j1)
        auto window = [&](int k, int j0, int j1, int &w0, int &nsub) {
            const int c0 = (int)((ulo[k] + pos[j0]) >> kFrac), c1 = (int)((uhi[k] + pos[j1 - 1]) >> kFrac) + 1;
            w0 = max(c0, 0) & ~7;
            nsub = (min(c1, P.n_q - 1) - w0) / kSub + 1;
        };
        int failed = 0;
        if (warp == kIssuer) {
            if (lane == 0 && any) {
                auto batch = [&](bool wide) {   // wide: orders 0..7, else 0..6
                    const uint32_t b = g & 1u, u = g >> 1;
                    if (!tc::mbar_wait(full + b, u & 1u, kWait) ||
                        (u > 0 && !tc::mbar_wait(empty + b, (u - 1u) & 1u, kWait)))
                        return false;
                    tc::tc_fence_after();
                    const __half *B = Bs + (size_t)b * kDig * kSub * kp;
                    for (int kk = 0; kk < kp / 16; ++kk) {
                        const uint64_t bd = desc(B, 256u * (uint32_t)kk);
#pragma unroll
                        for (int i = 0; i < kDig; ++i) {
                            const uint64_t ad = desc(As + (size_t)i * kS * kp, 256u * (uint32_t)kk);
                            if (wide && i == 1)   // the first of order 7's products, by itself: it starts the sum
                                tc::mma_f16_ss(tmem + b * kAccCols + (uint32_t)(kDig * kSub), ad,
                                               desc(B + (size_t)(kDig - 1) * kSub * kp, 256u * (uint32_t)kk),
                                               tc::idesc_f16_f32(kS, kSub), kk != 0);
                            const int digits = kDig - i + (wide && i > 1 ? 1 : 0);
                            tc::mma_f16_ss(tmem + b * kAccCols + (uint32_t)(i * kSub), ad, bd,
                                           tc::idesc_f16_f32(kS, (uint32_t)(digits * kSub)), (kk | i) != 0);
                        }
                    }
                    tc::mma_commit(done + b);
                    ++g;
                    return true;
                };
                auto digits = [&]() { return tc::mbar_wait(fullA, (ga++) & 1u, kWait); };
                for (int k = 0; k < K && !failed; ++k)
                    failed = !digits() || !batch(true) || !batch(true);
                for (int ch = ch0; ch < ch1 && !failed; ++ch)
                    for (int k = 0; k < K && !failed; ++k) {
                        int w0, nsub;
                        window(k, ch * jnom, min(NT, (ch + 1) * jnom), w0, nsub);
                        if (K > 1)
                            failed = !digits();
                        for (int t = 0; t < nsub && !failed; ++t)
                            failed = !batch(false);
                    }
            }
            __syncwarp();
        } else if (warp == kStager) {
            if (lane == 0 && any) {
                auto stage = [&](const __half *src, size_t stride) {
                    const uint32_t b = g & 1u, u = g >> 1;
                    if (u > 0 && !tc::mbar_wait(done + b, (u - 1u) & 1u, kWait))
                        return false;
                    __half *dst = Bs + (size_t)b * kDig * kSub * kp;
                    tc::mbar_expect_tx(full + b, kDig * sub_bytes);
                    for (int p = 0; p < kDig; ++p)
                        tc::bulk_g2s(dst + (size_t)p * kSub * kp, src + (size_t)p * stride, sub_bytes, full + b);
                    ++g;
                    return true;
                };
                auto digits = [&](int k) {
                    // every batch so far is complete: nothing reads the old digits any more
                    if (g > 0 && !tc::mbar_wait(done + ((g - 1u) & 1u), ((g - 1u) >> 1) & 1u, kWait))
                        return false;
                    tc::mbar_expect_tx(fullA, (uint32_t)ab);
                    tc::bulk_g2s(As, scratch + (size_t)k * kDig * kS * kp, (uint32_t)ab, fullA);
                    ++ga;
                    return true;
                };
                for (int k = 0; k < K && !failed; ++k) {
                    const __half *T = X.t_dig + (size_t)k * kDig * kBlk * kp;
                    failed = !digits(k) || !stage(T, (size_t)kBlk * kp) ||
                             !stage(T + (size_t)kSub * kp, (size_t)kBlk * kp);
                }
                for (int ch = ch0; ch < ch1 && !failed; ++ch)
                    for (int k = 0; k < K && !failed; ++k) {
                        int w0, nsub;
                        window(k, ch * jnom, min(NT, (ch + 1) * jnom), w0, nsub);
                        if (K > 1)
                            failed = !digits(k);
                        const size_t part_h = (size_t)P.tc_groups * kp * 8;
                        const __half *src = X.q_dig + (size_t)k * kDig * part_h + (size_t)(w0 >> 3) * kp * 8;
                        for (int t = 0; t < nsub && !failed; ++t)
                            failed = !stage(src + (size_t)t * kSub * kp, part_h);
                    }
            }
            __syncwarp();
        } else if (any && !live) {
            // the four warps of a lane quarter without samples: its accumulators stay where they are
            auto pass = [&]() {
                const uint32_t b = g & 1u;
                const bool ok = tc::mbar_wait(done + b, (g >> 1) & 1u, kWait);
                ++g;
                __syncwarp();
                tc::mbar_arrive_if(empty + b, lane == 0);
                return ok;
            };
            for (int k = 0; k < K && !failed; ++k)
                failed = !pass() || !pass();
            for (int ch = ch0; ch < ch1 && !failed; ++ch)
                for (int k = 0; k < K && !failed; ++k) {
                    int w0, nsub;
                    window(k, ch * jnom, min(NT, (ch + 1) * jnom), w0, nsub);
                    for (int t = 0; t < nsub && !failed; ++t)
                        failed = !pass();
                }
        } else if (any) {
            const int q = warp & 3, cb = warp >> 2, s = 32 * q + lane;   // drain: quarter, 8 columns of 32
            const int gs = s_of, gh = grp;                               // gather: sample, quarter of the bins
            const bool mine = gid[gs] != 0xffffffffu && !bad[gs];
            // drain one batch of kN orders into rows 1 + 32 sub.. of R
            auto drain = [&](int sub, auto orders) {
                constexpr int kN = decltype(orders)::value;
                const uint32_t b = g & 1u;
                const int ok = tc::mbar_wait(done + b, (g >> 1) & 1u, kWait) ? 1 : 0;
                ++g;
                tc::tc_fence_after();
                long long *out = Rs + (size_t)(1 + kSub * sub + 8 * cb) * kS + s;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t v[kN][4];
#pragma unroll
                    for (int o = 0; o < kN; ++o)
                        tc::tmem_ld4(tmem + ((uint32_t)(32 * q) << 16) + b * kAccCols +
                                         (uint32_t)(o * kSub + 8 * cb + 4 * h),
                                     v[o]);
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        out[(4 * h + i) * kS] = join_orders(v, i);
                }
                tc::tc_fence_before();
                __syncwarp();
                tc::mbar_arrive_if(empty + b, lane == 0);
                return ok;
            };
            const int qbar = 2 + q;
            const int sc = scs[gs];

            // ---- template term: W = Z T, quad = kappa sum_k sum_n z_n W_n
            wide128 qacc = 0;
            int et = X.t_exp[0];
            for (int k = 1; k < K; ++k)
                et = max(et, X.t_exp[k]);
            for (int k = 0; k < K && !failed; ++k) {
                tc::named_bar_or(qbar, kConsumers / 4, 0);   // R free
                const std::integral_constant<int, kOrders> all{};
                const int ok0 = drain(0, all), ok1 = drain(1, all);
                failed = tc::named_bar_or(qbar, kConsumers / 4, !ok0 || !ok1 || abort_s);
                if (failed)
                    break;
                wide128 acc = 0;   // below 2^120
                const __half *zs = scratch + ((size_t)k * kDig * kS + (size_t)(gs >> 3) * 8) * kp + (gs & 7) * 8;
                for (int kc = gh; kc < kcs; kc += kQ) {
                    uint32_t w[kDig][4];
#pragma unroll
                    for (int p = 0; p < kDig; ++p) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(zs + (size_t)p * kS * kp + kc * 64);
                        w[p][0] = v.x;
                        w[p][1] = v.y;
                        w[p][2] = v.z;
                        w[p][3] = v.w;
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int nn = 8 * kc + j;
                        if (nn >= 2 * M)
                            break;
                        long long I = 0;
#pragma unroll
                        for (int p = 0; p < kDig; ++p) {
                            const uint32_t hb = w[p][j >> 1] >> (16 * (j & 1));
                            I = I * 256 + (long long)__half2int_rn(__ushort_as_half((unsigned short)hb));
                        }
                        acc += (wide128)I * Rs[(size_t)(1 + nn) * kS + gs];
                    }
                }
                qacc += acc >> min(et - X.t_exp[k], 127);   // (a unit of W is 2^55 of these)
            }
            // the four partials of a sample belong to the warps of its quarter (q == gs / 32); they
            // meet in rows of R behind the last component's
            long long *const qs = Rs + (size_t)(kBlk - 2 * kQ) * kS + gs;
            qs[2 * gh * kS] = (long long)qacc;
            qs[(2 * gh + 1) * kS] = (long long)(qacc >> 64);
            failed = tc::named_bar_or(qbar, kConsumers / 4, failed);
            double quad = 0.0;
            float quad_lo = 0.f;
            if (gh == 0 || lnL_t) {
                qacc = 0;
#pragma unroll
                for (int h = 0; h < kQ; ++h)
                    qacc += (wide128)qs[(2 * h + 1) * kS] << 64 | (uint64_t)qs[2 * h * kS];
                // the 62 leading bits as two doubles
                const uint64_t mag = (uint64_t)((qacc < 0 ? -qacc : qacc) >> 64);
                const int sh = mag ? __clzll((long long)mag) - 2 : 62;
                const Two v = two_of((long long)((qacc << sh) >> 64));
                const int e = 64 - sh + 56 - 2 * sc - (55 - et);
                const double lo = P.kappa * mul_pow2(v.lo, e);
                quad = P.kappa * mul_pow2(v.hi, e);
                quad_lo = fabs(lo) < 1e30 ? (float)lo : 0.f;
            }

            const int lexp = 56 - sc - sq;   // lin = X 2^lexp
            DiffScale ds;
            ds.set(lexp);
            Lse run{LLONG_MIN, 0ull};
            for (int ch = ch0; ch < ch1 && !failed; ++ch) {
                const int j0 = ch * jnom, J = min(jnom, NT - j0);
                const int jq = (J + kQ - 1) / kQ, jb = j0 + gh * jq;
                const int jn = mine ? max(0, min(jq, j0 + J - jb)) : 0;   // this thread's bins
                long long lin[kBpt];
#pragma unroll
                for (int i = 0; i < kBpt; ++i)
                    lin[i] = 0;
                for (int k = 0; k < K && !failed; ++k) {
                    int w0, nsub;
                    window(k, j0, j0 + J, w0, nsub);
                    const long long uk = U0[k * kS + gs];
                    // columns that this warp's samples reach with this thread's share of the bins:
                    // the other blocks of the window are not looked through
                    const int wlo = __reduce_min_sync(0xffffffffu, jn > 0 ? (int)((uk + pos[jb]) >> kFrac) : INT_MAX);
                    const int whi =
                        __reduce_max_sync(0xffffffffu, jn > 0 ? (int)((uk + pos[jb + jn - 1]) >> kFrac) : INT_MIN);
                    for (int t = 0; t < nsub; t += 2) {
                        tc::named_bar_or(qbar, kConsumers / 4, 0);   // the previous block's gathers are done
                        if (cb == 3 && t > 0)
                            Rs[s] = Rs[(size_t)kBlk * kS + s];
                        const std::integral_constant<int, kDig> most{};
                        int ok = drain(0, most);
                        if (t + 1 < nsub)
                            ok &= drain(1, most);
                        if ((failed = tc::named_bar_or(qbar, kConsumers / 4, !ok || abort_s)))
                            break;
                        const int rel = w0 + kSub * t - 1;
                        const unsigned cols = (unsigned)(kSub * min(2, nsub - t));
                        if (whi < rel || wlo >= rel + (int)cols)   // (also a warp without bins)
                            continue;
#pragma unroll
                        for (int i = 0; i < kBpt; ++i) {
                            const long long u = uk + pos[min(jb + i, NT - 1)];
                            const int c = (int)(u >> kFrac) - rel;
                            if (i < jn && (unsigned)c < cols) {
                                const long long *r = Rs + (size_t)c * kS + gs;
                                const long long r0 = r[0], dr = (r[kS] - r0) * 2;
                                const long long f63 = (u << (63 - kFrac)) & 0x7fffffffffffffffLL;
                                lin[i] += r0 + __mul64hi(dr, f63);
                            }
                        }
                    }
                }
                if (failed)
                    break;
                long long cm = LLONG_MIN;
#pragma unroll
                for (int i = 0; i < kBpt; ++i)
                    if (i < jn)
                        cm = max(cm, lin[i]);
                if (lnL_t) {
                    const int64_t row = (int64_t)gid[gs] * NT + jb;
                    if (gid[gs] != 0xffffffffu && !mine)   // a flagged sample has no values
                        for (int i = 0; i < jq && jb + i < j0 + J; ++i)
                            lnL_t[row + i] = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
                    for (int i = 0; i < kBpt; ++i)
                        if (i < jn)
                            lnL_t[row + i] = __dsub_rn(mul_pow2((double)lin[i], lexp), quad);
                }
                // the four threads' maxima, then their terms relative to the chunk's maximum (sums
                // of the same scale: additions, no exponentials to merge them), where R was
                tc::named_bar_or(qbar, kConsumers / 4, 0);
                Rs[gh * kS + gs] = cm;
                tc::named_bar_or(qbar, kConsumers / 4, 0);
                cm = max(max(Rs[gs], Rs[kS + gs]), max(Rs[2 * kS + gs], Rs[3 * kS + gs]));
                uint64_t terms = 0ull;
#pragma unroll
                for (int i = 0; i < kBpt; ++i)
                    if (i < jn)
                        terms += term64(ds, (uint64_t)cm - (uint64_t)lin[i], tbl);
                Rs[(kQ + gh) * kS + gs] = (long long)terms;
                tc::named_bar_or(qbar, kConsumers / 4, 0);
                if (gh == 0) {
                    const Lse c{cm, terms + (uint64_t)Rs[(kQ + 1) * kS + gs] + (uint64_t)Rs[(kQ + 2) * kS + gs] +
                                        (uint64_t)Rs[(kQ + 3) * kS + gs]};
                    if (!split)
                        run = ch == 0 ? c : merge64(ds, run, c, tbl);
                    else
                        records[((int64_t)ch * n_tiles + tile) * cut.samples + gs] = c;
                }
            }
            // the sample's value (or what the combination needs), by its first thread
            if (!failed && gh == 0 && gid[gs] != 0xffffffffu) {
                const uint32_t gi = gid[gs];
                int flags = bad[gs];
                if (!split) {
                    const double r = flags ? __longlong_as_double(0x7ff8000000000000LL)
                                           : lse_value(run, lexp, quad, quad_lo, NT);
                    if (!isfinite(r))
                        flags |= kErrNonFinite;
                    lnL_tmarg[gi] = r;
                    if (lnw && lnpw)
                        lnw[gi] = r + lnpw[gi];
                } else if (ch0 == 0) {
                    records[((int64_t)n_chunks * n_tiles + tile) * cut.samples + gs] =
                        Lse{__double_as_longlong(quad), pack_info(lexp, flags, quad_lo)};
                }
                if (flags)
                    atomicOr(err, flags);
            }
        } else if (!producer && grp == 0 && gid[s_of] != 0xffffffffu) {
            // no sample of the tile has finite delays
            const uint32_t gi = gid[s_of];
            const double r = __longlong_as_double(0x7ff8000000000000LL);
            atomicOr(err, bad[s_of] | kErrNonFinite);
            if (lnL_t)
                for (int j = ch0 * jnom; j < min(NT, ch1 * jnom); ++j)
                    lnL_t[(int64_t)gi * NT + j] = r;
            if (!split) {
                lnL_tmarg[gi] = r;
                if (lnw && lnpw)
                    lnw[gi] = r;
            } else if (ch0 == 0) {
                records[((int64_t)n_chunks * n_tiles + tile) * cut.samples + s_of] = Lse{0, pack_info(0, kErrNonFinite, 0.f)};
            }
        }
        if (fused && split)
            __threadfence();   // this thread's records, before its block's arrival
        failed = __syncthreads_or(failed || abort_s);
        if (fused && split && tid == 0) {   // (every unit arrives, a failed one too: the counts end at zero)
            last_s = atomicAdd(X.arrived + tile, 1) == parts - 1;
            if (last_s)
                X.arrived[tile] = 0;
        }
        if (failed) {
            if (tid == 0) {
                atomicOr(err, kErrTimeout);
                abort_s = 1;
            }
            __syncthreads();
            continue;
        }
        if (fused && split) {
            __syncthreads();
            if (last_s && !producer && grp == 0 && gid[s_of] != 0xffffffffu) {
                __threadfence();
                merge_sample(records, n_tiles * cut.samples, tile * cut.samples + s_of, n_chunks, NT, tbl, gid[s_of],
                             lnL_tmarg, lnpw, lnw, err);
            }
        }
    }
    // leave: no copy of this block still landing (after a failure the issuer may not have
    // consumed the last ones; bounded waits), then free the tensor memory
    if (warp == kStager && lane == 0) {
        for (uint32_t b = 0; b < 2; ++b) {
            const uint32_t uses = (g + 1u - b) >> 1;
            if (uses > 0)
                tc::mbar_wait(full + b, (uses - 1u) & 1u, kWait);
        }
        if (ga > 0)
            tc::mbar_wait(fullA, (ga - 1u) & 1u, kWait);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, 512);
    }
}

// Merges the chunks' sums of every sample (nothing to do when the bins were not split) and
// resets the unit counter, after a launch that does not merge for itself.
__global__ void combine64_kernel(const Lse *__restrict__ records, const long long *__restrict__ pos, const uint32_t *__restrict__ perm, int64_t n,
                                 const uint32_t *__restrict__ n_dev, uint32_t skip, int planned, int grid, int n_t, double *__restrict__ lnL_tmarg,
                                 const double *__restrict__ lnpw, double *__restrict__ lnw, int *err,
                                 int *unit_counter)
{
    if (blockIdx.x == 0 && threadIdx.x == 0)
        *unit_counter = 0;   // for the next launch
    const int64_t n_use = device_count(n, n_dev, skip);
    const int n_chunks = (n_t + kChunk - 1) / kChunk;
    const Cut64 cut = planned ? Cut64{kS, 1, (n_use + kS - 1) / kS} : cut64(n_use, grid, n_chunks);
    if (planned ? !has_records(cut.tiles, n_chunks) : cut.parts == 1)
        return;
    const int64_t padded = cut.tiles * cut.samples;
    __shared__ uint64_t tbl[kTable];
    for (int i = threadIdx.x; i < kTable; i += blockDim.x)
        tbl[i] = (uint64_t)pos[n_t + i];
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_use; i += (int64_t)gridDim.x * blockDim.x) {
        merge_sample(records, padded, i, n_chunks, n_t, tbl, perm ? perm[i] : (uint32_t)i, lnL_tmarg, lnpw, lnw, err);
    }
}

}  // namespace

cudaError_t launch_lnl_tc64(const Problem &P, const Tc64 &X, const double *theta, const uint32_t *perm, int64_t n,
                            double *lnL_tmarg, double *lnL_t, const double *lnpw, double *lnw, int *err,
                            cudaStream_t st, const uint32_t *n_dev, uint32_t skip, int *launched)
{
    if (n <= 0)
        return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = allow_max_dynamic_smem(lnl_tc64_kernel);
    if (e != cudaSuccess)
        return e;
    const size_t smem = std::max(kMinSmem, layout64(P.K, P.M, P.n_t).end);
    const int64_t tiles = (n + kS - 1) / kS;
    const int grid = (int)std::min<int64_t>(sms, 16 * tiles);
    // Planned are whole batches whose tiles' widths differ by more than the plan costs: two detectors
    // or more (one detector's sort key is its delay) whose delays span many batches of columns.
    // 16384 Hz, 20,011 samples: 3 detectors, 21 modes 1.06 times the speed of an even split, 2, 9
    // 1.12; 40,000 1.04 and 1.01; 12,000 0.92 and 0.94.  4096 Hz or one detector, 20,011 samples 0.98
    // to 0.99, 8200 0.72 to 0.85.  The time bins of the others are split evenly, and so are those of a
    // device-side list: its iteration has other kernels beside it or behind it, and more units mean
    // more prologues (twelve solves as one graph 9.2 -> 9.8 ms when their lists were planned).
    double span = 0.0;
    for (int k = 0; k < P.K; ++k) {
        double r2 = 0.0;
        for (int i = 0; i < 3; ++i)
            r2 += P.xfs[k][i] * P.xfs[k][i];
        span = std::max(span, 2.0 * std::sqrt(r2));
    }
    const int planned = !n_dev && tiles >= kPlanFrom && P.K > 1 && span >= kPlanSpan ? 1 : 0;
    if (planned) {
        e = cudaMemsetAsync(X.unit_counts, 0, kPlanClasses * sizeof(int), st);
        if (e != cudaSuccess)
            return e;
        units64_kernel<<<(unsigned)((tiles + kPlanWarps - 1) / kPlanWarps), 32 * kPlanWarps, 0, st>>>(
            plan_problem(P), theta, perm, n, n_dev, skip, grid, X.units, X.units_cap, X.unit_counts);
    }
    // a block per unit: the last of a tile's units merges its chunks' sums, and no kernel follows
    // (5 to 14 us of a call of 1 to 2000 samples: 512 of 2 detectors, 2 modes, 401 bins 118 -> 109,
    // the plain kernel 116)
    const Cut64 cut = cut64(n, grid, (P.n_t + kChunk - 1) / kChunk);
    const int fused = !n_dev && !planned && cut.tiles * cut.parts <= grid ? 1 : 0;
    lnl_tc64_kernel<<<grid, kThreads, smem, st>>>(P, X, theta, perm, n, lnL_tmarg, lnL_t, lnpw, lnw, err,
                                                  X.unit_counter, n_dev, skip, planned, fused);
    if (launched)
        *launched = 2 + planned - fused;
    if (fused)
        return cudaGetLastError();
    // the split depends on the device count; it never has more tiles than there are records for
    const int64_t most = std::min<int64_t>(tiles, split_tiles(n, P.n_t));
    combine64_kernel<<<(int)std::max<int64_t>(1, most), 128, 0, st>>>(reinterpret_cast<const Lse *>(X.records), X.pos, perm, n,
                                                                    n_dev, skip, planned, grid, P.n_t, lnL_tmarg, lnpw, lnw, err,
                                                                    X.unit_counter);
    return cudaGetLastError();
}

cudaError_t prepare_tc64_kernels() { return allow_max_dynamic_smem(lnl_tc64_kernel); }

}  // namespace rift
