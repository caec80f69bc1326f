// Sampler, sort and reduction kernels of the ILE hot path.
//
//   draw      - product-form adaptive sampling prior (arXiv:2505.11655 Sec. II B): every
//               extrinsic coordinate is drawn through its prior-CDF coordinate v in [0,1)
//               from a B-bin histogram, so p/p_s = prod_d 1 / (B P_d[b_d] / sum_b P_d[b]).
//   sort      - counting sort of samples by sky cell (keeps a tile's Q windows close).
//   reduce    - ln Z = ln mean w, sigma, n_eff = sum w / max w (Eq. (neff)),
//               n_ESS = (sum w)^2 / sum w^2 (Sec. IV A), all in float64, deterministic
//               two-level reductions.
//   adapt     - 1-D weighted histograms of the weights, mixed with a uniform floor.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <mutex>

#include "draws.cuh"
#include "ile_kernels.h"

namespace rift {

// ======================================================================== draw

constexpr int kDrawThreads = 256;

__global__ void __launch_bounds__(kDrawThreads) draw_kernel(SamplerDev S, SkyGrid G,
                                                            const uint32_t *__restrict__ iter_base, uint32_t iter_off,
                                                            int64_t n, double *__restrict__ theta,
                                                            double *__restrict__ lnpw, uint64_t *__restrict__ bins,
                                                            uint32_t *__restrict__ key)
{
    const uint32_t iter = *iter_base + iter_off;
    extern __shared__ double sC[];
    hist_load_tables(S, sC);
    __syncthreads();
    const uint32_t k0 = (uint32_t)S.seed, k1 = (uint32_t)(S.seed >> 32);
    const double d3lo = S.d_min * S.d_min * S.d_min, d3hi = S.d_max * S.d_max * S.d_max;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double v[6], lr, th[6];
        uint64_t packed;
        hist_draw_one(sC, S.B, S.marg, iter, i, k0, k1, v, lr, packed);
        hist_theta(v, d3lo, d3hi, th);
        double *out = theta + 6 * i;
#pragma unroll
        for (int d = 0; d < 6; ++d)
            out[d] = th[d];
        lnpw[i] = lr;
        bins[i] = packed;
        // on the (right ascension, sin declination) grid the cell follows from the prior
        // coordinates themselves: alpha / 2 pi = v0 and (sin delta + 1) / 2 = v1
        key[i] = G.mode == kSortSky ? sky_cell_v(v[0], v[1], G) : sky_cell(th[0], th[1], G);
    }
}

static int sm_count()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

static int grid_for(int64_t n, int threads, int per_sm)
{
    int64_t want = (n + threads - 1) / threads;
    int64_t cap = (int64_t)sm_count() * per_sm;
    return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

cudaError_t launch_draw(const SamplerDev &S, const SkyGrid &G, const uint32_t *iter_base, uint32_t iter_off, int64_t n,
                        double *theta, double *lnpw, uint64_t *bins, uint32_t *key, cudaStream_t st)
{
    if (n <= 0)
        return cudaSuccess;
    size_t smem = sizeof(double) * hist_table_doubles(S.B);
    if (smem > 48 * 1024) {
        cudaError_t e = allow_max_dynamic_smem(draw_kernel);
        if (e != cudaSuccess)
            return e;
    }
    draw_kernel<<<grid_for(n, kDrawThreads, 8), kDrawThreads, smem, st>>>(S, G, iter_base, iter_off, n, theta, lnpw, bins, key);
    return cudaGetLastError();
}

__global__ void keys_kernel(SkyGrid G, const double *__restrict__ theta, int64_t n, uint32_t *__restrict__ key)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        key[i] = sky_cell(theta[6 * i], theta[6 * i + 1], G);
}

cudaError_t launch_keys(const SkyGrid &G, const double *theta, int64_t n, uint32_t *key, cudaStream_t st)
{
    if (n <= 0)
        return cudaSuccess;
    keys_kernel<<<grid_for(n, 256, 8), 256, 0, st>>>(G, theta, n, key);
    return cudaGetLastError();
}

SkyGrid sky_grid_for(int64_t n, int per_cell)
{
    int order = 4;
    while (order < kMaxOrder && ((int64_t)per_cell << (2 * order)) < n)
        ++order;
    return SkyGrid{order, 1 << (2 * order)};
}

// ======================================================================== stable sort by sky cell
//
// Least-significant-digit radix sort of the keys (digits of up to 10 bits, as wide as the keys
// need for the fewest passes), stable in the sample index: samples of one cell keep their draw
// order, so the tiles the likelihood kernels form, and with them every float32 result, are the
// same from run to run.  Each pass:
//   hist     digit counts of every tile of 2048 keys, and their totals per digit;
//   rows     exclusive sums of each digit's counts over the tiles;
//   scatter  each warp ranks its contiguous 256 keys of the tile digit by digit with a warp
//            match (ranks in registers), then writes every key at digit base + tile row + rank.
// The work of a pass is a few microseconds; what bounds it is the latency of one block's chain
// of rounds, so the tiles are small enough to spread 50,000 keys over 25 SMs (with 8192-key
// tiles and a three-kernel scan of the counts a sort of 250,000 20-bit keys took 180 us).
// Up to 4096 keys are sorted by one block instead: (key, index) words by a bitonic network.

constexpr int kRadixThreads = 256;
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kRadixRounds = 8;
constexpr int kRadixPerWarp = 32 * kRadixRounds;
constexpr int kRadixTile = kRadixWarps * kRadixPerWarp;
constexpr int kSmallSort = 4096;      // keys of a one-block sort (12 index bits beside 20 key bits)
constexpr int kSmallThreads = 1024;

template <typename K>
__global__ void __launch_bounds__(kRadixThreads) radix_hist_kernel(const K *__restrict__ keys, int64_t n, int shift,
                                                                   int buckets, uint32_t *__restrict__ hist,
                                                                   uint32_t *__restrict__ totals)
{
    __shared__ uint32_t h[kRadixBuckets];
    for (int d = threadIdx.x; d < buckets; d += kRadixThreads)
        h[d] = 0u;
    const int64_t base = (int64_t)blockIdx.x * kRadixTile;
    K k[kRadixRounds];
#pragma unroll
    for (int r = 0; r < kRadixRounds; ++r) {
        const int64_t i = base + r * kRadixThreads + threadIdx.x;
        k[r] = i < n ? keys[i] : (K)0;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRadixRounds; ++r)
        if (base + r * kRadixThreads + threadIdx.x < n)
            atomicAdd(&h[(uint32_t)(k[r] >> shift) & (uint32_t)(buckets - 1)], 1u);
    __syncthreads();
    for (int d = threadIdx.x; d < buckets; d += kRadixThreads) {
        const uint32_t c = h[d];
        hist[(size_t)blockIdx.x * buckets + d] = c;
        if (c)
            atomicAdd(totals + d, c);
    }
}

// One block per 32 digits (a lane each); warp w owns a contiguous range of tiles.
__global__ void __launch_bounds__(1024) radix_rows_kernel(uint32_t *__restrict__ hist, int nblk, int buckets)
{
    __shared__ uint32_t tot[32][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t *col = hist + blockIdx.x * 32 + lane;
    const int per = (nblk + 31) / 32, b0 = min(nblk, w * per), b1 = min(nblk, b0 + per);
    uint32_t sum = 0;
#pragma unroll 8
    for (int b = b0; b < b1; ++b)
        sum += col[(size_t)b * buckets];
    tot[w][lane] = sum;
    __syncthreads();
    uint32_t run = 0;
    for (int v = 0; v < w; ++v)
        run += tot[v][lane];
#pragma unroll 8
    for (int b = b0; b < b1; ++b) {
        const uint32_t c = col[(size_t)b * buckets];
        col[(size_t)b * buckets] = run;
        run += c;
    }
}

template <typename K>
__global__ void __launch_bounds__(kRadixThreads) radix_scatter_kernel(const K *__restrict__ keys_in,
                                                                      const uint32_t *__restrict__ vals_in, int64_t n,
                                                                      int shift, int buckets,
                                                                      const uint32_t *__restrict__ hist,
                                                                      const uint32_t *__restrict__ totals,
                                                                      K *__restrict__ keys_out,
                                                                      uint32_t *__restrict__ vals_out)
{
    __shared__ uint32_t wpos[kRadixWarps][kRadixBuckets];   // per-warp digit counts, then positions
    __shared__ uint32_t wtot[kRadixWarps];
    constexpr int kPer = kRadixBuckets / kRadixThreads;     // digits per thread in the scan of the totals
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int d = threadIdx.x; d < buckets; d += kRadixThreads)
#pragma unroll
        for (int v = 0; v < kRadixWarps; ++v)
            wpos[v][d] = 0u;
    const int64_t base = (int64_t)blockIdx.x * kRadixTile + (int64_t)w * kRadixPerWarp;
    K k[kRadixRounds];
    uint32_t rank[kRadixRounds];
#pragma unroll
    for (int r = 0; r < kRadixRounds; ++r) {
        const int64_t i = base + 32 * r + lane;
        k[r] = i < n ? keys_in[i] : (K)0;
    }
    // exclusive sums of the digit totals: kPer consecutive digits per thread
    uint32_t t[kPer], mine = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int d = threadIdx.x * kPer + q;
        t[q] = mine;
        mine += d < buckets ? totals[d] : 0u;
    }
    uint32_t x = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o)
            x += y;
    }
    if (lane == 31)
        wtot[w] = x;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRadixRounds; ++r) {
        const bool ok = base + 32 * r + lane < n;
        const uint32_t d = ok ? (uint32_t)(k[r] >> shift) & (uint32_t)(buckets - 1) : 0xffffffffu;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        uint32_t before = 0;
        if (ok)
            before = wpos[w][d];
        __syncwarp();
        rank[r] = before + __popc(peers & ((1u << lane) - 1u));
        if (ok && lane == __ffs(peers) - 1)
            wpos[w][d] = before + (uint32_t)__popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // first position of each digit for each warp: the digit's base, the tile's row, then the
    // warps in order
    uint32_t off = x - mine;
    for (int v = 0; v < w; ++v)
        off += wtot[v];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int d = threadIdx.x * kPer + q;
        if (d >= buckets)
            break;
        uint32_t run = off + t[q] + hist[(size_t)blockIdx.x * buckets + d];
#pragma unroll
        for (int v = 0; v < kRadixWarps; ++v) {
            const uint32_t c = wpos[v][d];
            wpos[v][d] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRadixRounds; ++r) {
        const int64_t i = base + 32 * r + lane;
        if (i < n) {
            const uint32_t pos = wpos[w][(uint32_t)(k[r] >> shift) & (uint32_t)(buckets - 1)] + rank[r];
            if (vals_out)
                vals_out[pos] = vals_in ? vals_in[i] : (uint32_t)i;
            if (keys_out)
                keys_out[pos] = k[r];
        }
    }
}

// At most kSmallSort keys of at most 20 bits, one block: words (key, index) are distinct, so
// any sort of them is the stable one; the network runs over `size` words, a power of two.
__global__ void __launch_bounds__(kSmallThreads) small_sort_kernel(const uint32_t *__restrict__ keys, int n, int size,
                                                                   uint32_t *__restrict__ perm)
{
    __shared__ uint32_t a[kSmallSort];
    for (int i = threadIdx.x; i < size; i += (int)blockDim.x)
        a[i] = i < n ? (keys[i] << 12) | (uint32_t)i : 0xffffffffu;
    for (int len = 2; len <= size; len <<= 1)
        for (int step = len >> 1; step > 0; step >>= 1) {
            __syncthreads();
            for (int e = threadIdx.x; e < size / 2; e += (int)blockDim.x) {
                const int i = 2 * e - (e & (step - 1)), j = i + step;
                const uint32_t u = a[i], v = a[j];
                if ((u > v) == ((i & len) == 0)) {
                    a[i] = v;
                    a[j] = u;
                }
            }
        }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += (int)blockDim.x)
        perm[i] = a[i] & 4095u;
}

// Exclusive scan of L counts in place: per-tile totals of 4096 counts, a scan of the
// totals (recursively when there are more than 1024 tiles), then a block-level scan
// of each tile offset by its total.  Coalesced loads and stores; each thread owns 16
// consecutive counts staged through shared memory.  32-bit for the sort, 64-bit for
// the fair draws' fixed-point weights.
constexpr int kScanTile = 4096;
constexpr int kScanThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kScanThreads) scan_totals_kernel(const T *__restrict__ counts, int n_cells,
                                                                   T *__restrict__ totals)
{
    __shared__ T red[kScanThreads / 32];
    const int base = blockIdx.x * kScanTile;
    T v = 0;
    for (int i = threadIdx.x; i < kScanTile; i += kScanThreads)
        if (base + i < n_cells)
            v += counts[base + i];
#pragma unroll
    for (int o = 16; o; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0)
        red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        T t = 0;
        for (int w = 0; w < kScanThreads / 32; ++w)
            t += red[w];
        totals[blockIdx.x] = t;
    }
}

// Block-wide exclusive scan of one value per thread; returns this thread's offset.
template <typename T> __device__ T block_exclusive_scan(T v, T *warp_tot)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o)
            x += y;
    }
    if (lane == 31)
        warp_tot[w] = x;
    __syncthreads();
    if (w == 0) {
        T t = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : (T)0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o)
                t += y;
        }
        warp_tot[lane] = t;
    }
    __syncthreads();
    return x - v + (w > 0 ? warp_tot[w - 1] : (T)0);
}

template <typename T> __global__ void __launch_bounds__(1024) scan_top_kernel(T *totals, int nb)
{
    __shared__ T warp_tot[32];
    const T v = threadIdx.x < nb ? totals[threadIdx.x] : (T)0;
    const T e = block_exclusive_scan(v, warp_tot);
    if (threadIdx.x < nb)
        totals[threadIdx.x] = e;
}

template <typename T>
__global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(T *__restrict__ counts, int n_cells,
                                                                  const T *__restrict__ totals)
{
    constexpr int per = kScanTile / kScanThreads;
    __shared__ T tile[kScanTile + kScanTile / 32];   // padded: thread-strided reads avoid conflicts
    __shared__ T warp_tot[32];
    const int base = blockIdx.x * kScanTile;
    for (int i = threadIdx.x; i < kScanTile; i += kScanThreads)
        tile[i + (i >> 5)] = base + i < n_cells ? counts[base + i] : (T)0;
    __syncthreads();
    T loc[per], run = 0;
#pragma unroll
    for (int q = 0; q < per; ++q) {
        const int i = threadIdx.x * per + q;
        loc[q] = run;
        run += tile[i + (i >> 5)];
    }
    const T off = block_exclusive_scan(run, warp_tot) + totals[blockIdx.x];
#pragma unroll
    for (int q = 0; q < per; ++q) {
        const int i = threadIdx.x * per + q;
        tile[i + (i >> 5)] = off + loc[q];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kScanTile; i += kScanThreads)
        if (base + i < n_cells)
            counts[base + i] = tile[i + (i >> 5)];
}

// Exclusive scan of data[0, L) in place; scratch holds the totals of every level.
template <typename T> static int launch_scan(T *data, int L, T *scratch, cudaStream_t st)
{
    const int nb = (L + kScanTile - 1) / kScanTile;
    scan_totals_kernel<T><<<nb, kScanThreads, 0, st>>>(data, L, scratch);
    int launched = 1;
    if (nb <= 1024) {
        scan_top_kernel<T><<<1, 1024, 0, st>>>(scratch, nb);
        ++launched;
    } else {
        launched += launch_scan<T>(scratch, nb, scratch + nb, st);
    }
    scan_apply_kernel<T><<<nb, kScanThreads, 0, st>>>(data, L, scratch);
    return launched + 1;
}

size_t scan_scratch_words(int64_t L)
{
    size_t words = 0;
    while (L > 1) {
        L = (L + kScanTile - 1) / kScanTile;
        words += (size_t)L;
    }
    return words + 1;
}

cudaError_t launch_scan_u64(uint64_t *data, int64_t L, uint64_t *scratch, cudaStream_t st, int *launched)
{
    const int k = L > 0 ? launch_scan<uint64_t>(data, (int)L, scratch, st) : 0;
    if (launched)
        *launched = k;
    return cudaGetLastError();
}

// digit counts of every tile and pass totals
static size_t radix_words(int64_t n_max)
{
    const int64_t nblk = (n_max + kRadixTile - 1) / kRadixTile;
    return (size_t)kRadixBuckets * (size_t)((nblk > 0 ? nblk : 1) + kRadixPasses);
}

size_t sort_scratch_words(int64_t n_max) { return radix_words(n_max) + (size_t)(2 * n_max + 64); }

size_t sort64_scratch_words(int64_t n_max) { return radix_words(n_max) + 64; }

// One pass over the digit of `bits` bits at `shift`; totals zeroed by the caller.
template <typename K>
static void radix_pass(const K *in, const uint32_t *vin, int64_t n, int shift, int bits, uint32_t *hist,
                       uint32_t *totals, K *out, uint32_t *vout, cudaStream_t st)
{
    const int nblk = (int)((n + kRadixTile - 1) / kRadixTile), buckets = 1 << bits;
    radix_hist_kernel<K><<<nblk, kRadixThreads, 0, st>>>(in, n, shift, buckets, hist, totals);
    radix_rows_kernel<<<buckets / 32, 1024, 0, st>>>(hist, nblk, buckets);
    radix_scatter_kernel<K><<<nblk, kRadixThreads, 0, st>>>(in, vin, n, shift, buckets, hist, totals, out, vout);
}

// passes of a sort of `bits`-bit keys, and the digit width (5 bits at least: whole warps of
// digits)
static int radix_plan(int bits, int *digit)
{
    const int passes = bits <= 0 ? 0 : (bits + kRadixBits - 1) / kRadixBits;
    *digit = passes ? std::max(5, (bits + passes - 1) / passes) : 0;
    return passes;
}

cudaError_t launch_sort(const SkyGrid &G, const uint32_t *key, int64_t n, uint32_t *scratch, uint32_t *perm,
                        cudaStream_t st, int *launched)
{
    if (launched)
        *launched = 0;
    if (n <= 0)
        return cudaSuccess;
    int bits = 0, digit = 0;
    while ((1ll << bits) < (int64_t)G.n_cells)
        ++bits;
    if (n <= kSmallSort && bits <= 20) {
        int size = 2;
        while (size < n)
            size <<= 1;
        small_sort_kernel<<<1, std::min(kSmallThreads, std::max(32, size / 2)), 0, st>>>(key, (int)n, size, perm);
        if (launched)
            *launched = 1;
        return cudaGetLastError();
    }
    const int passes = radix_plan(std::max(bits, 1), &digit);
    uint32_t *totals = scratch, *hist = totals + kRadixPasses * kRadixBuckets;
    uint32_t *key_tmp = scratch + radix_words(n), *val_tmp = key_tmp + n;
    cudaError_t e = cudaMemsetAsync(totals, 0, sizeof(uint32_t) * kRadixBuckets * passes, st);
    if (e != cudaSuccess)
        return e;
    for (int pass = 0; pass < passes; ++pass) {
        const bool last = pass == passes - 1;
        radix_pass<uint32_t>(pass == 0 ? key : key_tmp, pass == 0 ? nullptr : val_tmp, n, pass * digit, digit, hist,
                             totals + pass * kRadixBuckets, last ? nullptr : key_tmp, last ? perm : val_tmp, st);
    }
    if (launched)
        *launched = 3 * passes;
    return cudaGetLastError();
}

cudaError_t launch_sort64(uint64_t *keys, uint64_t *tmp, int64_t n, int bits, uint32_t *scratch, cudaStream_t st,
                          int *launched)
{
    if (launched)
        *launched = 0;
    if (n <= 0)
        return cudaSuccess;
    int digit = 0;
    const int passes = radix_plan(bits, &digit);
    if (passes > kRadixPasses)
        return cudaErrorInvalidValue;
    uint32_t *totals = scratch, *hist = totals + kRadixPasses * kRadixBuckets;
    if (passes) {
        cudaError_t e = cudaMemsetAsync(totals, 0, sizeof(uint32_t) * kRadixBuckets * passes, st);
        if (e != cudaSuccess)
            return e;
    }
    uint64_t *in = keys, *out = tmp;
    for (int pass = 0; pass < passes; ++pass) {
        radix_pass<uint64_t>(in, nullptr, n, pass * digit, digit, hist, totals + pass * kRadixBuckets, out, nullptr, st);
        std::swap(in, out);
    }
    if (in != keys) {   // odd number of passes: the sorted keys are in tmp
        cudaError_t e = cudaMemcpyAsync(keys, in, sizeof(uint64_t) * n, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess)
            return e;
    }
    if (launched)
        *launched = 3 * passes;
    return cudaGetLastError();
}

cudaError_t launch_scan_u32(uint32_t *data, int64_t L, uint32_t *scratch, cudaStream_t st, int *launched)
{
    const int k = L > 0 ? launch_scan<uint32_t>(data, (int)L, scratch, st) : 0;
    if (launched)
        *launched = k;
    return cudaGetLastError();
}

// ======================================================================== reductions (float64)

constexpr int kRedThreads = 256;

struct Acc {
    double mx, s1, s2, lmx;
    int bad;
};

__device__ __forceinline__ Acc acc_merge(Acc a, Acc b)
{
    Acc r;
    r.mx = fmax(a.mx, b.mx);
    double fa = (a.mx == -INFINITY) ? 0.0 : exp(a.mx - r.mx);
    double fb = (b.mx == -INFINITY) ? 0.0 : exp(b.mx - r.mx);
    r.s1 = a.s1 * fa + b.s1 * fb;
    r.s2 = a.s2 * fa * fa + b.s2 * fb * fb;
    r.lmx = fmax(a.lmx, b.lmx);
    r.bad = a.bad | b.bad;
    return r;
}

// Block-wide maximum of (mx, lmx, bad), then sum of (s1, s2).  The maximum comes first and the
// sums are taken relative to it, so that no merge step needs an exponential: a float64
// exponential is a chain of some forty operations on this part's slow float64 pipe, and the
// former merge of (maximum, sums) records had two of them at each of its ten levels (250,000
// samples: 52 + 35 us for the partial sums and the final merge).
__device__ void block_max(Acc &a)
{
    __shared__ double smx[32], slm[32];
    __shared__ int sbad[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        a.mx = fmax(a.mx, __shfl_xor_sync(0xffffffffu, a.mx, o));
        a.lmx = fmax(a.lmx, __shfl_xor_sync(0xffffffffu, a.lmx, o));
        a.bad |= __shfl_xor_sync(0xffffffffu, a.bad, o);
    }
    if (lane == 0) {
        smx[w] = a.mx;
        slm[w] = a.lmx;
        sbad[w] = a.bad;
    }
    __syncthreads();
    for (int v = 0; v < nw; ++v) {
        a.mx = fmax(a.mx, smx[v]);
        a.lmx = fmax(a.lmx, slm[v]);
        a.bad |= sbad[v];
    }
}

__device__ void block_sum(Acc &a)   // every thread gets the sums
{
    __shared__ double ss1[32], ss2[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        a.s1 += __shfl_xor_sync(0xffffffffu, a.s1, o);
        a.s2 += __shfl_xor_sync(0xffffffffu, a.s2, o);
    }
    if (lane == 0) {
        ss1[w] = a.s1;
        ss2[w] = a.s2;
    }
    __syncthreads();
    a.s1 = a.s2 = 0.0;
    for (int v = 0; v < nw; ++v) {
        a.s1 += ss1[v];
        a.s2 += ss2[v];
    }
}

// exp(t) for t <= 0: float64, or float32 for terms that carry float32 errors already
// (float64 exponentials run on this part's slow float64 pipe)
__device__ __forceinline__ double term_exp(double t, bool f32)
{
    return f32 ? (double)expf((float)t) : exp(t);
}

// Pass 1: per block, over a contiguous stripe (deterministic for a fixed n).
__global__ void __launch_bounds__(kRedThreads) reduce_partial_kernel(const double *__restrict__ lnw,
                                                                     const double *__restrict__ lnL, int64_t n,
                                                                     double *__restrict__ partial, bool f32)
{
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = (int64_t)blockIdx.x * per;
    const int64_t b1 = min(n, b0 + per);
    // the stripe's maximum first, then sums relative to it
    Acc a{-INFINITY, 0.0, 0.0, -INFINITY, 0};
    for (int64_t i = b0 + threadIdx.x; i < b1; i += blockDim.x) {
        const double x = lnw[i];
        if (!isfinite(x)) {
            a.bad = 1;
            continue;
        }
        a.mx = fmax(a.mx, x);
        a.lmx = fmax(a.lmx, lnL[i]);
    }
    block_max(a);
    for (int64_t i = b0 + threadIdx.x; i < b1; i += blockDim.x) {
        const double x = lnw[i];
        // (a term below e^-60 of the stripe's largest cannot reach the sums' last bit, however many
        // of the at most 2^31 samples are such; most samples of a loud event are)
        if (!isfinite(x) || x - a.mx < -60.0)
            continue;
        const double e = term_exp(x - a.mx, f32);
        a.s1 += e;
        a.s2 += e * e;
    }
    block_sum(a);
    if (threadIdx.x == 0) {
        double *o = partial + 5 * blockIdx.x;
        o[0] = a.mx;
        o[1] = a.s1;
        o[2] = a.s2;
        o[3] = a.lmx;
        o[4] = (double)a.bad;
    }
}

// Pass 2: one block merges the partials in block order; writes the iteration's
// statistics and merges them into the pooled accumulators.
__global__ void __launch_bounds__(kRedThreads) reduce_final_kernel(const double *__restrict__ partial, int nb, int64_t n,
                                                                   double *__restrict__ stats, int slot,
                                                                   double *__restrict__ pooled, int reset, int *err)
{
    Acc a{-INFINITY, 0.0, 0.0, -INFINITY, 0};
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        const double *o = partial + 5 * b;
        a.mx = fmax(a.mx, o[0]);
        a.lmx = fmax(a.lmx, o[3]);
        a.bad |= o[4] != 0.0;
    }
    block_max(a);
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        const double *o = partial + 5 * b;
        if (o[0] == -INFINITY)
            continue;
        const double f = exp(o[0] - a.mx);
        a.s1 += o[1] * f;
        a.s2 += o[2] * f * f;
    }
    block_sum(a);
    // the record and the pooled one by a warp per float64 chain (every thread has the sums)
    const double N = (double)n;
    double *s = stats + 8 * slot;
    __shared__ double ln_n;
    double ln_s1 = 0.0;
    if (threadIdx.x == 0) {
        ln_s1 = log(a.s1);
    } else if (threadIdx.x == 32) {
        ln_n = log(N);
    } else if (threadIdx.x == 64) {
        const double var = a.s2 / (a.s1 * a.s1) - 1.0 / N;
        s[1] = sqrt(var > 0.0 ? var : 0.0);
    } else if (threadIdx.x == 96) {
        Acc pool = reset ? Acc{-INFINITY, 0.0, 0.0, -INFINITY, 0} : Acc{pooled[0], pooled[1], pooled[2], pooled[4], 0};
        const double pn = reset ? 0.0 : pooled[3];
        pool = acc_merge(pool, a);
        pooled[0] = pool.mx;
        pooled[1] = pool.s1;
        pooled[2] = pool.s2;
        pooled[3] = pn + N;
        pooled[4] = pool.lmx;
    } else if (threadIdx.x == 128) {
        s[2] = a.s1;
        s[3] = a.s1 * a.s1 / a.s2;
        s[4] = a.mx;
        s[5] = a.lmx;
        s[6] = N;
        s[7] = 0.0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        s[0] = a.mx + ln_s1 - ln_n;
        if (a.bad || !isfinite(s[0]))
            atomicOr(err, kErrNonFinite);
    }
}

cudaError_t launch_reduce(const double *lnw, const double *lnL, int64_t n, double *partial, double *stats, int slot,
                          double *pooled, int reset_pooled, int *err, cudaStream_t st, bool f32_terms)
{
    int nb = kRedBlocks;
    if ((int64_t)nb * 64 > n)
        nb = (int)((n + 63) / 64);
    if (nb < 1)
        nb = 1;
    reduce_partial_kernel<<<nb, kRedThreads, 0, st>>>(lnw, lnL, n, partial, f32_terms);
    reduce_final_kernel<<<1, kRedThreads, 0, st>>>(partial, nb, n, stats, slot, pooled, reset_pooled, err);
    return cudaGetLastError();
}

__global__ void pooled_final_kernel(const double *__restrict__ pooled, double *__restrict__ out, uint32_t *iter_base,
                                    uint32_t advance)
{
    *iter_base += advance;
    double N = pooled[3];
    double var = pooled[2] / (pooled[1] * pooled[1]) - 1.0 / N;
    out[0] = pooled[0] + log(pooled[1]) - log(N);
    out[1] = sqrt(var > 0.0 ? var : 0.0);
    out[2] = pooled[1];
    out[3] = pooled[1] * pooled[1] / pooled[2];
    out[4] = pooled[4];
    out[5] = N;
}

cudaError_t launch_pooled_final(const double *pooled, double *out, uint32_t *iter_base, uint32_t advance,
                                cudaStream_t st)
{
    pooled_final_kernel<<<1, 1, 0, st>>>(pooled, out, iter_base, advance);
    return cudaGetLastError();
}

// ======================================================================== adaptation

constexpr int kHistBlocks = 152;

// Histogram weights are summed exactly, in 128-bit fixed point with 2^-90 resolution
// (lo, hi words): integer addition does not depend on the order in which samples
// arrive, so the adapted sampler is bitwise reproducible however the blocks and
// atomics interleave (and a solve's result does not depend on what else runs).
// Weights are w = exp(beta (ln w_i - max ln w)) <= 1; at most 2^31 samples keep the
// sum below 2^121.
constexpr int kFixShift = 90;

__device__ __forceinline__ void to_fixed(double w, uint64_t &lo, uint64_t &hi)
{
    lo = hi = 0;
    if (!(w > 0.0))
        return;
    w = fmin(w, 1.0);
    const uint64_t bits = (uint64_t)__double_as_longlong(w);
    const int e = (int)((bits >> 52) & 0x7ff) - 1023;
    if (e < -kFixShift - 1)
        return;
    const uint64_t m = (bits & ((1ull << 52) - 1)) | (1ull << 52);   // w = m 2^(e-52)
    const int s = e - 52 + kFixShift;                                  // W = m 2^s
    if (s >= 64) {
        hi = m << (s - 64);
    } else if (s > 0) {
        lo = m << s;
        hi = m >> (64 - s);
    } else if (s > -64) {
        lo = m >> (-s);
    }
}

__device__ __forceinline__ void add_fixed(unsigned long long *lo, unsigned long long *hi, uint64_t a_lo, uint64_t a_hi)
{
    if (a_lo) {
        const unsigned long long old = atomicAdd(lo, (unsigned long long)a_lo);
        if (old + a_lo < old)
            ++a_hi;   // this addition wrapped the low word
    }
    if (a_hi)
        atomicAdd(hi, (unsigned long long)a_hi);
}

__global__ void __launch_bounds__(256) hist_partial_kernel(SamplerDev S, const uint64_t *__restrict__ bins,
                                                           const double *__restrict__ lnw, int64_t n,
                                                           const double *__restrict__ stats, int slot,
                                                           uint64_t *__restrict__ partial, bool f32)
{
    extern __shared__ unsigned long long sF[];   // [6][B][2] = (lo, hi) per bin
    const int B = S.B;
    for (int e = threadIdx.x; e < 12 * B; e += blockDim.x)
        sF[e] = 0ull;
    __syncthreads();
    const double mx = stats[8 * slot + 4];
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = (int64_t)blockIdx.x * per, b1 = min(n, b0 + per);
    for (int64_t i = b0 + threadIdx.x; i < b1; i += blockDim.x) {
        double x = lnw[i];
        if (!isfinite(x))
            continue;
        const double t = S.temper * (x - mx);
        if (t < -64.0)   // below 2^-92: zero in the sums' resolution
            continue;
        uint64_t lo, hi;
        to_fixed(term_exp(t, f32), lo, hi);
        if (!(lo | hi))
            continue;
        uint64_t pk = bins[i];
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            const int e = d * B + (int)((pk >> (10 * d)) & 1023u);
            add_fixed(&sF[2 * e], &sF[2 * e + 1], lo, hi);
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 12 * B; e += blockDim.x)
        partial[(size_t)blockIdx.x * 12 * B + e] = sF[e];
}

// Masses P of dimension d and their running sums C (shared memory) to the sampler's tables.
__device__ __forceinline__ void write_cdf(const SamplerDev &S, int d, const double *P, const double *C)
{
    const int B = S.B;
    if (threadIdx.x == 0)
        S.C[d * (B + 1)] = 0.0;
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
        S.P[d * B + b] = P[b];
        S.C[d * (B + 1) + b + 1] = C[b];
        S.L[d * B + b] = log(B * P[b] / C[B - 1]);
    }
}

// Sum the partial histograms exactly (128-bit); P <- (1-eps) H / sum H + eps / B; rebuild C.
// One block per dimension: the bins' sums over the block partials are split across the
// block's threads (integer sums, so the same H in any split), then one warp finishes.
constexpr int kAdaptFinalThreads = 256;
__global__ void __launch_bounds__(kAdaptFinalThreads) adapt_final_kernel(SamplerDev S,
                                                                         const uint64_t *__restrict__ partial, int nb)
{
    const int B = S.B, d = blockIdx.x;
    if (d >= 6 || (S.marg && d == 5))   // a marginalised distance keeps its masses
        return;
    // (the masses and their running sums in shared memory: a serial loop over global memory
    // was most of this kernel's time)
    __shared__ double H[RIFT_MAX_BINS], C[RIFT_MAX_BINS];
    __shared__ unsigned long long acc[3][kAdaptFinalThreads];
    const int tpb = B < kAdaptFinalThreads ? kAdaptFinalThreads / B : 1;   // threads per bin
    const int t = threadIdx.x, j = t % tpb, b0 = t / tpb, bstride = kAdaptFinalThreads / tpb;
    for (int bb = 0; bb < B; bb += bstride) {
        const int b = bb + b0;
        const bool mine = b0 < bstride && b < B;
        // the low words are summed as two 32-bit halves (no carry chain between the
        // loads), then recombined exactly
        uint64_t l0 = 0, l1 = 0, hi = 0;
        if (mine) {
#pragma unroll 4
            for (int k = j; k < nb; k += tpb) {
                const uint64_t *q = partial + (size_t)k * 12 * B + 2 * (d * B + b);
                const uint64_t lo = q[0];
                l0 += lo & 0xffffffffull;
                l1 += lo >> 32;
                hi += q[1];
            }
        }
        acc[0][t] = l0;
        acc[1][t] = l1;
        acc[2][t] = hi;
        __syncthreads();
        if (mine && j == 0) {
            for (int u = 1; u < tpb; ++u) {
                l0 += acc[0][t + u];
                l1 += acc[1][t + u];
                hi += acc[2][t + u];
            }
            const uint64_t a = l0 + (l1 << 32);
            hi += (l1 >> 32) + (a < l0 ? 1u : 0u);
            H[b] = ldexp((double)hi, 64 - kFixShift) + ldexp((double)a, -kFixShift);
        }
        __syncthreads();
    }
    if (t < 32) {
        double tot = 0.0;
        for (int b = t; b < B; b += 32)
            tot += H[b];
#pragma unroll
        for (int o = 16; o; o >>= 1)
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
        const bool adapt = tot > 0.0 && isfinite(tot);
        for (int b = t; b < B; b += 32)
            H[b] = adapt ? (1.0 - S.floor_eps) * H[b] / tot + S.floor_eps / B : S.P[d * B + b];
        __syncwarp();
        if (t == 0) {
            double run = 0.0;
            for (int b = 0; b < B; ++b)
                C[b] = run += H[b];
        }
    }
    __syncthreads();
    write_cdf(S, d, H, C);
}

cudaError_t launch_adapt(const SamplerDev &S, const uint64_t *bins, const double *lnw, int64_t n, const double *stats,
                         int slot, uint64_t *hist_partial, cudaStream_t st, bool f32_terms)
{
    int nb = kHistBlocks;
    if ((int64_t)nb * 256 > n)
        nb = (int)((n + 255) / 256);
    if (nb < 1)
        nb = 1;
    size_t smem = sizeof(uint64_t) * 12 * S.B;
    if (smem > 48 * 1024) {
        cudaError_t e = allow_max_dynamic_smem(hist_partial_kernel);
        if (e != cudaSuccess)
            return e;
    }
    hist_partial_kernel<<<nb, 256, smem, st>>>(S, bins, lnw, n, stats, slot, hist_partial, f32_terms);
    adapt_final_kernel<<<6, kAdaptFinalThreads, 0, st>>>(S, hist_partial, nb);
    return cudaGetLastError();
}

// One block per dimension (one thread a dimension, with a logarithm per bin in turn, took 93 us
// for 64 bins).
__global__ void __launch_bounds__(128) build_cdf_kernel(SamplerDev S)
{
    __shared__ double P[RIFT_MAX_BINS], C[RIFT_MAX_BINS];
    const int d = blockIdx.x;
    for (int b = threadIdx.x; b < S.B; b += blockDim.x)
        P[b] = S.P[d * S.B + b];
    __syncthreads();
    if (threadIdx.x == 0) {
        double run = 0.0;
        for (int b = 0; b < S.B; ++b)
            C[b] = run += P[b];
    }
    __syncthreads();
    write_cdf(S, d, P, C);
}

cudaError_t launch_build_cdf(const SamplerDev &S, cudaStream_t st)
{
    build_cdf_kernel<<<6, 128, 0, st>>>(S);
    return cudaGetLastError();
}

cudaError_t prepare_sampler_kernels()
{
    cudaError_t e = allow_max_dynamic_smem(draw_kernel);
    return e != cudaSuccess ? e : allow_max_dynamic_smem(hist_partial_kernel);
}

}  // namespace rift

// ======================================================================== reduction without allocation
//
// rift_ile_reduce_noalloc runs the same two reduction kernels as the library's own
// marginalisation, but its scratch (block partials, the running record and the
// error word) lives in the file-scope array below instead of in buffers from
// cudaMalloc.  Every GPU that loads the library holds this array until the
// process exits.  Host code must not hand the symbol itself to a kernel (on the
// host it names a stand-in, not device memory): its device address is taken once
// per device with cudaGetSymbolAddress, with that device current.

namespace {

constexpr int kNoallocPartials = 5 * rift::kRedBlocks;   // [kRedBlocks][5] block partials
constexpr int kNoallocPooled = kNoallocPartials;         // 8 doubles: running record
constexpr int kNoallocErr = kNoallocPooled + 8;          // error word (int in a double slot)
constexpr int kNoallocDoubles = kNoallocErr + 8;          // 1536 doubles = 12 KiB

static __device__ __align__(256) double g_reduce_scratch[kNoallocDoubles];

constexpr int kNoallocMaxDevices = 64;
std::mutex g_noalloc_mutex;
double *g_noalloc_ptr[kNoallocMaxDevices] = {};

// Device address of the scratch array on the current device (looked up once).
int noalloc_scratch(double **out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoallocMaxDevices) {
        cudaGetLastError();
        return RIFT_ECUDA;
    }
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_reduce_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return RIFT_ECUDA;
        }
        g_noalloc_ptr[dev] = static_cast<double *>(p);
    }
    *out = g_noalloc_ptr[dev];
    return RIFT_OK;
}

}  // namespace

extern "C" int rift_ile_reduce_noalloc(const double *lnw, const double *lnL, int64_t n, double *out, void *cuda_stream)
{
    if (!lnw || !out || n < 1 || n > RIFT_NOALLOC_MAX_SAMPLES)
        return RIFT_EINVAL;
    double *scratch = nullptr;
    int rc = noalloc_scratch(&scratch);
    if (rc != RIFT_OK)
        return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    int *err = reinterpret_cast<int *>(scratch + kNoallocErr);
    int flags = 0;
    if (cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess ||
        rift::launch_reduce(lnw, lnL ? lnL : lnw, n, scratch, out, 0, scratch + kNoallocPooled, 1, err, st) !=
            cudaSuccess ||
        cudaMemcpyAsync(&flags, err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        return RIFT_ECUDA;
    }
    return (flags & rift::kErrNonFinite) ? RIFT_ENONFINITE : RIFT_OK;
}
