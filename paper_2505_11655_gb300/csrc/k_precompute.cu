// Overlaps Q, U, V from frequency-domain inputs (arXiv:2505.11655, Sec. II A, Eq. QUV):
// on a mirror-symmetric two-sided grid f_j with inverse-PSD weights w_k(f), shared mode
// waveforms h_lm(f) and per-detector data d_k(f),
//   Q_k,lm(t_s)   = 2 sum_j w_k(f_j) exp(2 pi i f_j t_s) conj(h_lm(f_j)) d_k(f_j),
//                   t_s = q_t0_k + s / f_s on each detector's Q grid;
//   U_k,lm,l'm'   = 2 sum_j w_k conj(h_lm) h_l'm',   V_k,lm,l'm' = 2 sum_j w_k h_lm(-f_j) h_l'm'(f_j).
// U is Hermitian and V symmetric (the weights are symmetric in f), so only pairs
// lm <= l'm' are summed and mirrored (the halving the paper describes for U and V).
// All in float64.
//
// Q by a fast Fourier transform.  When the frequencies lie on a lattice f_j = f_0 + n_j df
// (integers n_j spanning fewer than L = f_s / df points, L a power of two), then with
// t_s = q_t0 + s / f_s,
//   exp(2 pi i f_j t_s) = exp(2 pi i f_j q_t0) exp(2 pi i f_0 s / f_s) exp(2 pi i n_j s / L),
// so Q_k,lm(t_s) = exp(2 pi i f_0 s / f_s) Y[s mod L], Y the length-L transform (sign +)
// of X[n_j] = A_j exp(2 pi i f_j q_t0): O(L log L) per (detector, mode) instead of
// O(n_q F).  Only the outputs s < n_q are needed: with P the power of two >= n_q (at most L)
// and R = L / P,
//   Y[s] = sum_r exp(2 pi i r s / L) Z_r[s mod P],  Z_r the length-P transform of X[R m + r],
// so one block per (detector, mode, r) runs a radix-4 Stockham (self-sorting) FFT in shared
// memory, reading h and the data products directly, and a second kernel sums the R terms of
// each output.  The float64 pipe bounds both (a 4 s segment at 4096 Hz, 3 detectors, 21 modes:
// ~50e6 operations of two a clock and SM).  Longer outputs or larger R take a radix-2 transform,
// one kernel per stage over every sequence at once; grids off a lattice (or with L not a power
// of two) the direct sum.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "ile_kernels.h"

namespace rift {

constexpr int kPcThreads = 128;   // Q samples per block
constexpr int kPcChunk = 64;      // frequencies staged per pass

// A[k][m][j] = 2 w_k(f_j) conj(h_m(f_j)) d_k(f_j)
__global__ void qfreq_kernel(const double2 *__restrict__ h, const double2 *__restrict__ d,
                             const double *__restrict__ w, int K, int M, int F, double2 *__restrict__ A)
{
    const int64_t total = (int64_t)K * M * F;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(e % F), m = (int)((e / F) % M), k = (int)(e / ((int64_t)F * M));
        const double2 hm = h[(size_t)m * F + j], dk = d[(size_t)k * F + j];
        const double s = 2.0 * w[(size_t)k * F + j];
        // conj(h) d
        A[e] = make_double2(s * (hm.x * dk.x + hm.y * dk.y), s * (hm.x * dk.y - hm.y * dk.x));
    }
}

// One thread per (detector, Q sample); all modes accumulated together.
__global__ void __launch_bounds__(kPcThreads) q_series_kernel(const double2 *__restrict__ A,
                                                              const double *__restrict__ f, int K, int M, int F,
                                                              const double *__restrict__ q_t0, double fs, int n_q,
                                                              double2 *__restrict__ Q)
{
    __shared__ double2 sA[kMaxModes * kPcChunk];
    __shared__ double sf[kPcChunk];
    const int k = blockIdx.y;
    const int s = blockIdx.x * kPcThreads + threadIdx.x;
    const double t = q_t0[k] + (double)s / fs;
    double re[kMaxModes], im[kMaxModes];
#pragma unroll
    for (int m = 0; m < kMaxModes; ++m)
        re[m] = im[m] = 0.0;
    for (int j0 = 0; j0 < F; j0 += kPcChunk) {
        const int nj = min(kPcChunk, F - j0);
        __syncthreads();
        for (int e = threadIdx.x; e < M * kPcChunk; e += kPcThreads) {
            const int m = e / kPcChunk, j = e % kPcChunk;
            sA[e] = j < nj ? A[((size_t)k * M + m) * F + j0 + j] : make_double2(0.0, 0.0);
        }
        for (int j = threadIdx.x; j < kPcChunk; j += kPcThreads)
            sf[j] = j < nj ? f[j0 + j] : 0.0;
        __syncthreads();
        for (int j = 0; j < nj; ++j) {
            double sn, cs;
            sincospi(2.0 * sf[j] * t, &sn, &cs);
#pragma unroll
            for (int m = 0; m < kMaxModes; ++m) {
                if (m < M) {
                    const double2 a = sA[m * kPcChunk + j];
                    re[m] += a.x * cs - a.y * sn;
                    im[m] += a.x * sn + a.y * cs;
                }
            }
        }
    }
    if (s < n_q) {
#pragma unroll
        for (int m = 0; m < kMaxModes; ++m)
            if (m < M)
                Q[((size_t)k * M + m) * n_q + s] = make_double2(re[m], im[m]);
    }
}

// U and V of every pair a <= b, mirrored.  Eight float64 multiply-adds a pair and frequency: the
// float64 pipe (two a clock and SM) bounds it, so the frequencies are split over two blocks per
// SM, a block stages tiles of 32 frequencies of h(f), h(-f) and 2 w h(f) in shared memory, and a
// thread owns one pair (several when there are more pairs than threads; a share of the tile's
// frequencies when there are few).  Partial sums of the blocks are added in their order.  One
// warp per pair with all loads from L2, a few warps per SM, took 461 us for 3 detectors, 21 modes
// and 16384 frequencies.
constexpr int kUvThreads = 256;
constexpr int kUvTile = 32;
constexpr int kUvPer = (kMaxModes * (kMaxModes + 1) / 2 + kUvThreads - 1) / kUvThreads;   // pairs per thread

__device__ __forceinline__ void uv_pair(int p, int M, int &a, int &b)
{
    a = 0;
    while (p >= M - a) {   // pair index -> (a, b), a <= b
        p -= M - a;
        ++a;
    }
    b = a + p;
}

__global__ void __launch_bounds__(kUvThreads) uv_partial_kernel(const double2 *__restrict__ h,
                                                                const double *__restrict__ w, int M, int F,
                                                                double *__restrict__ part)
{
    extern __shared__ double2 uvs[];
    double2 *hp = uvs, *hm = hp + kUvTile * M, *hw = hm + kUvTile * M;   // [kUvTile][M]
    const int k = blockIdx.y, pairs = M * (M + 1) / 2;
    const int groups = pairs < kUvThreads ? kUvThreads / pairs : 1;      // threads per pair
    const int g = pairs < kUvThreads ? threadIdx.x / pairs : 0;
    const int p0 = pairs < kUvThreads ? threadIdx.x - g * pairs : threadIdx.x;
    const int per = (F + gridDim.x - 1) / gridDim.x;
    const int j0 = blockIdx.x * per, j1 = min(F, j0 + per);
    double acc[kUvPer][4];
    int pa[kUvPer], pb[kUvPer];
#pragma unroll
    for (int q = 0; q < kUvPer; ++q) {
        acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0.0;
        const int p = p0 + q * kUvThreads;
        pa[q] = pb[q] = 0;
        if (p < pairs && g < groups)
            uv_pair(p, M, pa[q], pb[q]);
    }
    for (int t0 = j0; t0 < j1; t0 += kUvTile) {
        const int nj = min(kUvTile, j1 - t0);
        __syncthreads();
        for (int e = threadIdx.x; e < M * kUvTile; e += kUvThreads) {
            const int m = e / kUvTile, j = e % kUvTile;
            if (j < nj) {
                const double2 v = h[(size_t)m * F + t0 + j];
                const double s = 2.0 * w[(size_t)k * F + t0 + j];
                hp[j * M + m] = v;
                hw[j * M + m] = make_double2(s * v.x, s * v.y);
                hm[j * M + m] = h[(size_t)m * F + (F - 1 - t0 - j)];   // h(-f)
            }
        }
        __syncthreads();
        if (g < groups)
            for (int j = g; j < nj; j += groups)
#pragma unroll
                for (int q = 0; q < kUvPer; ++q)
                    if (p0 + q * kUvThreads < pairs) {
                        const double2 a = hp[j * M + pa[q]], c = hm[j * M + pa[q]], b = hw[j * M + pb[q]];
                        acc[q][0] = fma(a.x, b.x, fma(a.y, b.y, acc[q][0]));
                        acc[q][1] = fma(a.x, b.y, fma(-a.y, b.x, acc[q][1]));
                        acc[q][2] = fma(c.x, b.x, fma(-c.y, b.y, acc[q][2]));
                        acc[q][3] = fma(c.x, b.y, fma(c.y, b.x, acc[q][3]));
                    }
    }
    double *out = part + (size_t)(k * gridDim.x + blockIdx.x) * 4 * pairs;   // [4][pairs]
    if (groups == 1) {
#pragma unroll
        for (int q = 0; q < kUvPer; ++q)
            if (g == 0 && p0 + q * kUvThreads < pairs)
                for (int c = 0; c < 4; ++c)
                    out[c * pairs + p0 + q * kUvThreads] = acc[q][c];
        return;
    }
    // the threads of a pair in order
    __shared__ double red[4][kUvThreads];
    for (int c = 0; c < 4; ++c)
        red[c][threadIdx.x] = acc[0][c];
    __syncthreads();
    for (int e = threadIdx.x; e < 4 * pairs; e += kUvThreads) {
        const int c = e / pairs, p = e - c * pairs;
        double v = 0.0;
        for (int u = 0; u < groups; ++u)
            v += red[c][u * pairs + p];
        out[e] = v;
    }
}

// One warp per (detector, pair): the blocks' sums in a fixed order.
__global__ void uv_final_kernel(const double *__restrict__ part, int nch, int K, int M, double2 *__restrict__ U,
                                double2 *__restrict__ V)
{
    const int lane = threadIdx.x & 31, pairs = M * (M + 1) / 2;
    const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (e >= K * pairs)
        return;
    const int k = e / pairs, p = e - k * pairs;
    int a, b;
    uv_pair(p, M, a, b);
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    const double *q = part + (size_t)k * nch * 4 * pairs + p;
    for (int c = lane; c < nch; c += 32)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            v[i] += q[(size_t)(4 * c + i) * pairs];
#pragma unroll
    for (int o = 16; o; o >>= 1)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    if (lane)
        return;
    if (a == b)
        v[1] = 0.0;   // w |h|^2 is real (the fused products leave a rounding residual)
    const size_t ab = ((size_t)k * M + a) * M + b, ba = ((size_t)k * M + b) * M + a;
    U[ab] = make_double2(v[0], v[1]);
    U[ba] = make_double2(v[0], -v[1]);
    V[ab] = make_double2(v[2], v[3]);
    V[ba] = make_double2(v[2], v[3]);
}

// ---------------------------------------------------------------- FFT path for Q

// T[e] = exp(2 pi i e / L), e < L / 2
__global__ void fft_twiddle_kernel(int L, double2 *__restrict__ T)
{
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < L / 2; e += gridDim.x * blockDim.x) {
        double sn, cs;
        sincospi(2.0 * (double)e / (double)L, &sn, &cs);
        T[e] = make_double2(cs, sn);
    }
}

// X [K M][L] (zeroed): X[km][n_j] = A[km][j] exp(2 pi i f_j q_t0_k)
__global__ void fft_scatter_kernel(const double2 *__restrict__ A, const double *__restrict__ f,
                                   const int *__restrict__ nidx, int K, int M, int F, const double *__restrict__ q_t0,
                                   int L, double2 *__restrict__ X)
{
    const int64_t total = (int64_t)K * M * F;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(e % F);
        const int64_t km = e / F;
        const int k = (int)(km / M);
        double sn, cs;
        sincospi(2.0 * f[j] * q_t0[k], &sn, &cs);
        const double2 a = A[e];
        X[km * L + nidx[j]] = make_double2(a.x * cs - a.y * sn, a.x * sn + a.y * cs);
    }
}

// One radix-2 Stockham stage (sub-transforms of length Ns combined into 2 Ns) of every
// sequence: butterfly j < L/2 of a sequence reads j and j + L/2 and writes
// (j / Ns) 2 Ns + j % Ns and that plus Ns, with twiddle exp(2 pi i (j % Ns) / (2 Ns)).
__global__ void fft_stage_kernel(const double2 *__restrict__ in, double2 *__restrict__ out, int L, int Ns,
                                 const double2 *__restrict__ T, int64_t n_seq)
{
    const int half = L >> 1;
    const int64_t total = n_seq * half;
    const int tstride = half / Ns;   // T index step: (j % Ns) L / (2 Ns)
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = e / half;
        const int j = (int)(e - q * half);
        const int kk = j & (Ns - 1);
        const double2 w = T[(size_t)kk * tstride];
        const double2 a = in[q * L + j], b0 = in[q * L + j + half];
        const double2 b = make_double2(b0.x * w.x - b0.y * w.y, b0.x * w.y + b0.y * w.x);
        const int64_t o = q * L + (int64_t)(j / Ns) * 2 * Ns + kk;
        out[o] = make_double2(a.x + b.x, a.y + b.y);
        out[o + Ns] = make_double2(a.x - b.x, a.y - b.y);
    }
}

// Q[km][s] = exp(2 pi i f_0 s / f_s) Y[km][s mod L]
__global__ void fft_extract_kernel(const double2 *__restrict__ Y, int64_t n_seq, int L, double f0, double fs, int n_q,
                                   double2 *__restrict__ Q)
{
    const int64_t total = n_seq * n_q;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t km = e / n_q;
        const int s = (int)(e - km * n_q);
        double sn, cs;
        sincospi(2.0 * f0 * ((double)s / fs), &sn, &cs);
        const double2 y = Y[km * L + (s & (L - 1))];
        Q[e] = make_double2(y.x * cs - y.y * sn, y.x * sn + y.y * cs);
    }
}

// ---------------------------------------------------------------- pruned transform

constexpr int kFftMaxP = 8192;      // 128 KB of shared memory
constexpr int kFftMaxR = 64;
constexpr int kFftMaxThreads = 512;
constexpr int kFftItems = kFftMaxP / 4 / kFftMaxThreads;   // radix-4 butterflies per thread

bool fft_pruned(int L, int n_q, int *P, int *R)
{
    int p = 2;
    while (p < n_q && p < L)
        p <<= 1;
    if (P) {
        *P = p;
        *R = L / p;
    }
    return p <= kFftMaxP && L / p <= kFftMaxR;
}

// D[k][j] = 2 w_k(f_j) d_k(f_j) exp(2 pi i f_j q_t0_k), and jidx[n_j] = j (-1 elsewhere)
__global__ void fft_data_kernel(const double2 *__restrict__ d, const double *__restrict__ w,
                                const double *__restrict__ f, const int *__restrict__ nidx, int K, int F,
                                const double *__restrict__ q_t0, double2 *__restrict__ D, int *__restrict__ jidx)
{
    const int64_t total = (int64_t)K * F;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(e / F), j = (int)(e - (int64_t)k * F);
        double sn, cs;
        sincospi(2.0 * f[j] * q_t0[k], &sn, &cs);
        const double s = 2.0 * w[e];
        const double2 v = d[e];
        D[e] = make_double2(s * (v.x * cs - v.y * sn), s * (v.x * sn + v.y * cs));
        if (k == 0)
            jidx[nidx[j]] = j;
    }
}

// Z[km][r][.] = length-P transform (sign +) of X[R m + r] = conj(h_m(f_j)) D_k(f_j), j = jidx[R m + r]
__global__ void __launch_bounds__(kFftMaxThreads) fft_block_kernel(const double2 *__restrict__ h,
                                                                   const double2 *__restrict__ D,
                                                                   const int *__restrict__ jidx, int M, int F, int P,
                                                                   int R, const double2 *__restrict__ T,
                                                                   double2 *__restrict__ Z)
{
    extern __shared__ double2 fx[];
    const int r = blockIdx.x, km = blockIdx.y, k = km / M, m = km - k * M;
    const int half = (P * R) >> 1;   // entries of T
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const int j = jidx[R * i + r];
        double2 x = make_double2(0.0, 0.0);
        if (j >= 0) {
            const double2 a = h[(size_t)m * F + j], b = D[(size_t)k * F + j];
            x = make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
        }
        fx[i] = x;
    }
    // exp(2 pi i e / (P R)), e < P R
    auto tw = [&](int e) {
        const double2 t = T[e < half ? e : e - half];
        return e < half ? t : make_double2(-t.x, -t.y);
    };
    auto mul = [](double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); };
    int Ns = 1;
    double2 v[kFftItems][4];
    if ((__ffs(P) - 1) & 1) {   // an odd number of factors 2: one radix-2 stage (no twiddles) first
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2 * kFftItems; ++q) {
            const int j = threadIdx.x + q * blockDim.x;
            if (j < P / 2) {
                v[q >> 1][2 * (q & 1)] = fx[j];
                v[q >> 1][2 * (q & 1) + 1] = fx[j + P / 2];
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2 * kFftItems; ++q) {
            const int j = threadIdx.x + q * blockDim.x;
            if (j < P / 2) {
                const double2 a = v[q >> 1][2 * (q & 1)], b = v[q >> 1][2 * (q & 1) + 1];
                fx[2 * j] = make_double2(a.x + b.x, a.y + b.y);
                fx[2 * j + 1] = make_double2(a.x - b.x, a.y - b.y);
            }
        }
        Ns = 2;
    }
    const int quarter = P >> 2;
    for (; Ns < P; Ns <<= 2) {
        const int step = quarter / Ns * R;   // T index of one unit of kk
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kFftItems; ++q) {
            const int j = threadIdx.x + q * blockDim.x;
            if (j < quarter) {
                const int kk = j & (Ns - 1);
                v[q][0] = fx[j];
                v[q][1] = fx[j + quarter];
                v[q][2] = fx[j + 2 * quarter];
                v[q][3] = fx[j + 3 * quarter];
                if (Ns > 1) {
                    v[q][1] = mul(v[q][1], tw(kk * step));
                    v[q][2] = mul(v[q][2], tw(2 * kk * step));
                    v[q][3] = mul(v[q][3], tw(3 * kk * step));
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kFftItems; ++q) {
            const int j = threadIdx.x + q * blockDim.x;
            if (j < quarter) {
                const int o = (j & ~(Ns - 1)) * 4 + (j & (Ns - 1));
                const double2 s02 = make_double2(v[q][0].x + v[q][2].x, v[q][0].y + v[q][2].y);
                const double2 d02 = make_double2(v[q][0].x - v[q][2].x, v[q][0].y - v[q][2].y);
                const double2 s13 = make_double2(v[q][1].x + v[q][3].x, v[q][1].y + v[q][3].y);
                const double2 d13 = make_double2(v[q][1].x - v[q][3].x, v[q][1].y - v[q][3].y);
                fx[o] = make_double2(s02.x + s13.x, s02.y + s13.y);
                fx[o + Ns] = make_double2(d02.x - d13.y, d02.y + d13.x);       // + i d13
                fx[o + 2 * Ns] = make_double2(s02.x - s13.x, s02.y - s13.y);
                fx[o + 3 * Ns] = make_double2(d02.x + d13.y, d02.y - d13.x);   // - i d13
            }
        }
    }
    __syncthreads();
    double2 *out = Z + ((size_t)km * R + r) * P;
    for (int i = threadIdx.x; i < P; i += blockDim.x)
        out[i] = fx[i];
}

// Q[km][s] = exp(2 pi i f_0 s / f_s) sum_r exp(2 pi i r s / L) Z[km][r][s mod P]
__global__ void fft_combine_kernel(const double2 *__restrict__ Z, int KM, int P, int R, const double2 *__restrict__ T,
                                   double f0, double fs, int n_q, double2 *__restrict__ Q)
{
    const int L = P * R, half = L >> 1;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n_q; s += gridDim.x * blockDim.x) {
        const int km = blockIdx.y, sl = s & (L - 1);
        const double2 *z = Z + (size_t)km * R * P + (sl & (P - 1));
        double re = z[0].x, im = z[0].y;
#pragma unroll 4
        for (int r = 1; r < R; ++r) {
            const int e = (int)(((int64_t)r * sl) & (L - 1));
            double2 t = T[e < half ? e : e - half];
            if (e >= half)
                t = make_double2(-t.x, -t.y);
            const double2 v = z[(size_t)r * P];
            re += v.x * t.x - v.y * t.y;
            im += v.x * t.y + v.y * t.x;
        }
        double sn, cs;
        sincospi(2.0 * f0 * ((double)s / fs), &sn, &cs);
        Q[(size_t)km * n_q + s] = make_double2(re * cs - im * sn, re * sn + im * cs);
    }
}

// ---------------------------------------------------------------- input checks

// Weights finite, non-negative and symmetric in f, frequencies finite and mirror-symmetric:
// the first violation in the order of a loop over j, then the frequency, then the detectors, as
// 4 (j (K + 1) + [0 frequency, 1 + k weights]) + code; and the smallest step and largest modulus of
// the frequencies (non-negative doubles order like their bits).
__global__ void waveform_check_kernel(const double *__restrict__ f, const double *__restrict__ w, int K, int F,
                                      WaveformInfo *__restrict__ info)
{
    unsigned long long bad = ~0ull, gap = ~0ull, fm = 0ull;
    const int64_t total = (int64_t)(K + 1) * F;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(e / F), j = (int)(e - (int64_t)c * F);
        const double *row = c == 0 ? f : w + (size_t)(c - 1) * F;
        const double a = row[j], b = row[F - 1 - j];
        int code = 0;
        if (c == 0) {
            code = !isfinite(a) || b != -a ? kWaveformInvalid : 0;
            fm = max(fm, (unsigned long long)__double_as_longlong(fabs(a)));
            if (j > 0) {
                const double g = a - row[j - 1];
                gap = min(gap, g > 0.0 ? (unsigned long long)__double_as_longlong(g) : 0ull);
            }
        } else
            code = !isfinite(a) ? kWaveformNonFinite : a < 0.0 || a != b ? kWaveformInvalid : 0;
        if (code)
            bad = min(bad, 4ull * ((unsigned long long)j * (K + 1) + c) + code);
    }
    if (bad != ~0ull)
        atomicMin(&info->bad, bad);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        gap = min(gap, __shfl_xor_sync(0xffffffffu, gap, o));
        fm = max(fm, __shfl_xor_sync(0xffffffffu, fm, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (gap != ~0ull)
            atomicMin(&info->gap, gap);
        if (fm)
            atomicMax(&info->fmax, fm);
    }
}

int waveform_lattice(double fs, unsigned long long gap)
{
    double df;
    memcpy(&df, &gap, 8);
    if (!(df > 0.0) || !(fs / df < 1e9))
        return 0;
    const double Lr = fs / df;
    const long long L = std::llround(Lr);
    return L >= 2 && L <= (1ll << 26) && (L & (L - 1)) == 0 && std::fabs(Lr - (double)L) <= 1e-9 * (double)L ? (int)L : 0;
}

// The lattice f_j = f_0 + n_j df (df the smallest step; ascending frequencies, integers n_j to
// 1e-9 relative, below L = f_s / df): n_j to nidx, info->off set when a frequency lies off it.
__global__ void waveform_lattice_kernel(const double *__restrict__ f, int F, double fs, int *__restrict__ nidx,
                                        WaveformInfo *__restrict__ info)
{
    const double df = __longlong_as_double((long long)info->gap), fmax = __longlong_as_double((long long)info->fmax);
    const double f0 = f[0];
    bool off = !(df > 0.0) || !(fs / df < 1e9);
    const long long L = off ? 0 : llround(fs / df);
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < F; j += gridDim.x * blockDim.x) {
        const long long n = off ? -1 : llround((f[j] - f0) / df);
        if (n < 0 || n >= L || fabs(f[j] - f0 - (double)n * df) > 1e-9 * (fmax > 1.0 ? fmax : 1.0))
            off = true;
        else
            nidx[j] = (int)n;
    }
    if (off)
        info->off = 1;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        info->f0 = f0;
}

cudaError_t launch_waveform_check(const double *f, const double *w, int K, int F, double fs, int *nidx,
                                  WaveformInfo *info, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(info, 0, sizeof(WaveformInfo), st);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(&info->bad, 0xff, 2 * sizeof(info->bad), st);   // bad and gap
    if (e != cudaSuccess)
        return e;
    const int64_t total = (int64_t)(K + 1) * F;
    waveform_check_kernel<<<(int)std::min<int64_t>((total + 255) / 256, 152 * 8), 256, 0, st>>>(f, w, K, F, info);
    waveform_lattice_kernel<<<std::min((F + 255) / 256, 152 * 8), 256, 0, st>>>(f, F, fs, nidx, info);
    return cudaGetLastError();
}

static int uv_chunks(int K, int F) { return std::max(1, std::min((F + kUvTile - 1) / kUvTile, 2 * 152 / K)); }

size_t uv_scratch_doubles(int K, int M, int F) { return (size_t)K * uv_chunks(K, F) * 4 * (M * (M + 1) / 2); }

cudaError_t launch_precompute(const double2 *h, const double2 *d, const double *w, const double *f, int K, int M,
                              int F, const double *q_t0_dev, double fs, int n_q, double2 *A_scratch, double *uv_scratch,
                              double2 *Q, double2 *U, double2 *V, cudaStream_t st, const FftPlan *fft, int *launched)
{
    const int64_t nA = (int64_t)K * M * F, nseq = (int64_t)K * M;
    int k = 0, P = 0, R = 0;
    cudaError_t e = cudaSuccess;
    if (fft)
        fft_twiddle_kernel<<<std::max(1, std::min(fft->L / 2 / 256, 152 * 8)), 256, 0, st>>>(fft->L, fft->T);
    if (fft && fft_pruned(fft->L, n_q, &P, &R)) {
        if ((e = cudaMemsetAsync(fft->jidx, 0xff, sizeof(int) * (size_t)fft->L, st)) != cudaSuccess)
            return e;
        const int64_t nd = (int64_t)K * F;
        fft_data_kernel<<<(int)std::min<int64_t>((nd + 255) / 256, 152 * 8), 256, 0, st>>>(d, w, f, fft->nidx, K, F,
                                                                                          q_t0_dev, A_scratch, fft->jidx);
        const size_t smem = sizeof(double2) * (size_t)P;
        if (smem > 48 * 1024 && (e = allow_max_dynamic_smem(fft_block_kernel)) != cudaSuccess)
            return e;
        // butterflies of a stage spread over up to 512 threads
        const int threads = std::min(kFftMaxThreads, std::max(32, P / 4));
        fft_block_kernel<<<dim3(R, (unsigned)nseq), threads, smem, st>>>(h, A_scratch, fft->jidx, M, F, P, R, fft->T,
                                                                        fft->X);
        fft_combine_kernel<<<dim3((n_q + 127) / 128, (unsigned)nseq), 128, 0, st>>>(fft->X, (int)nseq, P, R, fft->T,
                                                                                    fft->f0, fs, n_q, Q);
        k += 4;
    } else if (fft) {
        const int L = fft->L;
        qfreq_kernel<<<(int)std::min<int64_t>((nA + 255) / 256, 152 * 8), 256, 0, st>>>(h, d, w, K, M, F, A_scratch);
        if ((e = cudaMemsetAsync(fft->X, 0, sizeof(double2) * (size_t)nseq * L, st)) != cudaSuccess)
            return e;
        fft_scatter_kernel<<<(int)std::min<int64_t>((nA + 255) / 256, 152 * 8), 256, 0, st>>>(
            A_scratch, f, fft->nidx, K, M, F, q_t0_dev, L, fft->X);
        double2 *a = fft->X, *b = fft->Y;
        const int64_t nb = nseq * (L / 2);
        for (int Ns = 1; Ns < L; Ns <<= 1) {
            fft_stage_kernel<<<(int)std::min<int64_t>((nb + 255) / 256, 152 * 16), 256, 0, st>>>(a, b, L, Ns, fft->T,
                                                                                                 nseq);
            std::swap(a, b);
            ++k;
        }
        const int64_t nqt = nseq * n_q;
        fft_extract_kernel<<<(int)std::min<int64_t>((nqt + 255) / 256, 152 * 8), 256, 0, st>>>(a, nseq, L, fft->f0,
                                                                                              fs, n_q, Q);
        k += 4;
    } else {
        qfreq_kernel<<<(int)std::min<int64_t>((nA + 255) / 256, 152 * 8), 256, 0, st>>>(h, d, w, K, M, F, A_scratch);
        dim3 grid((n_q + kPcThreads - 1) / kPcThreads, K);
        q_series_kernel<<<grid, kPcThreads, 0, st>>>(A_scratch, f, K, M, F, q_t0_dev, fs, n_q, Q);
        k += 2;
    }
    const int nch = uv_chunks(K, F), pairs = M * (M + 1) / 2;
    const size_t uv_smem = sizeof(double2) * 3 * kUvTile * M;
    if (uv_smem > 40 * 1024 && (e = allow_max_dynamic_smem(uv_partial_kernel)) != cudaSuccess)
        return e;   // (beside the static array of the pairs' threads)
    uv_partial_kernel<<<dim3(nch, K), kUvThreads, uv_smem, st>>>(h, w, M, F, uv_scratch);
    uv_final_kernel<<<(K * pairs + 7) / 8, 256, 0, st>>>(uv_scratch, nch, K, M, U, V);
    if (launched)
        *launched = k + 2;
    return cudaGetLastError();
}

}  // namespace rift
