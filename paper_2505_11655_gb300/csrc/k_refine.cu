// Float64 re-evaluation of the samples that carry weight (precision mode RIFT_MIXED).
//
// At high signal-to-noise ratio ln L ~ 1e4 is a difference of data and template
// terms of the same size, and float32 rounding of those terms alone is ~1e-3
// (arXiv:2505.11655 Sec. II A, Eq. (def:lnL:Decomposed)).  Only samples whose weight
// can matter are redone: ln w_i >= max ln w - margin.  For each of them (one warp):
//   1. coefficients c_k,lm, arrival delays and the template term in float64;
//   2. the data term of every bin in float32 (float32 Q planes and coefficients),
//      which locates the bins that can matter for the time marginal;
//   3. every bin whose float32 ln L lies within kRefineBins of the sample's float32
//      maximum is recomputed in float64 (float64 Q, float64 interpolation);
//   4. the time marginal is a float64 log-sum-exp over the mixed values.
// Bins left in float32 sit more than kRefineBins below the maximum, where their
// absolute error (<~1e-2) cannot move the marginal by more than e^-kRefineBins.
#include <cfloat>
#include <cmath>

#include "ile_kernels.h"

namespace rift {

constexpr int kRefThreads = 128;   // 4 warps, one sample each
constexpr double kRefineBins = 40.0;

// Selection of the samples with key[perm[i]] >= max - margin, in the order of perm (index
// order when null; the sky sort, which is stable, so the list, and everything computed from it, is the same from
// run to run): block b of the grid owns the contiguous range [b per, (b + 1) per) of perm;
// pass 1 counts per block, a single block scans the counts, pass 2 writes each block's
// matches at its offset in order.  In the sort's order neighbours of the list keep close
// arrival delays, so the tensor-core pass over the list needs few windows per tile (in
// index order its tiles span the sky: a three-member portfolio's 2 x 200k samples took 14.4
// ms, now 10.7; twelve uneven solves as one graph 61.8 ms, now 49.8).
constexpr int kSelThreads = 256;
constexpr int kSelMaxBlocks = kSelectWords - 1;

__global__ void __launch_bounds__(kSelThreads) select_count_kernel(const double *__restrict__ key,
                                                                    const uint32_t *__restrict__ perm, int64_t n,
                                                                    const double *__restrict__ stats, int slot,
                                                                    double margin, uint32_t *__restrict__ blk)
{
    const double cut = stats[8 * slot + 4] - margin;   // max ln w (or max ln L) of the batch
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = (int64_t)blockIdx.x * per, b1 = min(n, b0 + per);
    uint32_t c = 0;
    for (int64_t i = b0 + threadIdx.x; i < b1; i += kSelThreads)
        c += key[perm ? perm[i] : i] >= cut ? 1u : 0u;
    c = __reduce_add_sync(0xffffffffu, c);
    __shared__ uint32_t ws[kSelThreads / 32];
    if ((threadIdx.x & 31) == 0)
        ws[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < kSelThreads / 32; ++w)
            t += ws[w];
        blk[blockIdx.x] = t;
    }
}

// exclusive scan of the nb <= kSelMaxBlocks block counts in place; the total goes to *count
__global__ void __launch_bounds__(kSelMaxBlocks) select_scan_kernel(uint32_t *__restrict__ blk, int nb,
                                                                    uint32_t *__restrict__ count)
{
    __shared__ uint32_t ws[kSelMaxBlocks / 32];
    const int t = threadIdx.x, lane = t & 31;
    const uint32_t c = t < nb ? blk[t] : 0u;
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o)
            x += y;
    }
    if (lane == 31)
        ws[t >> 5] = x;
    __syncthreads();
    for (int v = 0; v < (t >> 5); ++v)
        x += ws[v];
    if (t < nb)
        blk[t] = x - c;
    if (t == (int)blockDim.x - 1)
        *count = x;
}

__global__ void __launch_bounds__(kSelThreads) select_write_kernel(const double *__restrict__ key,
                                                                    const uint32_t *__restrict__ perm, int64_t n,
                                                                    const double *__restrict__ stats, int slot,
                                                                    double margin, const uint32_t *__restrict__ blk,
                                                                    uint32_t *__restrict__ idx)
{
    const double cut = stats[8 * slot + 4] - margin;
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = (int64_t)blockIdx.x * per, b1 = min(n, b0 + per);
    __shared__ uint32_t ws[kSelThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t base = blk[blockIdx.x];
    for (int64_t c0 = b0; c0 < b1; c0 += kSelThreads) {
        const int64_t i = c0 + threadIdx.x;
        const uint32_t g = i < b1 ? (perm ? perm[i] : (uint32_t)i) : 0u;
        const bool take = i < b1 && key[g] >= cut;
        const unsigned mask = __ballot_sync(0xffffffffu, take);
        if (lane == 0)
            ws[warp] = (uint32_t)__popc(mask);
        __syncthreads();
        uint32_t before = 0, total = 0;
        for (int w = 0; w < kSelThreads / 32; ++w) {
            before += w < warp ? ws[w] : 0u;
            total += ws[w];
        }
        if (take)
            idx[base + before + (uint32_t)__popc(mask & ((1u << lane) - 1))] = g;
        base += total;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kRefThreads) refine_kernel(Problem P, const double *__restrict__ theta,
                                                              const uint32_t *__restrict__ idx,
                                                              const uint32_t *__restrict__ count,
                                                              double *__restrict__ lnL_tmarg, const double *__restrict__ lnpw,
                                                              double *__restrict__ lnw, int *err,
                                                              const double *__restrict__ v32, int64_t v32_rows)
{
    extern __shared__ double rsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int K = P.K, M = P.M, KM = K * M, NT = P.n_t;
    double2 *c64 = reinterpret_cast<double2 *>(rsm) + (size_t)warp * (KM + K + M);
    double2 *F64 = c64 + KM;
    double2 *Y64 = F64 + K;
    double *vals = rsm + (size_t)wpb * 2 * (KM + K + M) + (size_t)warp * NT;
    __shared__ double dts[kRefThreads / 32][kMaxDet];
    const uint32_t n_sel = *count;
    for (uint32_t w = blockIdx.x * wpb + warp; w < n_sel; w += gridDim.x * wpb) {
        const uint32_t s = idx[w];
        const double *th = theta + 6 * (size_t)s;
        Sky sky = sky_of(th[0], th[1], P.gmst);
        const double x = P.dist_marg ? 1.0 : P.d_ref / th[5];
        if (lane < K) {
            double s2p, c2p;
            sincos(2.0 * th[2], &s2p, &c2p);
            Cx<double> F = response<double>(P, lane, sky, c2p, s2p);
            F64[lane] = make_double2(x * F.re, x * F.im);
            dts[warp][lane] = arrival_delay(P, lane, sky);
        }
        for (int m = lane; m < M; m += 32) {
            double cpow[kMaxPow + 1], spow[kMaxPow + 1];
            half_angle_powers<double>(th[4], cpow, spow);
            Cx<double> Y = harmonic<double>(P, m, cpow, spow, th[3]);
            Y64[m] = make_double2(Y.re, Y.im);
        }
        __syncwarp();
        for (int q = lane; q < KM; q += 32) {
            const double2 F = F64[q / M], Y = Y64[q % M];
            c64[q] = make_double2(F.x * Y.x - F.y * Y.y, F.x * Y.y + F.y * Y.x);
        }
        __syncwarp();
        // template term in float64
        double part = 0.0;
        for (int q = lane; q < KM; q += 32) {
            const int k = q / M, a = q % M;
            const double2 *Ur = P.U64 + ((size_t)k * M + a) * M;
            const double2 *Vr = P.V64 + ((size_t)k * M + a) * M;
            double ur = 0, ui = 0, vr = 0, vi = 0;
#pragma unroll 7
            for (int b = 0; b < M; ++b) {
                const double2 cb = c64[k * M + b], u = Ur[b], v = Vr[b];
                ur += u.x * cb.x - u.y * cb.y;
                ui += u.x * cb.y + u.y * cb.x;
                vr += v.x * cb.x - v.y * cb.y;
                vi += v.x * cb.y + v.y * cb.x;
            }
            const double2 ca = c64[q];
            part += (ca.x * ur + ca.y * ui) + (ca.x * vr - ca.y * vi);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
            part += __shfl_xor_sync(0xffffffffu, part, o);
        const double quad = P.kappa * part;
        // float32 ln L at every bin: from the tiled kernel's second pass over the selected
        // samples when it ran for this one, else recomputed here
        float mx32 = -INFINITY;
        if ((int64_t)w < v32_rows) {
            const double *row = v32 + (size_t)w * NT;
            for (int j = lane; j < NT; j += 32) {
                const double v = row[j];
                vals[j] = v;
                mx32 = fmaxf(mx32, (float)v);
            }
        } else
        for (int j = lane; j < NT; j += 32) {
            const double tj = P.t_lo + j * P.t_step;
            float lin = 0.f;
            for (int k = 0; k < K; ++k) {
                const double u = (tj + dts[warp][k] - P.q_t0[k]) * P.fs;
                const double fl = floor(u);
                if (!(fl >= 0.0) || fl + 1.0 > (double)(P.n_q - 1)) {
                    atomicOr(err, kErrRange);
                    continue;
                }
                const int i = (int)fl;
                const float f = (float)(u - fl);
                const float *Qk = P.Qr32 + (size_t)k * 2 * M * P.n_q_pad + i;
                // the loads of several modes in flight at once (the Q planes live in L2)
#pragma unroll 7
                for (int m = 0; m < M; ++m) {
                    const double2 c = c64[k * M + m];
                    const float *qr = Qk + (size_t)(2 * m) * P.n_q_pad, *qi = qr + P.n_q_pad;
                    const float vr = fmaf(f, qr[1] - qr[0], qr[0]), vi = fmaf(f, qi[1] - qi[0], qi[0]);
                    lin = fmaf((float)c.x, vr, fmaf((float)c.y, vi, lin));
                }
            }
            const double v = P.dist_marg ? (double)ln_dist_marg32(P, lin, (float)quad) : (double)lin - quad;
            vals[j] = v;
            mx32 = fmaxf(mx32, (float)v);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
            mx32 = fmaxf(mx32, __shfl_xor_sync(0xffffffffu, mx32, o));
        __syncwarp();
        // float64 data term at the bins that can matter
        double mx = -INFINITY;
        for (int j = lane; j < NT; j += 32) {
            double v = vals[j];
            if (v >= (double)mx32 - kRefineBins) {
                const double tj = P.t_lo + j * P.t_step;
                double lin = 0.0;
                for (int k = 0; k < K; ++k) {
                    const double u = (tj + dts[warp][k] - P.q_t0[k]) * P.fs;
                    const double fl = floor(u);
                    if (!(fl >= 0.0) || fl + 1.0 > (double)(P.n_q - 1))
                        continue;
                    const int i = (int)fl;
                    const double f = u - fl;
                    const double2 *Qk = P.Q64 + (size_t)k * M * P.n_q + i;
#pragma unroll 7
                    for (int m = 0; m < M; ++m) {
                        const double2 q0 = Qk[(size_t)m * P.n_q], q1 = Qk[(size_t)m * P.n_q + 1];
                        const double2 c = c64[k * M + m];
                        lin += c.x * ((1.0 - f) * q0.x + f * q1.x) + c.y * ((1.0 - f) * q0.y + f * q1.y);
                    }
                }
                v = P.dist_marg ? ln_dist_marg64(P, lin, quad) : lin - quad;
                vals[j] = v;
            }
            mx = fmax(mx, v);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
            mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        double sum = 0.0;
        for (int j = lane; j < NT; j += 32)
            sum += exp(vals[j] - mx);
#pragma unroll
        for (int o = 16; o; o >>= 1)
            sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) {
            const double r = mx + log(sum) - log((double)NT);
            if (!isfinite(r))
                atomicOr(err, kErrNonFinite);
            lnL_tmarg[s] = r;
            if (lnw && lnpw)
                lnw[s] = r + lnpw[s];
        }
        __syncwarp();
    }
}

// The same re-evaluation (of the plain likelihood) with a block per sample, for short lists: bins
// over the block's threads, the near-peak ones compacted first, and every sum in refine_kernel's
// order, so that a sample's value is the same bits.  That is what it is for: the first iterations
// of a loud solve hang on a handful of samples, and what follows amplifies their last bits (the
// masses of two runs 2e-13 apart after one iteration are 1e-4 apart after three at n_eff 1 to 3),
// so they are taken in the plain float64 arithmetic.  It costs what the tensor-core kernel does on
// such lists, whose prologue and chunks take 107 us however short the list (3 detectors, 21 modes,
// 1001 bins: 110 us a list in the mean of a loud solve); a warp per sample took 250 us, as each
// sub-partition's float64 pipe then works for one warp at a time.
constexpr int kFewThreads = 512;

__global__ void __launch_bounds__(kFewThreads) refine_few_kernel(Problem P, const double *__restrict__ theta,
                                                                 const uint32_t *__restrict__ idx,
                                                                 const uint32_t *__restrict__ count, uint32_t most,
                                                                 double *__restrict__ lnL_tmarg,
                                                                 const double *__restrict__ lnpw,
                                                                 double *__restrict__ lnw, int *err)
{
    extern __shared__ double rsm[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = P.K, M = P.M, KM = K * M, NT = P.n_t;
    double2 *c64 = reinterpret_cast<double2 *>(rsm), *F64 = c64 + KM, *Y64 = F64 + K;
    double *dts = reinterpret_cast<double *>(Y64 + M), *tq = dts + K, *vals = tq + KM;
    int *list = reinterpret_cast<int *>(vals + NT);
    __shared__ double quad_s, mx_s[kFewThreads / 32];
    __shared__ float mx32_s[kFewThreads / 32];
    __shared__ int near_s;
    const uint32_t n_sel = *count;
    if (n_sel > most)
        return;
    for (uint32_t w = blockIdx.x; w < n_sel; w += gridDim.x) {
        const uint32_t s = idx[w];
        const double *th = theta + 6 * (size_t)s;
        if (warp == 0) {
            Sky sky = sky_of(th[0], th[1], P.gmst);
            const double x = P.d_ref / th[5];
            if (lane < K) {
                double s2p, c2p;
                sincos(2.0 * th[2], &s2p, &c2p);
                Cx<double> F = response<double>(P, lane, sky, c2p, s2p);
                F64[lane] = make_double2(x * F.re, x * F.im);
                dts[lane] = arrival_delay(P, lane, sky);
            }
        } else if (warp == 1) {
            for (int m = lane; m < M; m += 32) {
                double cpow[kMaxPow + 1], spow[kMaxPow + 1];
                half_angle_powers<double>(th[4], cpow, spow);
                Cx<double> Y = harmonic<double>(P, m, cpow, spow, th[3]);
                Y64[m] = make_double2(Y.re, Y.im);
            }
        }
        if (tid == 0)
            near_s = 0;
        __syncthreads();
        for (int q = tid; q < KM; q += kFewThreads) {
            const double2 F = F64[q / M], Y = Y64[q % M];
            c64[q] = make_double2(F.x * Y.x - F.y * Y.y, F.x * Y.y + F.y * Y.x);
        }
        __syncthreads();
        // template term, a row per thread (of the last warps, which have the fewest bins below)
        for (int q = (tid + kFewThreads / 8) % kFewThreads; q < KM; q += kFewThreads) {
            const int k = q / M, a = q % M;
            const double2 *Ur = P.U64 + ((size_t)k * M + a) * M;
            const double2 *Vr = P.V64 + ((size_t)k * M + a) * M;
            double ur = 0, ui = 0, vr = 0, vi = 0;
#pragma unroll 7
            for (int b = 0; b < M; ++b) {
                const double2 cb = c64[k * M + b], u = Ur[b], v = Vr[b];
                ur += u.x * cb.x - u.y * cb.y;
                ui += u.x * cb.y + u.y * cb.x;
                vr += v.x * cb.x - v.y * cb.y;
                vi += v.x * cb.y + v.y * cb.x;
            }
            const double2 ca = c64[q];
            tq[q] = (ca.x * ur + ca.y * ui) + (ca.x * vr - ca.y * vi);
        }
        // the data term of every bin in float32
        for (int j = tid; j < NT; j += kFewThreads) {
            const double tj = P.t_lo + j * P.t_step;
            float lin = 0.f;
            for (int k = 0; k < K; ++k) {
                const double u = (tj + dts[k] - P.q_t0[k]) * P.fs;
                const double fl = floor(u);
                if (!(fl >= 0.0) || fl + 1.0 > (double)(P.n_q - 1)) {
                    atomicOr(err, kErrRange);
                    continue;
                }
                const int i = (int)fl;
                const float f = (float)(u - fl);
                const float *Qk = P.Qr32 + (size_t)k * 2 * M * P.n_q_pad + i;
#pragma unroll 7
                for (int m = 0; m < M; ++m) {
                    const double2 c = c64[k * M + m];
                    const float *qr = Qk + (size_t)(2 * m) * P.n_q_pad, *qi = qr + P.n_q_pad;
                    const float vr = fmaf(f, qr[1] - qr[0], qr[0]), vi = fmaf(f, qi[1] - qi[0], qi[0]);
                    lin = fmaf((float)c.x, vr, fmaf((float)c.y, vi, lin));
                }
            }
            vals[j] = (double)lin;
        }
        __syncthreads();
        if (warp == 0) {
            double part = 0.0;
            for (int q = lane; q < KM; q += 32)
                part += tq[q];
#pragma unroll
            for (int o = 16; o; o >>= 1)
                part += __shfl_xor_sync(0xffffffffu, part, o);
            if (lane == 0)
                quad_s = P.kappa * part;
        }
        __syncthreads();
        const double quad = quad_s;
        float mx32 = -INFINITY;
        for (int j = tid; j < NT; j += kFewThreads) {
            const double v = vals[j] - quad;
            vals[j] = v;
            mx32 = fmaxf(mx32, (float)v);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
            mx32 = fmaxf(mx32, __shfl_xor_sync(0xffffffffu, mx32, o));
        if (lane == 0)
            mx32_s[warp] = mx32;
        __syncthreads();
        for (int v = 0; v < kFewThreads / 32; ++v)
            mx32 = fmaxf(mx32, mx32_s[v]);
        for (int j = tid; j < NT; j += kFewThreads)
            if (vals[j] >= (double)mx32 - kRefineBins)
                list[atomicAdd(&near_s, 1)] = j;
        __syncthreads();
        // float64 data term at the bins that can matter
        const int near = near_s;
        for (int e = tid; e < near; e += kFewThreads) {
            const int j = list[e];
            const double tj = P.t_lo + j * P.t_step;
            double lin = 0.0;
            for (int k = 0; k < K; ++k) {
                const double u = (tj + dts[k] - P.q_t0[k]) * P.fs;
                const double fl = floor(u);
                if (!(fl >= 0.0) || fl + 1.0 > (double)(P.n_q - 1))
                    continue;
                const int i = (int)fl;
                const double f = u - fl;
                const double2 *Qk = P.Q64 + (size_t)k * M * P.n_q + i;
#pragma unroll 7
                for (int m = 0; m < M; ++m) {
                    const double2 q0 = Qk[(size_t)m * P.n_q], q1 = Qk[(size_t)m * P.n_q + 1];
                    const double2 c = c64[k * M + m];
                    lin += c.x * ((1.0 - f) * q0.x + f * q1.x) + c.y * ((1.0 - f) * q0.y + f * q1.y);
                }
            }
            vals[j] = lin - quad;
        }
        __syncthreads();
        double mx = -INFINITY;
        for (int j = tid; j < NT; j += kFewThreads)
            mx = fmax(mx, vals[j]);
#pragma unroll
        for (int o = 16; o; o >>= 1)
            mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0)
            mx_s[warp] = mx;
        __syncthreads();
        for (int v = 0; v < kFewThreads / 32; ++v)
            mx = fmax(mx, mx_s[v]);
        for (int j = tid; j < NT; j += kFewThreads) {
            const double d = vals[j] - mx;
            vals[j] = d < -750.0 ? 0.0 : exp(d);   // (exp gives 0 there)
        }
        __syncthreads();
        if (warp == 0) {
            double sum = 0.0;
            for (int j = lane; j < NT; j += 32)
                sum += vals[j];
#pragma unroll
            for (int o = 16; o; o >>= 1)
                sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == 0) {
                const double r = mx + log(sum) - log((double)NT);
                if (!isfinite(r))
                    atomicOr(err, kErrNonFinite);
                lnL_tmarg[s] = r;
                if (lnw && lnpw)
                    lnw[s] = r + lnpw[s];
            }
        }
        __syncthreads();
    }
}

static size_t few_smem(const Problem &P)
{
    return sizeof(double) * (3 * (size_t)P.K * P.M + 3 * P.K + 2 * P.M + P.n_t) + sizeof(int) * (size_t)P.n_t;
}

cudaError_t launch_refine_few(const Problem &P, const double *theta, const uint32_t *idx, const uint32_t *count,
                              uint32_t most, double *lnL_tmarg, const double *lnpw, double *lnw, int *err,
                              cudaStream_t st)
{
    const size_t smem = few_smem(P);
    if (smem > 40 * 1024) {
        cudaError_t e = allow_max_dynamic_smem(refine_few_kernel);
        if (e != cudaSuccess)
            return e;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = (int)most < 2 * sms ? (int)most : 2 * sms;
    refine_few_kernel<<<grid, kFewThreads, smem, st>>>(P, theta, idx, count, most, lnL_tmarg, lnpw, lnw, err);
    return cudaGetLastError();
}

cudaError_t launch_select(const double *key, const uint32_t *perm, int64_t n, const double *stats, int slot,
                          double margin, uint32_t *idx, uint32_t *count, cudaStream_t st)
{
    if (n <= 0)
        return cudaSuccess;
    // block counts live after the count word
    uint32_t *blk = count + 1;
    const int64_t want = (n + 4 * kSelThreads - 1) / (4 * kSelThreads);
    const int grid = (int)(want < kSelMaxBlocks ? (want > 0 ? want : 1) : kSelMaxBlocks);
    select_count_kernel<<<grid, kSelThreads, 0, st>>>(key, perm, n, stats, slot, margin, blk);
    select_scan_kernel<<<1, (grid + 31) / 32 * 32, 0, st>>>(blk, grid, count);
    select_write_kernel<<<grid, kSelThreads, 0, st>>>(key, perm, n, stats, slot, margin, blk, idx);
    return cudaGetLastError();
}

cudaError_t launch_refine(const Problem &P, const double *theta, const uint32_t *idx, const uint32_t *count,
                          int64_t max_count, double *lnL_tmarg, const double *lnpw, double *lnw, int *err,
                          cudaStream_t st, const double *v32, int64_t v32_rows)
{
    if (max_count <= 0)
        return cudaSuccess;
    const int wpb = kRefThreads / 32;
    const size_t smem = sizeof(double) * ((size_t)wpb * 2 * (P.K * P.M + P.K + P.M) + (size_t)wpb * P.n_t);
    if (smem > 48 * 1024) {
        cudaError_t e = allow_max_dynamic_smem(refine_kernel);
        if (e != cudaSuccess)
            return e;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t want = (max_count + wpb - 1) / wpb;
    const int grid = (int)(want < (int64_t)sms * 8 ? want : (int64_t)sms * 8);
    refine_kernel<<<grid, kRefThreads, smem, st>>>(P, theta, idx, count, lnL_tmarg, lnpw, lnw, err, v32,
                                                   v32 ? v32_rows : 0);
    return cudaGetLastError();
}

cudaError_t prepare_refine_kernels()
{
    cudaError_t e = allow_max_dynamic_smem(refine_kernel);
    return e != cudaSuccess ? e : allow_max_dynamic_smem(refine_few_kernel);
}

}  // namespace rift
