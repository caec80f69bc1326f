// Host core of the ILE library: configuration checks, device buffers, the order of
// kernel launches for each entry point of include/rift_ile.h, and result assembly.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <array>
#include <mutex>
#include <new>
#include <set>
#include <utility>
#include <vector>

#include "ile_handle.h"

using namespace rift;

namespace {

constexpr uint64_t kStateMagic = 0x31454C4954464952ull;   // "RIFTILE1"
constexpr uint32_t kStateVersion = 1;

struct StateHeader {
    uint64_t magic;
    uint32_t version;
    uint32_t n_bins;
    uint64_t seed;
    uint32_t iteration;
    uint32_t reserved;
};

// Shared memory a block may use on sm_103a (for sizing without a CUDA call).
constexpr int kSmemOptin = 227 * 1024;

// Q window padding of the float32 planes: one chunk window past the end.
constexpr int kQPad = 256 + 16;

}  // namespace


namespace rift {
namespace host {

// Device buffers come from the device's stream-ordered memory pool on the handle's
// stream: no device-wide synchronisation, and freed blocks stay cached for the next
// handle (the pool's release threshold is raised once per process).
void keep_pool_cached()
{
    static std::once_flag once;
    std::call_once(once, [] {
        int dev = 0;
        cudaMemPool_t pool;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
            uint64_t thr = UINT64_MAX;
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
        }
        cudaGetLastError();
    });
}

void release(rift_ile_t *h)
{
    if (!h)
        return;
    if (h->graph)
        cudaGraphExecDestroy(h->graph);
    for (void *p : h->allocs)
        cudaFreeAsync(p, h->stream);
    h->allocs.clear();
    cudaStreamSynchronize(h->stream);
    for (auto &row : h->ev)
        for (auto &e : row)
            cudaEventDestroy(e);
    if (h->own_stream)
        cudaStreamDestroy(h->stream);
    cudaGetLastError();
    delete h;
}

int ensure_events(rift_ile_t *h, int n)
{
    while ((int)h->ev.size() < n) {
        std::array<cudaEvent_t, 4> row{};
        for (auto &e : row)
            if (cudaEventCreate(&e) != cudaSuccess) {
                cudaGetLastError();
                return RIFT_ECUDA;
            }
        h->ev.push_back(row);
    }
    return RIFT_OK;
}

double factorial(int n)
{
    double r = 1.0;
    for (int i = 2; i <= n; ++i)
        r *= i;
    return r;
}

// Wigner small-d d^l_{m',2}(beta) written as a sum over s of
//   (-1)^(m'-2+s) sqrt((l+m')!(l-m')!(l+2)!(l-2)!) / ((l+2-s)! s! (m'-2+s)! (l-m'-s)!)
//   cos(beta/2)^(2l+2-m'-2s) sin(beta/2)^(m'-2+2s),
// so that -2Y_lm(beta, .) = sqrt((2l+1)/4pi) d^l_{m,2}(beta) e^{i m .}.
int wigner_table(int l, int m, double *coef, int8_t *pc, int8_t *ps)
{
    const double norm = std::sqrt((2.0 * l + 1.0) / (4.0 * kPi));
    const double root = std::sqrt(factorial(l + m) * factorial(l - m) * factorial(l + 2) * factorial(l - 2));
    int s0 = std::max(0, 2 - m), s1 = std::min(l + 2, l - m);
    int nt = 0;
    for (int s = s0; s <= s1; ++s) {
        int sign_exp = m - 2 + s;
        double sign = (std::abs(sign_exp) % 2) ? -1.0 : 1.0;
        double v = sign * root / (factorial(l + 2 - s) * factorial(s) * factorial(m - 2 + s) * factorial(l - m - s));
        if (nt >= kMaxWTerms)
            return -1;
        coef[nt] = norm * v;
        pc[nt] = (int8_t)(2 * l + 2 - m - 2 * s);
        ps[nt] = (int8_t)(m - 2 + 2 * s);
        ++nt;
    }
    return nt;
}

// Fourier coefficients of d(iota) = sum_t coef_t cos(iota/2)^pc_t sin(iota/2)^ps_t, a trigonometric
// polynomial of degree l in iota (pc_t + ps_t = 2 l), even for even m and odd for odd m (the
// second index of d^l_{m,2} is even).  With z = exp(i iota/2) a term is
// 4^-l i^-ps (z + 1/z)^pc (z - 1/z)^ps, whose expansion in z has integer coefficients; they are
// summed over t in double-float64 (as discrete sums of long double functions, emulated on some
// hosts, the tables of 21 modes took 2.2 ms of every handle's creation).
void polar_fourier(int l, int m, const double *coef, const int8_t *pc, const int8_t *ps, int nt, double *alpha)
{
    double hi[kMaxL + 1] = {}, lo[kMaxL + 1] = {};
    for (int t = 0; t < nt; ++t) {
        int w[2 * kMaxL + 1] = {1};   // of z^(2 l - 2 n)
        for (int f = 0; f < 2 * l; ++f)
            for (int n = f + 1; n > 0; --n)
                w[n] += f < pc[t] ? w[n - 1] : -w[n - 1];
        for (int u = 0; u <= l; ++u) {   // exp(i u iota) = z^(2 u)
            const double c = ((ps[t] >> 1) & 1) ? -w[l - u] : w[l - u];
            const double p = c * coef[t], v = hi[u] + p, r = v - hi[u];
            lo[u] += std::fma(c, coef[t], -p) + ((hi[u] - (v - r)) + (p - r));
            hi[u] = v;
        }
    }
    for (int u = 0; u <= l; ++u)
        alpha[u] = std::ldexp(hi[u] + lo[u], (u ? 1 : 0) - 2 * l);
}

// Gauss-Legendre nodes and weights on [-1, 1]: Newton's method on P_n from the
// three-term recurrence, starting at the Chebyshev-like guesses cos(pi (i + 3/4) / (n + 1/2)).
void gauss_legendre(int n, double *t, double *w)
{
    for (int i = 0; i < n; ++i) {
        double x = std::cos(kPi * (i + 0.75) / (n + 0.5)), dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= n; ++k) {
                const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (x * p1 - p0) / (x * x - 1.0);
            const double dx = p1 / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-16)
                break;
        }
        t[n - 1 - i] = x;   // ascending
        w[n - 1 - i] = 2.0 / ((1.0 - x * x) * dp * dp);
    }
}

int map_err(int flags)
{
    if (flags & kErrTimeout)
        return RIFT_ETIMEOUT;
    if (flags & kErrRange)
        return RIFT_ERANGE;
    if (flags & kErrNonFinite)
        return RIFT_ENONFINITE;
    return RIFT_OK;
}


SamplerDev sampler_of(const rift_ile_t *h)
{
    SamplerDev S;
    S.P = h->P;
    S.C = h->C;
    S.L = h->Lg;
    S.B = h->cfg.n_bins;
    S.d_min = h->cfg.d_min_mpc;
    S.d_max = h->cfg.d_max_mpc;
    S.floor_eps = h->cfg.adapt_floor;
    S.temper = h->cfg.adapt_temper;
    S.seed = h->cfg.seed;
    S.marg = h->cfg.distance_marg;
    return S;
}

int validate(const rift_ile_config *c)
{
    if (!c || c->n_det < 1 || c->n_det > RIFT_MAX_DET || c->n_modes < 1 || c->n_modes > RIFT_MAX_MODES)
        return RIFT_EINVAL;
    if (c->distance_marg != 0 && c->distance_marg != 1)
        return RIFT_EINVAL;
    if (!c->det_tensor || !c->det_pos_m || !c->lm || !c->q_t0_s)
        return RIFT_EINVAL;
    if (!(c->fs_hz > 0) || c->n_q < 2 || c->n_t < 1 || !(c->t_hi_s >= c->t_lo_s))
        return RIFT_EINVAL;
    if (!(c->d_ref_mpc > 0) || !(c->d_min_mpc > 0) || !(c->d_max_mpc > c->d_min_mpc))
        return RIFT_EINVAL;
    if (c->quad_norm != RIFT_QUAD_QUARTER && c->quad_norm != RIFT_QUAD_HALF)
        return RIFT_EINVAL;
    if (c->precision != RIFT_FP64 && c->precision != RIFT_FP32 && c->precision != RIFT_MIXED)
        return RIFT_EINVAL;
    if (c->n_bins < 2 || c->n_bins > RIFT_MAX_BINS || !(c->adapt_floor >= 0 && c->adapt_floor < 1) ||
        !(c->adapt_temper > 0))
        return RIFT_EINVAL;
    if (c->max_samples < 1 || c->max_samples > (int64_t)0x7fffffff)
        return RIFT_EINVAL;
    std::set<std::pair<int, int>> seen;
    for (int i = 0; i < c->n_modes; ++i) {
        int l = c->lm[2 * i], m = c->lm[2 * i + 1];
        if (l < 2 || l > kMaxL || m < -l || m > l || !seen.insert({l, m}).second)
            return RIFT_EINVAL;
    }
    for (int k = 0; k < c->n_det; ++k) {
        for (int i = 0; i < 9; ++i)
            if (!std::isfinite(c->det_tensor[9 * k + i]))
                return RIFT_EINVAL;
        double r = 0;
        for (int i = 0; i < 3; ++i) {
            if (!std::isfinite(c->det_pos_m[3 * k + i]))
                return RIFT_EINVAL;
            r += c->det_pos_m[3 * k + i] * c->det_pos_m[3 * k + i];
        }
        double rc = std::sqrt(r) / kC;
        double umin = (c->t_lo_s - rc - c->q_t0_s[k]) * c->fs_hz;
        double umax = (c->t_hi_s + rc - c->q_t0_s[k]) * c->fs_hz;
        if (!(umin >= 1e-3) || !(umax <= (double)(c->n_q - 2) - 1e-3))
            return RIFT_ERANGE;
    }
    return RIFT_OK;
}

// Builds float32 planes and Gram copies from the float64 device copies; flags NaN/Inf.
__global__ void prep_overlaps_kernel(const double2 *__restrict__ Q64, const double2 *__restrict__ U64,
                                     const double2 *__restrict__ V64, int K, int M, int n_q, int n_q_pad,
                                     float *__restrict__ Qr32, float2 *__restrict__ U32, float2 *__restrict__ V32,
                                     int *err)
{
    const int64_t total = (int64_t)K * 2 * M * n_q_pad;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t row = e / n_q_pad;
        int c = (int)(e - row * n_q_pad);
        int k = (int)(row / (2 * M)), r = (int)(row % (2 * M));
        float v = 0.f;
        if (c < n_q) {
            double2 q = Q64[((int64_t)k * M + r / 2) * n_q + c];
            double x = (r & 1) ? q.y : q.x;
            if (!isfinite(x))
                atomicOr(err, kErrNonFinite);
            v = (float)x;
        }
        Qr32[e] = v;
    }
    const int64_t g = (int64_t)K * M * M;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < g; e += (int64_t)gridDim.x * blockDim.x) {
        double2 u = U64[e], v = V64[e];
        if (!isfinite(u.x) || !isfinite(u.y) || !isfinite(v.x) || !isfinite(v.y))
            atomicOr(err, kErrNonFinite);
        U32[e] = make_float2((float)u.x, (float)u.y);
        V32[e] = make_float2((float)v.x, (float)v.y);
    }
}

int sync_and_err(rift_ile_t *h, int *flags_out)
{
    int flags = 0;
    CK(cudaMemcpyAsync(&h->host_out[0], h->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    std::memcpy(&flags, &h->host_out[0], sizeof(int));
    if (flags_out)
        *flags_out = flags;
    return map_err(flags);
}

bool use_fp32(const rift_ile_t *h) { return h->cfg.precision != RIFT_FP64; }

bool use_tc64(const rift_ile_t *h) { return h->tc64_on && !h->plain64; }

// Without a tuned plan: tensor-core tiles from this batch size.  They are faster from 10,000 to
// 30,000 samples up (99,999 samples, us, CUDA cores | tensor cores: 2 detectors, 9 modes, 16384 Hz
// 1067 | 471; 3, 21 2164 | 808; 2, 2, 4096 Hz 523 | 310), but their operands are float16 pairs (22
// bits): below the line a batch keeps the float32 products of the CUDA-core kernel.  20,000 samples,
// rms error of ln L, CUDA cores | tensor cores: 2 detectors, 9 modes, SNR 20 2.2e-5 | 2.3e-5, SNR 40
// 3.0e-5 | 3.6e-5, SNR 150 5.9e-5 | 1.8e-4; 1 detector, 12 modes, SNR 40 4.0e-5 | 5.5e-5, SNR 150
// 1.2e-4 | 6.0e-4.
constexpr int64_t kTcMinBatch = 100000;

bool use_tc(const rift_ile_t *h, int64_t n)
{
    if (!h->tc_ok || h->tc_mode == 0)
        return false;
    if (h->tc_mode == 1)
        return true;
    return h->plan.tc >= 0 ? h->plan.tc == 1 : n >= kTcMinBatch;
}

// Below this many samples the CUDA-core kernel takes them in index order: their windows'
// union costs less than the sort.
constexpr int64_t kCoreUnsorted = 1024;

bool sorts_batch(const rift_ile_t *h, int64_t n) { return use_tc(h, n) || n > kCoreUnsorted; }

cudaError_t sort_batch(rift_ile_t *h, int64_t n, int *launched)
{
    *launched = 0;
    return sorts_batch(h, n) ? launch_sort(h->grid, h->key, n, h->sort_scratch, h->perm, h->stream, launched) : cudaSuccess;
}

cudaError_t launch_tiled(rift_ile_t *h, const double *theta, int64_t n, double *lnL_tmarg, double *lnL_t,
                         const double *lnpw, double *lnw)
{
    const BinTable bt{h->bin_i, h->bin_f, std::log((double)h->prob.n_t)};
    PeakOut po;
    if (h->fix_on) {
        po.q = h->aux_q;
        po.m = h->aux_m;
        po.j = h->aux_j;
    }
    const bool tc = use_tc(h, n);
    if (tc)
        h->launches += 1;   // the work units
    cudaError_t e = tc ? launch_lnl_tc(h->prob, bt, theta, h->perm, n, lnL_tmarg, lnL_t, lnpw, lnw, h->err,
                                       TcUnits{h->tc_unit_list, h->tc_unit_cap, h->tile_counter}, h->stream,
                                       nullptr, 0, 0, po)
                       : launch_lnl_fp32(h->prob, bt, theta, sorts_batch(h, n) ? h->perm : nullptr, n, lnL_tmarg,
                                         lnL_t, lnpw, lnw, h->err, h->stream, po);
    if (e != cudaSuccess || !h->fix_on)
        return e;
    // the samples whose float32 terms are large enough for their rounding to reach the
    // parity bar: template term and peak data term again in double-float
    int k = 0;
    e = launch_fix(h->prob, bt, h->fix, theta, n, po, tc ? kPeakBlockTc : 1, h->fix_thr, h->fix_idx, h->fix_count,
                   lnL_tmarg, lnL_t, lnpw, lnw, h->err, h->stream, &k);
    h->launches += k;
    return e;
}

// RIFT_MIXED: samples whose log-weight is within kMixedMargin of the batch maximum
// are re-evaluated in float64 (their weight relative to the largest is >= e^-40).
constexpr double kMixedMargin = 40.0;
// the float32 modes correct every sample whose template term plus largest data term
// exceeds this (k_fixup.cu)
constexpr float kFixThreshold = 600.f;

// Below this many samples the sort costs more than it saves (2 detectors, 2 modes, 401 bins:
// 512 samples 137 us sorted, 110 us unsorted; with 3 detectors and 21 modes the sort's windows
// and launches break even there).
constexpr int64_t kTc64Unsorted = 512;

// Whether the tensor-core kernel in chunks of the handle's batch size beats the plain kernel on
// more samples than that: a chunk costs about 90 us + 2e-3 us x (detectors x modes x bins), a sample
// of the plain kernel 0.1 us + 2e-5 us x the same.  Measured (draws of 2 detectors, 2 modes, 401 bins
// and of 3, 21, 1001; us by chunks | plain): batch size 64 84 a chunk | 0.14 a draw and 150 | 1.35, 512
// 99 | 0.14 and 229 | 1.35; 20,000 draws of the small problem on a handle for 64 samples 26318 | 2821.
bool pays_in_chunks(const rift_ile_t *h)
{
    const double w = (double)h->prob.K * h->prob.M * h->prob.n_t;
    return (double)h->cap * (0.1 + 2e-5 * w) >= 90.0 + 2e-3 * w;
}

int lnl_float64(rift_ile_t *h, const double *theta, int64_t n, bool keyed, double *lnL_tmarg, double *lnL_t,
                const double *lnpw, double *lnw)
{
    if (!use_tc64(h)) {
        CK(launch_lnl_fp64(h->prob, theta, n, lnL_tmarg, lnL_t, lnpw, lnw, h->err, h->stream));
        h->launches += 1;
        return RIFT_OK;
    }
    // a few tiles fill the device by splitting the bins, whatever their windows' width
    const bool sort = n > kTc64Unsorted;
    int k = 0;
    if (sort) {
        if (!keyed) {
            RK(grid_for_batch(h, n));
            CK(launch_keys(h->grid, theta, n, h->key, h->stream));
        }
        CK(launch_sort(h->grid, h->key, n, h->sort_scratch, h->perm, h->stream, &k));
        k += keyed ? 0 : 1;
    }
    int l = 0;
    CK(launch_lnl_tc64(h->prob, h->x64, theta, sort ? h->perm : nullptr, n, lnL_tmarg, lnL_t, lnpw, lnw, h->err,
                       h->stream, nullptr, 0, &l));
    h->launches += k + l;
    return RIFT_OK;
}

// Up to this many selected samples are re-evaluated by a block each in plain float64, longer lists
// on the tensor cores (the count is on the device: each of the two kernels looks at it and leaves
// when it is not its own).
constexpr uint32_t kRefineFew = 512;

int refine_batch(rift_ile_t *h, const double *theta, int64_t n, double *lnL_tmarg, const double *lnpw, double *lnw)
{
    const double *key = lnw ? lnw : lnL_tmarg;
    CK(launch_reduce(key, lnL_tmarg, n, h->red_partial, h->stats, kScratchSlot, h->pooled_scratch, 1, h->err,
                     h->stream));
    CK(launch_select(key, sorts_batch(h, n) ? h->perm : nullptr, n, h->stats, kScratchSlot, kMixedMargin, h->sel_idx, h->sel_count, h->stream));
    if (use_tc64(h)) {
        CK(launch_refine_few(h->prob, theta, h->sel_idx, h->sel_count, kRefineFew, lnL_tmarg, lnpw, lnw, h->err,
                             h->stream));
        CK(launch_lnl_tc64(h->prob, h->x64, theta, h->sel_idx, n, lnL_tmarg, nullptr, lnpw, lnw, h->err,
                           h->stream, h->sel_count, kRefineFew));
        h->launches += 8;
        return RIFT_OK;
    }
    // the tensor-core kernel recomputes the float32 per-bin ln L of the first refine_rows
    // selected samples (a few tiles), so the refinement itself evaluates only the bins
    // within its margin in float64
    int64_t rows = 0;
    if (h->refine_bins && use_tc(h, n)) {
        const BinTable bt{h->bin_i, h->bin_f, std::log((double)h->prob.n_t)};
        rows = std::min<int64_t>(h->refine_rows, n);
        CK(launch_lnl_tc(h->prob, bt, theta, h->sel_idx, rows, lnL_tmarg, h->refine_bins, lnpw, lnw, h->err,
                         TcUnits{h->tc_unit_list, h->tc_unit_cap, h->tile_counter}, h->stream, h->sel_count, 1, n));
        h->launches += 2;
    }
    CK(launch_refine(h->prob, theta, h->sel_idx, h->sel_count, n, lnL_tmarg, lnpw, lnw, h->err, h->stream,
                     h->refine_bins, rows));
    h->launches += 6;
    return RIFT_OK;
}

// Cells per side of a face, at most 2^kMaxFaceOrder (19-bit keys: two digits of the sort).
constexpr int kMaxFaceOrder = 8;

// Sky grid sized for a batch of n samples.
int grid_for_batch(rift_ile_t *h, int64_t n)
{
    SkyGrid g = sky_grid_for(n, h->plan.per_cell);
    const Problem &P = h->prob;
    const bool delay3 = P.K >= 3 && h->plan.delay3;
    if (P.K >= 3 && !delay3) {   // the six faces of a cube
        g.order = 3;
        while (g.order < kMaxFaceOrder && ((6 * (int64_t)h->plan.per_cell) << (2 * g.order)) < n)
            ++g.order;
        g.n_cells = 6 << (2 * g.order);
    }
    if (P.K <= 2 || delay3) {
        g.mode = P.K == 1 ? kSortDelay1 : P.K == 2 ? kSortDelay2 : kSortDelay3;
        if (delay3) {   // as many cells as the sky grid, 8 per level of three delays
            g.order = std::max(1, 2 * g.order / 3);
            g.n_cells = 1 << (3 * g.order);
        }
        g.gmst = P.gmst;
        for (int k = 0; k < std::min(P.K, 3); ++k) {
            double r2 = 0.0;
            for (int i = 0; i < 3; ++i) {
                g.x[k][i] = P.xpos[k][i];
                r2 += P.xpos[k][i] * P.xpos[k][i];
            }
            g.span[k] = std::sqrt(r2);
        }
    }
    h->grid = g;
    return RIFT_OK;
}

// Stage timer: inside a graph capture the record becomes an event node, so replays
// time themselves.
cudaError_t mark(rift_ile_t *h, int slot, int stage)
{
    if (!h->timed)
        return cudaSuccess;
    if (h->capturing)
        return cudaEventRecordWithFlags(h->ev[slot][stage], h->stream, cudaEventRecordExternal);
    return cudaEventRecord(h->ev[slot][stage], h->stream);
}

// ln L for n device-resident samples (theta [n][6]); perm/key scratch from the handle.
int eval_device(rift_ile_t *h, const double *theta, int64_t n, double *lnL_tmarg, double *lnL_t, const double *lnpw,
                double *lnw)
{
    if (!use_fp32(h))
        return lnl_float64(h, theta, n, false, lnL_tmarg, lnL_t, lnpw, lnw);
    RK(choose_plan(h, n, false));
    RK(grid_for_batch(h, n));
    int sorted = 0;
    if (sorts_batch(h, n)) {
        CK(launch_keys(h->grid, theta, n, h->key, h->stream));
        CK(sort_batch(h, n, &sorted));
        ++sorted;
    }
    h->launches += 1 + sorted;   // keys, sort, likelihood
    CK(launch_tiled(h, theta, n, lnL_tmarg, lnL_t, lnpw, lnw));
    if (h->cfg.precision == RIFT_MIXED)
        RK(refine_batch(h, theta, n, lnL_tmarg, lnpw, lnw));
    return RIFT_OK;
}

// One draw -> sort -> likelihood -> reduce (-> adapt) iteration into stats slot `slot`;
// the draw uses sampler iteration (device counter + slot).
int run_iteration(rift_ile_t *h, int64_t n, int slot, bool adapt, bool reset_pooled)
{
    SamplerDev S = sampler_of(h);
    RK(grid_for_batch(h, n));
    CK(mark(h, slot, 0));
    CK(launch_draw(S, h->grid, h->iter_dev, (uint32_t)slot, n, h->theta, h->lnpw, h->bins, h->key, h->stream));
    int sorted = 0;
    if (use_fp32(h))
        CK(sort_batch(h, n, &sorted));
    CK(mark(h, slot, 1));
    if (!use_fp32(h)) {
        RK(lnl_float64(h, h->theta, n, true, h->lnL, nullptr, h->lnpw, h->lnw));
    } else {
        CK(launch_tiled(h, h->theta, n, h->lnL, nullptr, h->lnpw, h->lnw));
        if (h->cfg.precision == RIFT_MIXED)
            RK(refine_batch(h, h->theta, n, h->lnL, h->lnpw, h->lnw));
    }
    CK(mark(h, slot, 2));
    const bool f32_terms = h->cfg.precision == RIFT_FP32;
    CK(launch_reduce(h->lnw, h->lnL, n, h->red_partial, h->stats, slot, h->pooled, reset_pooled ? 1 : 0, h->err,
                     h->stream, f32_terms));
    if (adapt)
        CK(launch_adapt(S, h->bins, h->lnw, n, h->stats, slot, h->hist_partial, h->stream, f32_terms));
    CK(mark(h, slot, 3));
    h->launches += 1 + sorted + (use_fp32(h) ? 1 : 0) + 2 + (adapt ? 2 : 0);
    return RIFT_OK;
}

int enqueue_adapt(rift_ile_t *h, int32_t n_iter, int64_t n)
{
    CK(cudaMemsetAsync(h->err, 0, sizeof(int), h->stream));
    for (int g = 0; g < n_iter; ++g)
        RK(run_iteration(h, n, g, true, g == 0));
    CK(launch_pooled_final(h->pooled, h->final_out, h->iter_dev, (uint32_t)n_iter, h->stream));
    h->launches += 1;
    return RIFT_OK;
}

int collect_result(rift_ile_t *h, int n_iter, rift_ile_result *out)
{
    // host_out layout: [0] err word, [1..8) final, [8..) stats
    CK(cudaMemcpyAsync(&h->host_out[1], h->final_out, sizeof(double) * 6, cudaMemcpyDeviceToHost, h->stream));
    CK(cudaMemcpyAsync(&h->host_out[8], h->stats, sizeof(double) * 8 * n_iter, cudaMemcpyDeviceToHost, h->stream));
    int flags = 0;
    int rc = sync_and_err(h, &flags);
    if (!out)
        return rc;
    std::memset(out, 0, sizeof(*out));
    const double *f = &h->host_out[1];
    out->lnZ = f[0];
    out->sigma_lnZ = f[1];
    out->n_eff = f[2];
    out->n_ess = f[3];
    out->lnL_max = f[4];
    out->n_total = (int64_t)f[5];
    out->n_iter = n_iter;
    out->status = rc;
    for (int g = 0; g < n_iter; ++g) {
        const double *s = &h->host_out[8 + 8 * g];
        out->lnZ_iter[g] = s[0];
        out->sigma_iter[g] = s[1];
        out->n_eff_iter[g] = s[2];
        out->n_ess_iter[g] = s[3];
        if (!h->timed)
            continue;
        float a = 0, b = 0, c = 0, d = 0;
        cudaEventElapsedTime(&a, h->ev[g][0], h->ev[g][1]);
        cudaEventElapsedTime(&b, h->ev[g][1], h->ev[g][2]);
        cudaEventElapsedTime(&c, h->ev[g][2], h->ev[g][3]);
        cudaEventElapsedTime(&d, h->ev[g][0], h->ev[g][3]);
        out->time_ms[0] += a;
        out->time_ms[1] += b;
        out->time_ms[2] += c;
        out->time_ms[3] += d;
    }
    cudaGetLastError();
    return rc;
}

bool graphs_enabled()
{
    const char *env = std::getenv("RIFT_ILE_GRAPHS");
    return !(env && env[0] == '0');
}

void drop_graph(rift_ile_t *h)
{
    if (h->graph)
        cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
    h->graph_iter = 0;
    h->graph_n = 0;
}

// Capture enqueue_adapt(n_iter, n) on the handle's stream into h->graph.
int capture_adapt(rift_ile_t *h, int32_t n_iter, int64_t n)
{
    drop_graph(h);
    CK(cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
    const int64_t l0 = h->launches;
    h->capturing = true;
    int rc = enqueue_adapt(h, n_iter, n);
    h->capturing = false;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(h->stream, &g);
    const int64_t per_run = h->launches - l0;
    h->launches = l0;
    if (rc != RIFT_OK || e != cudaSuccess) {
        if (g)
            cudaGraphDestroy(g);
        cudaGetLastError();
        return rc != RIFT_OK ? rc : RIFT_ECUDA;
    }
    e = cudaGraphInstantiate(&h->graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        h->graph = nullptr;
        cudaGetLastError();
        return RIFT_ECUDA;
    }
    h->graph_iter = n_iter;
    h->graph_n = n;
    h->graph_plan = h->plan;
    h->graph_launches = per_run;
    return RIFT_OK;
}

}  // namespace host
}  // namespace rift

using namespace rift::host;

// ============================================================================ ABI

extern "C" {

const char *rift_ile_strerror(int code)
{
    switch (code) {
    case RIFT_OK: return "ok";
    case RIFT_EINVAL: return "invalid argument";
    case RIFT_ENOMEM: return "out of memory";
    case RIFT_ECUDA: return "CUDA error";
    case RIFT_ERANGE: return "time-shifted Q index outside the Q window";
    case RIFT_ENONFINITE: return "non-finite value in inputs or results";
    case RIFT_ETIMEOUT: return "bounded device wait timed out";
    case RIFT_ESTATE: return "call out of order or malformed state";
    default: return "unknown status";
    }
}

int rift_ile_create(const rift_ile_config *cfg, void *cuda_stream, rift_ile_t **out)
{
    if (!out)
        return RIFT_EINVAL;
    *out = nullptr;
    int v = validate(cfg);
    if (v != RIFT_OK)
        return v;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) {
        cudaGetLastError();
        return RIFT_ECUDA;
    }
    keep_pool_cached();
    rift_ile_t *h = new (std::nothrow) rift_ile_t();
    if (!h)
        return RIFT_ENOMEM;
    h->cfg = *cfg;
    const int K = cfg->n_det, M = cfg->n_modes;
    h->det_tensor.assign(cfg->det_tensor, cfg->det_tensor + 9 * K);
    h->det_pos.assign(cfg->det_pos_m, cfg->det_pos_m + 3 * K);
    h->q_t0.assign(cfg->q_t0_s, cfg->q_t0_s + K);
    h->lm.assign(cfg->lm, cfg->lm + 2 * M);
    h->cfg.det_tensor = h->det_tensor.data();
    h->cfg.det_pos_m = h->det_pos.data();
    h->cfg.q_t0_s = h->q_t0.data();
    h->cfg.lm = h->lm.data();
    h->stream = static_cast<cudaStream_t>(cuda_stream);
    if (!h->stream) {
        // a stream of the handle's own (blocking: ordered with the legacy default
        // stream), so that repeated adaptive sequences can be captured as graphs
        if (cudaStreamCreate(&h->stream) != cudaSuccess) {
            cudaGetLastError();
            delete h;
            return RIFT_ECUDA;
        }
        h->own_stream = true;
    }
    h->cap = cfg->max_samples;

    Problem &P = h->prob;
    P.K = K;
    P.M = M;
    P.n_q = cfg->n_q;
    P.n_t = cfg->n_t;
    P.n_q_pad = ((cfg->n_q + 3) & ~3) + kQPad;
    P.fs = cfg->fs_hz;
    P.t_lo = cfg->t_lo_s;
    P.t_step = cfg->n_t > 1 ? (cfg->t_hi_s - cfg->t_lo_s) / (cfg->n_t - 1) : 0.0;
    P.gmst = cfg->gmst_rad;
    P.d_ref = cfg->d_ref_mpc;
    P.kappa = cfg->quad_norm == RIFT_QUAD_HALF ? 0.5 : 0.25;
    P.dist_marg = cfg->distance_marg;
    P.dm_xlo = cfg->d_ref_mpc / cfg->d_max_mpc;
    P.dm_xhi = cfg->d_ref_mpc / cfg->d_min_mpc;
    P.dm_lnC = std::log(3.0 * cfg->d_ref_mpc * cfg->d_ref_mpc * cfg->d_ref_mpc /
                        (cfg->d_max_mpc * cfg->d_max_mpc * cfg->d_max_mpc -
                         cfg->d_min_mpc * cfg->d_min_mpc * cfg->d_min_mpc));
    P.dm_lnub = P.dm_lnC + std::log((1.0 / (P.dm_xlo * P.dm_xlo * P.dm_xlo) -
                                     1.0 / (P.dm_xhi * P.dm_xhi * P.dm_xhi)) / 3.0);
    gauss_legendre(16, P.gl16_t, P.gl16_w);
    {
        double t10[10], w10[10];
        gauss_legendre(10, t10, w10);
        for (int i = 0; i < 10; ++i) {
            P.gl10_tf[i] = (float)t10[i];
            P.gl10_wf[i] = (float)w10[i];
        }
    }
    P.dm_xlo_f = (float)P.dm_xlo;
    P.dm_xhi_f = (float)P.dm_xhi;
    P.dm_lnC_f = (float)P.dm_lnC;
    P.dm_lnub_f = (float)P.dm_lnub;
    for (int k = 0; k < K; ++k) {
        const double *D = cfg->det_tensor + 9 * k;
        P.Dten[k][0] = D[0];
        P.Dten[k][1] = D[4];
        P.Dten[k][2] = D[8];
        P.Dten[k][3] = 0.5 * (D[1] + D[3]);
        P.Dten[k][4] = 0.5 * (D[2] + D[6]);
        P.Dten[k][5] = 0.5 * (D[5] + D[7]);
        for (int i = 0; i < 6; ++i)
            P.Dten_f[k][i] = (float)P.Dten[k][i];
        for (int i = 0; i < 3; ++i)
            P.xpos[k][i] = cfg->det_pos_m[3 * k + i] / kC;
        P.q_t0[k] = cfg->q_t0_s[k];
        P.ufs0[k] = (P.t_lo - P.q_t0[k]) * P.fs;
        for (int i = 0; i < 3; ++i)
            P.xfs[k][i] = -P.xpos[k][i] * P.fs;
    }
    for (int m = 0; m < M; ++m) {
        P.mode_m[m] = cfg->lm[2 * m + 1];
        int nt = wigner_table(cfg->lm[2 * m], cfg->lm[2 * m + 1], P.wcoef[m], P.wpc[m], P.wps[m]);
        if (nt < 0) {
            release(h);
            return RIFT_EINVAL;
        }
        P.wn[m] = (int8_t)nt;
        for (int t = 0; t < nt; ++t)
            P.wcoef_f[m][t] = (float)P.wcoef[m][t];
    }

    int rc = RIFT_OK;
    const int64_t N = h->cap;
    const int B = cfg->n_bins;
    h->tc_unit_cap = tc_units_cap(N);
    if ((rc = dalloc(h, &h->Q64, (size_t)K * M * cfg->n_q)) || (rc = dalloc(h, &h->U64, (size_t)K * M * M)) ||
        (rc = dalloc(h, &h->V64, (size_t)K * M * M)) || (rc = dalloc(h, &h->Qr32, (size_t)K * 2 * M * P.n_q_pad)) ||
        (rc = dalloc(h, &h->U32, (size_t)K * M * M)) || (rc = dalloc(h, &h->V32, (size_t)K * M * M)) ||
        (rc = dalloc(h, &h->Ttc, (size_t)K * 2 * ((2 * M + 15) / 16 * 16) * ((2 * M + 15) / 16 * 16))) ||
        (rc = dalloc(h, &h->tt_exp, (size_t)K)) ||
        (rc = dalloc(h, &h->bin_i, (size_t)cfg->n_t)) || (rc = dalloc(h, &h->bin_f, (size_t)cfg->n_t)) ||
        (rc = dalloc(h, &h->theta, (size_t)N * 6)) || (rc = dalloc(h, &h->lnpw, (size_t)N)) ||
        (rc = dalloc(h, &h->lnL, (size_t)N)) || (rc = dalloc(h, &h->lnw, (size_t)N)) ||
        (rc = dalloc(h, &h->bins, (size_t)N)) || (rc = dalloc(h, &h->key, (size_t)N)) ||
        (rc = dalloc(h, &h->perm, (size_t)N)) || (rc = dalloc(h, &h->sort_scratch, sort_scratch_words(N))) ||
        (rc = dalloc(h, &h->tile_counter, (size_t)8)) ||
        (rc = dalloc(h, &h->tc_unit_list, (size_t)2 * tc_units_cap(N))) ||
        (rc = dalloc(h, &h->qmax_bits, (size_t)4)) ||
        (rc = dalloc(h, &h->Qtc, (size_t)K * 2 * ((cfg->n_q + 7) / 8 + 17) * ((2 * M + 15) / 16 * 16) * 8)) ||
        (rc = dalloc(h, &h->red_partial, (size_t)5 * kRedBlocks)) ||
        (rc = dalloc(h, &h->hist_partial, (size_t)152 * 12 * B)) ||
        (rc = dalloc(h, &h->stats, (size_t)8 * (RIFT_MAX_ITER + 1))) || (rc = dalloc(h, &h->pooled, (size_t)8)) ||
        (rc = dalloc(h, &h->pooled_scratch, (size_t)8)) || (rc = dalloc(h, &h->sel_idx, (size_t)N)) ||
        (rc = dalloc(h, &h->sel_count, (size_t)kSelectWords)) ||
        (rc = dalloc(h, &h->final_out, (size_t)8)) || (rc = dalloc(h, &h->P, (size_t)6 * B)) ||
        (rc = dalloc(h, &h->C, (size_t)6 * (B + 1))) || (rc = dalloc(h, &h->Lg, (size_t)6 * B)) || (rc = dalloc(h, &h->err, (size_t)4)) ||
        (rc = dalloc(h, &h->iter_dev, (size_t)4))) {
        release(h);
        return rc;
    }
    // the large-term correction runs in the float32 modes (not with the distance marginal,
    // whose per-bin values are no difference of two large terms)
    h->fix_on = cfg->precision != RIFT_FP64 && !cfg->distance_marg;
    if (h->fix_on) {
        int mmax = 0, lmax = 0;
        std::vector<double> alpha((size_t)M * (kMaxL + 1), 0.0);
        for (int m = 0; m < M; ++m) {
            mmax = std::max(mmax, std::abs(cfg->lm[2 * m + 1]));
            lmax = std::max(lmax, cfg->lm[2 * m]);
            polar_fourier(cfg->lm[2 * m], cfg->lm[2 * m + 1], P.wcoef[m], P.wpc[m], P.wps[m], P.wn[m],
                          alpha.data() + (size_t)m * (kMaxL + 1));
        }
        const int dmax = 2 * mmax, nf = 2 * lmax + 1;
        // behind them, their double-float parts (hi, lo)
        const size_t na = alpha.size();
        alpha.resize(2 * na);
        for (size_t i = 0; i < na; ++i) {
            const float pair[2] = {(float)alpha[i], (float)(alpha[i] - (double)(float)alpha[i])};
            std::memcpy(&alpha[na + i], pair, sizeof(double));
        }
        if ((rc = dalloc(h, &h->aux_q, (size_t)N)) || (rc = dalloc(h, &h->aux_m, (size_t)N)) ||
            (rc = dalloc(h, &h->aux_j, (size_t)N)) || (rc = dalloc(h, &h->fix_idx, (size_t)N)) ||
            (rc = dalloc(h, &h->fix_count, (size_t)4)) || (rc = dalloc(h, &h->fix_alpha, alpha.size())) ||
            (rc = dalloc(h, &h->fix_ga, (size_t)K * (dmax + 1) * nf)) ||
            (rc = dalloc(h, &h->fix_hb, (size_t)K * (2 * dmax + 1) * nf)) ||
            (rc = dalloc(h, &h->fix_qdf, (size_t)K * M * cfg->n_q))) {
            release(h);
            return rc;
        }
        if (cudaMemcpyAsync(h->fix_alpha, alpha.data(), sizeof(double) * alpha.size(), cudaMemcpyHostToDevice, h->stream) ||
            cudaStreamSynchronize(h->stream)) {
            cudaGetLastError();
            release(h);
            return RIFT_ECUDA;
        }
        h->fix = FixTables{h->fix_alpha, reinterpret_cast<const float2 *>(h->fix_alpha + na), h->fix_ga, h->fix_hb, h->fix_qdf, dmax, nf};
        // samples with quad32 + |max lin32| above this are corrected: below it the float32
        // rounding stays under 5e-4 (measured, ~3e-7 per unit of the terms at most)
        h->fix_thr = kFixThreshold;
        if (const char *env = std::getenv("RIFT_ILE_FIX_T"))
            h->fix_thr = (float)std::atof(env);
    }
    int dev = 0, max_smem = 0, major = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    P.tc_groups = (cfg->n_q + 7) / 8 + 17;
    {
        const char *env = std::getenv("RIFT_ILE_TC");
        h->tc64_on = cfg->precision != RIFT_FP32 && major == 10 && !(env && env[0] == '0') && lnl_tc64_fits(P, max_smem);
    }
    if (h->tc64_on) {
        unsigned char *scratch = nullptr, *records = nullptr;
        int *unit_counter = nullptr;
        long long *pos = nullptr;
        unsigned long long *units = nullptr;
        if ((rc = dalloc(h, &h->qmax64, tc64_scale_words(K, M))) || (rc = dalloc(h, &h->q_dig, tc64_q_halves(K, M, P.tc_groups))) ||
            (rc = dalloc(h, &h->t_dig, tc64_t_halves(K, M))) || (rc = dalloc(h, &h->t_exp64, (size_t)kMaxDet)) ||
            (rc = dalloc(h, &scratch, tc64_scratch_bytes(K, M, N, sms))) ||
            (rc = dalloc(h, &records, tc64_record_bytes(N, cfg->n_t))) || (rc = dalloc(h, &pos, (size_t)cfg->n_t + kTc64Table)) ||
            (rc = dalloc(h, &unit_counter, (size_t)8 + sms)) ||
            (rc = dalloc(h, &units, (size_t)2 * tc64_units_cap(N)))) {
            release(h);
            return rc;
        }
        h->x64 = Tc64{h->qmax64, h->q_dig, h->t_dig, h->t_exp64, scratch, records, unit_counter, unit_counter + 8, units,
                      tc64_units_cap(N), unit_counter + 4, pos, {}};
        std::vector<long long> host_pos(cfg->n_t + kTc64Table);
        tc64_positions(h->cfg, host_pos.data(), h->x64.u0);
        if (cudaMemsetAsync(unit_counter, 0, sizeof(int) * (8 + sms), h->stream) ||
            cudaMemcpyAsync(pos, host_pos.data(), sizeof(long long) * host_pos.size(), cudaMemcpyHostToDevice, h->stream) ||
            cudaStreamSynchronize(h->stream)) {
            cudaGetLastError();
            release(h);
            return RIFT_ECUDA;
        }
    }
    if (cfg->precision == RIFT_MIXED && !h->tc64_on) {
        h->refine_rows = std::min<int64_t>(N, kRefineRows);
        if ((rc = dalloc(h, &h->refine_bins, (size_t)h->refine_rows * cfg->n_t))) {
            release(h);
            return rc;
        }
    }
    h->host_out.assign(8 + 8 * (RIFT_MAX_ITER + 1) + 8, 0.0);

    // time-bin split table: j * beta = bin_i + bin_f
    std::vector<int> bi(cfg->n_t);
    std::vector<float> bf(cfg->n_t);
    for (int j = 0; j < cfg->n_t; ++j) {
        double jb = (cfg->n_t > 1 ? j * (cfg->t_hi_s - cfg->t_lo_s) / (cfg->n_t - 1) : 0.0) * cfg->fs_hz;
        double fl = std::floor(jb);
        bi[j] = (int)fl;
        bf[j] = (float)(jb - fl);
        if (bf[j] >= 1.0f)
            bf[j] = 0x1.fffffep-1f;
    }
    std::vector<double> P0((size_t)6 * B, 1.0 / B);
    if (cudaMemcpyAsync(h->bin_i, bi.data(), sizeof(int) * cfg->n_t, cudaMemcpyHostToDevice, h->stream) ||
        cudaMemcpyAsync(h->bin_f, bf.data(), sizeof(float) * cfg->n_t, cudaMemcpyHostToDevice, h->stream) ||
        cudaMemcpyAsync(h->P, P0.data(), sizeof(double) * 6 * B, cudaMemcpyHostToDevice, h->stream) ||
        cudaMemsetAsync(h->err, 0, sizeof(int) * 4, h->stream) ||
        cudaMemsetAsync(h->iter_dev, 0, sizeof(uint32_t) * 4, h->stream) || launch_build_cdf(sampler_of(h), h->stream) ||
        cudaStreamSynchronize(h->stream)) {
        cudaGetLastError();
        release(h);
        return RIFT_ECUDA;
    }
    P.Qtc = h->Qtc;
    P.qmax_bits = h->qmax_bits;
    {
        h->tc_ok = major == 10 && lnl_tc_fits(P, max_smem);
        const char *env = std::getenv("RIFT_ILE_TC");
        if (env && env[0] == '0')
            h->tc_mode = 0;
        else if (env && env[0] == '1')
            h->tc_mode = 1;
        if (prepare_sampler_kernels() != cudaSuccess || prepare_refine_kernels() != cudaSuccess ||
            prepare_tile_kernels() != cudaSuccess || (h->tc_ok && prepare_tc_kernels() != cudaSuccess) ||
            prepare_fix_kernels() != cudaSuccess || (h->tc64_on && prepare_tc64_kernels() != cudaSuccess)) {
            cudaGetLastError();
            release(h);
            return RIFT_ECUDA;
        }
    }
    P.Q64 = h->Q64;
    P.U64 = h->U64;
    P.V64 = h->V64;
    P.Qr32 = h->Qr32;
    P.U32 = h->U32;
    P.V32 = h->V32;
    P.Ttc = h->Ttc;
    P.tt_exp = h->tt_exp;
    *out = h;
    return RIFT_OK;
}

void rift_ile_destroy(rift_ile_t *h) { release(h); }

int64_t rift_ile_kernel_launches(const rift_ile_t *h) { return h ? h->launches : -1; }

int rift_ile_get_plan(const rift_ile_t *h, int32_t *lnl_kernel, int32_t *samples_per_cell)
{
    if (!h)
        return RIFT_EINVAL;
    const int64_t n = h->last_n > 0 ? h->last_n : h->cap;
    if (lnl_kernel)
        *lnl_kernel = !use_fp32(h) ? RIFT_KERNEL_FP64 : use_tc(h, n) ? RIFT_KERNEL_TENSOR : RIFT_KERNEL_CUDA_CORE;
    if (samples_per_cell)
        *samples_per_cell = h->plan.per_cell;
    return RIFT_OK;
}

int64_t rift_ile_footprint(const rift_ile_config *cfg)
{
    if (validate(cfg) != RIFT_OK)
        return -1;
    const int64_t K = cfg->n_det, M = cfg->n_modes, N = cfg->max_samples, B = cfg->n_bins, nt = cfg->n_t;
    const int64_t nq = cfg->n_q, nq_pad = ((nq + 3) & ~3) + kQPad;
    const int64_t groups = (nq + 7) / 8 + 17, kp = (2 * M + 15) / 16 * 16;
    // digits and scratch of the float64-accurate tensor-core kernel (k_tile_tc64.cu)
    Problem Pf{};
    Pf.K = cfg->n_det;
    Pf.M = cfg->n_modes;
    Pf.n_q = cfg->n_q;
    Pf.n_t = cfg->n_t;
    Pf.dist_marg = cfg->distance_marg;
    const bool digits = cfg->precision != RIFT_FP32 && lnl_tc64_fits(Pf, kSmemOptin);
    const int64_t sizes[] = {
        K * M * nq * 16, 2 * K * M * M * 16, K * 2 * M * nq_pad * 4, 2 * K * M * M * 8, K * 2 * kp * kp * 2, K * 4,
        2 * nt * 4,
        N * 6 * 8, 3 * N * 8, N * 8, 2 * N * 4, (int64_t)sort_scratch_words(N) * 4, 32, 16, 16 * tc_units_cap(N),
        K * 2 * groups * kp * 8 * 2, 5 * kRedBlocks * 8, 152 * 12 * B * 8, 8 * (RIFT_MAX_ITER + 1) * 8, 3 * 8 * 8,
        N * 4, 16, 6 * B * 8, 6 * (B + 1) * 8, 6 * B * 8, 16, (int64_t)kSelectWords * 4,
        cfg->precision == RIFT_MIXED && !digits ? std::min<int64_t>(N, kRefineRows) * nt * 8 : 0,
        digits ? 2 * (int64_t)(tc64_q_halves(K, M, groups) + tc64_t_halves(K, M)) + 8 * (int64_t)tc64_scale_words(K, M) + 8 * 16 + 152 * 4 + 8 * (nt + kTc64Table) +
                     (int64_t)(16 * tc64_units_cap(N) + tc64_scratch_bytes(K, M, N, 152) + tc64_record_bytes(N, cfg->n_t))
               : 0,
        // large-term correction: per-sample side outputs and list, double-float tables of the
        // template term (at most 13 x 13 + 25 x 13 coefficients a detector) and of Q
        cfg->precision != RIFT_FP64 && !cfg->distance_marg ? 4 * N * 4 + 16 + 16 * (kMaxL + 1) * M + 64 + K * 494 * 16 + K * M * nq * 16
                                                            : 0};
    int64_t total = 0;
    for (int64_t b : sizes)
        total += b + 16 + 255;
    // the unused ends of the slabs (at most a quarter each, 17 of them hold fifty buffers of the
    // largest size that shares one) and the rest of the last, event and stream
    // bookkeeping
    return total + 17 * (int64_t)(kSlab / 4) + (int64_t)kSlab + 64 * 1024;
}

int rift_ile_set_overlaps(rift_ile_t *h, const void *Q, const void *U, const void *V, int mem)
{
    if (!h || !Q || !U || !V || (mem != RIFT_MEM_HOST && mem != RIFT_MEM_DEVICE))
        return RIFT_EINVAL;
    const int K = h->prob.K, M = h->prob.M, nq = h->prob.n_q;
    const size_t qb = sizeof(double2) * (size_t)K * M * nq, gb = sizeof(double2) * (size_t)K * M * M;
    const cudaMemcpyKind kind = mem == RIFT_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    // symmetry checks on host copies of U, V (Sec. V A: U^* = U^T, V = V^T)
    std::vector<double> hu(2 * (size_t)K * M * M), hv(2 * (size_t)K * M * M);
    if (mem == RIFT_MEM_HOST) {
        std::memcpy(hu.data(), U, gb);
        std::memcpy(hv.data(), V, gb);
    } else {
        CK(cudaMemcpyAsync(hu.data(), U, gb, cudaMemcpyDeviceToHost, h->stream));
        CK(cudaMemcpyAsync(hv.data(), V, gb, cudaMemcpyDeviceToHost, h->stream));
        CK(cudaStreamSynchronize(h->stream));
    }
    for (int k = 0; k < K; ++k) {
        double su = 0, sv = 0;
        for (size_t e = 0; e < (size_t)2 * M * M; ++e) {
            double a = std::fabs(hu[2 * (size_t)k * M * M + e]), b = std::fabs(hv[2 * (size_t)k * M * M + e]);
            if (!std::isfinite(a) || !std::isfinite(b))
                return RIFT_ENONFINITE;
            su = std::max(su, a);
            sv = std::max(sv, b);
        }
        for (int a = 0; a < M; ++a)
            for (int b = 0; b < M; ++b) {
                size_t ab = 2 * (((size_t)k * M + a) * M + b), ba = 2 * (((size_t)k * M + b) * M + a);
                if (std::fabs(hu[ab] - hu[ba]) > 1e-10 * su || std::fabs(hu[ab + 1] + hu[ba + 1]) > 1e-10 * su)
                    return RIFT_EINVAL;
                if (std::fabs(hv[ab] - hv[ba]) > 1e-10 * sv || std::fabs(hv[ab + 1] - hv[ba + 1]) > 1e-10 * sv)
                    return RIFT_EINVAL;
            }
    }
    CK(cudaMemsetAsync(h->err, 0, sizeof(int), h->stream));
    CK(cudaMemcpyAsync(h->Q64, Q, qb, kind, h->stream));
    CK(cudaMemcpyAsync(h->U64, U, gb, kind, h->stream));
    CK(cudaMemcpyAsync(h->V64, V, gb, kind, h->stream));
    return install_overlaps(h);
}

int rift_ile_set_waveforms(rift_ile_t *h, int32_t n_freq, const double *freqs, const void *hlm, const void *data,
                           const double *weights, int mem)
{
    if (!h || n_freq < 2 || !freqs || !hlm || !data || !weights || (mem != RIFT_MEM_HOST && mem != RIFT_MEM_DEVICE))
        return RIFT_EINVAL;
    const int K = h->prob.K, M = h->prob.M, F = n_freq;
    const size_t fb = sizeof(double) * F, hb = sizeof(double2) * (size_t)M * F, db = sizeof(double2) * (size_t)K * F,
                 wb = sizeof(double) * (size_t)K * F;
    std::vector<void *> tmp;
    auto grab = [&](size_t bytes) -> void * {
        void *q = nullptr;
        if (cudaMallocAsync(&q, bytes, h->stream) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        tmp.push_back(q);
        return q;
    };
    auto A = static_cast<double2 *>(grab(sizeof(double2) * (size_t)K * M * F));
    auto t0 = static_cast<double *>(grab(sizeof(double) * K));
    auto uvp = static_cast<double *>(grab(sizeof(double) * uv_scratch_doubles(K, M, F)));
    auto nidx = static_cast<int *>(grab(sizeof(int) * F));
    auto info_dev = static_cast<WaveformInfo *>(grab(sizeof(WaveformInfo)));
    int launched = 0;
    const double *df = freqs, *dw = weights;
    const double2 *dh = static_cast<const double2 *>(hlm), *dd = static_cast<const double2 *>(data);
    int rc = (A && t0 && uvp && nidx && info_dev) ? RIFT_OK : RIFT_ENOMEM;
    if (rc == RIFT_OK && mem == RIFT_MEM_HOST) {
        auto f2 = static_cast<double *>(grab(fb));
        auto h2 = static_cast<double2 *>(grab(hb));
        auto d2 = static_cast<double2 *>(grab(db));
        auto w2 = static_cast<double *>(grab(wb));
        if (!f2 || !h2 || !d2 || !w2)
            rc = RIFT_ENOMEM;
        else if (cudaMemcpyAsync(f2, freqs, fb, cudaMemcpyHostToDevice, h->stream) ||
                 cudaMemcpyAsync(h2, hlm, hb, cudaMemcpyHostToDevice, h->stream) ||
                 cudaMemcpyAsync(d2, data, db, cudaMemcpyHostToDevice, h->stream) ||
                 cudaMemcpyAsync(w2, weights, wb, cudaMemcpyHostToDevice, h->stream))
            rc = RIFT_ECUDA;
        df = f2;
        dh = h2;
        dd = d2;
        dw = w2;
    }
    // mirror-symmetric grid, weights finite, non-negative and symmetric in f: checked on the
    // device (of device inputs, a copy of the grid and the weights to the host and the loops over
    // them took a fifth of the call).  Q by FFT when the grid lies on a lattice, else the direct
    // sum.  RIFT_ILE_DFT=1 forces the direct sum.
    WaveformInfo info{};
    if (rc == RIFT_OK &&
        (launch_waveform_check(df, dw, K, F, h->prob.fs, nidx, info_dev, h->stream) ||
         cudaMemcpyAsync(&info, info_dev, sizeof(info), cudaMemcpyDeviceToHost, h->stream) ||
         cudaStreamSynchronize(h->stream)))
        rc = RIFT_ECUDA;
    if (rc == RIFT_OK && info.bad != ~0ull)
        rc = (info.bad & 3ull) == (unsigned)kWaveformNonFinite ? RIFT_ENONFINITE : RIFT_EINVAL;
    FftPlan plan{};
    const int lattice = info.off ? 0 : waveform_lattice(h->prob.fs, info.gap);
    bool use_fft = rc == RIFT_OK && lattice > 0 &&
                   !(std::getenv("RIFT_ILE_DFT") && std::getenv("RIFT_ILE_DFT")[0] == '1');
    if (use_fft) {
        plan.L = lattice;
        plan.f0 = info.f0;
        plan.nidx = nidx;
        const bool pruned = fft_pruned(plan.L, h->prob.n_q);
        plan.X = static_cast<double2 *>(grab(sizeof(double2) * (size_t)K * M * plan.L));
        plan.T = static_cast<double2 *>(grab(sizeof(double2) * (size_t)(plan.L / 2)));
        if (pruned)
            plan.jidx = static_cast<int *>(grab(sizeof(int) * (size_t)plan.L));
        else
            plan.Y = static_cast<double2 *>(grab(sizeof(double2) * (size_t)K * M * plan.L));
        if (!plan.X || !plan.T || (pruned ? !plan.jidx : !plan.Y))
            use_fft = false;   // the direct sum needs no scratch of this size
    }
    if (rc == RIFT_OK &&
        (cudaMemcpyAsync(t0, h->q_t0.data(), sizeof(double) * K, cudaMemcpyHostToDevice, h->stream) ||
         cudaMemsetAsync(h->err, 0, sizeof(int), h->stream) ||
         launch_precompute(dh, dd, dw, df, K, M, F, t0, h->prob.fs, h->prob.n_q, A, uvp, h->Q64, h->U64, h->V64,
                           h->stream, use_fft ? &plan : nullptr, &launched)))
        rc = RIFT_ECUDA;
    if (rc == RIFT_OK)
        h->launches += launched + 2;
    for (void *q : tmp)
        cudaFreeAsync(q, h->stream);
    if (rc != RIFT_OK) {
        cudaStreamSynchronize(h->stream);
        cudaGetLastError();
        return rc;
    }
    return install_overlaps(h);
}

}  // extern "C"

namespace rift {
namespace host {

// float32 and tensor-core copies of the overlaps now in Q64/U64/V64; marks them set.
int install_overlaps(rift_ile_t *h)
{
    const int K = h->prob.K, M = h->prob.M, nq = h->prob.n_q;
    int64_t tot = (int64_t)K * 2 * M * h->prob.n_q_pad;
    int grid = (int)std::min<int64_t>((tot + 255) / 256, 152 * 8);
    prep_overlaps_kernel<<<grid, 256, 0, h->stream>>>(h->Q64, h->U64, h->V64, K, M, nq, h->prob.n_q_pad, h->Qr32,
                                                      h->U32, h->V32, h->err);
    CK(cudaGetLastError());
    h->launches += 1;
    if (h->tc_ok) {
        CK(launch_prep_tc(h->Q64, K, M, nq, h->prob.tc_groups, h->qmax_bits, h->Qtc, h->stream));
        CK(launch_prep_tt(h->U64, h->V64, K, M, h->Ttc, h->tt_exp, h->stream));
        h->launches += 3;
    }
    if (h->tc64_on) {
        CK(launch_prep_tc64(h->prob, h->qmax64, h->q_dig, h->t_dig, h->t_exp64, h->err, h->stream));
        h->launches += 3;
    }
    if (h->fix_on) {
        CK(launch_fix_prep(h->prob, h->fix, h->stream));
        h->launches += 2;
    }
    int flags = 0;
    int rc = sync_and_err(h, &flags);
    h->plain64 = (flags & kNoteUneven) != 0;
    h->have_overlaps = (rc == RIFT_OK);
    return rc;
}

}  // namespace host
}  // namespace rift

extern "C" {

int rift_ile_wait_selftest(rift_ile_t *h, int64_t limit_ns)
{
    if (!h || limit_ns < 1000 || limit_ns > 2000000000)
        return RIFT_EINVAL;
    CK(cudaMemsetAsync(h->err, 0, sizeof(int), h->stream));
    CK(launch_wait_probe((uint64_t)limit_ns, h->err, h->stream));
    h->launches += 1;
    return sync_and_err(h);
}

int rift_ile_get_overlaps(const rift_ile_t *h, void *Q, void *U, void *V, int mem)
{
    if (!h || (mem != RIFT_MEM_HOST && mem != RIFT_MEM_DEVICE))
        return RIFT_EINVAL;
    if (!h->have_overlaps)
        return RIFT_ESTATE;
    const int K = h->prob.K, M = h->prob.M;
    const cudaMemcpyKind kind = mem == RIFT_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    if (Q)
        CK(cudaMemcpyAsync(Q, h->Q64, sizeof(double2) * (size_t)K * M * h->prob.n_q, kind, h->stream));
    if (U)
        CK(cudaMemcpyAsync(U, h->U64, sizeof(double2) * (size_t)K * M * M, kind, h->stream));
    if (V)
        CK(cudaMemcpyAsync(V, h->V64, sizeof(double2) * (size_t)K * M * M, kind, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    return RIFT_OK;
}

int rift_ile_eval(rift_ile_t *h, const double *theta, int64_t n, int mem, double *lnL_tmarg, double *lnL_t)
{
    if (!h || n < 0 || (n > 0 && (!theta || !lnL_tmarg)) || (mem != RIFT_MEM_HOST && mem != RIFT_MEM_DEVICE))
        return RIFT_EINVAL;
    if (!h->have_overlaps)
        return RIFT_ESTATE;
    if (n == 0)
        return RIFT_OK;
    const int nt = h->prob.n_t;
    int64_t chunk = h->cap;
    double *stage_t = nullptr;
    if (lnL_t && mem == RIFT_MEM_HOST) {
        chunk = std::min<int64_t>(chunk, std::max<int64_t>(1, (int64_t)(64 << 20) / nt));
        void *q = nullptr;
        if (cudaMallocAsync(&q, sizeof(double) * (size_t)chunk * nt, h->stream) != cudaSuccess) {
            cudaGetLastError();
            return RIFT_ENOMEM;
        }
        stage_t = static_cast<double *>(q);
    }
    int rc = RIFT_OK;
    CK(cudaMemsetAsync(h->err, 0, sizeof(int), h->stream));
    h->last_n = 0;   // the staging buffers no longer hold a drawn batch
    for (int64_t i0 = 0; i0 < n && rc == RIFT_OK; i0 += chunk) {
        const int64_t c = std::min(chunk, n - i0);
        const double *th = theta + 6 * i0;
        double *o = lnL_tmarg + i0;
        double *ot = lnL_t ? lnL_t + i0 * nt : nullptr;
        if (mem == RIFT_MEM_HOST) {
            if (cudaMemcpyAsync(h->theta, th, sizeof(double) * 6 * c, cudaMemcpyHostToDevice, h->stream) != cudaSuccess) {
                rc = RIFT_ECUDA;
                break;
            }
            rc = eval_device(h, h->theta, c, h->lnL, stage_t, nullptr, nullptr);
            if (rc == RIFT_OK &&
                (cudaMemcpyAsync(o, h->lnL, sizeof(double) * c, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
                 (ot && cudaMemcpyAsync(ot, stage_t, sizeof(double) * c * nt, cudaMemcpyDeviceToHost, h->stream) !=
                            cudaSuccess)))
                rc = RIFT_ECUDA;
        } else {
            rc = eval_device(h, th, c, o, ot, nullptr, nullptr);
        }
    }
    if (stage_t)
        cudaFreeAsync(stage_t, h->stream);
    int rc2 = sync_and_err(h);
    return rc != RIFT_OK ? rc : rc2;
}

int rift_ile_coeffs(rift_ile_t *h, const double *theta, int64_t n, int mem, double *c, double *dt, double *quad)
{
    if (!h || n < 0 || (n > 0 && !theta) || (mem != RIFT_MEM_HOST && mem != RIFT_MEM_DEVICE))
        return RIFT_EINVAL;
    if (!h->have_overlaps)
        return RIFT_ESTATE;
    if (n == 0)
        return RIFT_OK;
    const bool fp64 = h->cfg.precision == RIFT_FP64;
    const int K = h->prob.K, M = h->prob.M;
    if (mem == RIFT_MEM_DEVICE) {
        CK(launch_coeffs(h->prob, fp64, theta, n, reinterpret_cast<double2 *>(c), dt, quad, h->stream));
        return sync_and_err(h);
    }
    const int64_t chunk = std::min<int64_t>(h->cap, 1 << 16);
    double2 *dc = nullptr;
    double *ddt = nullptr, *dq = nullptr;
    std::vector<void *> tmp;
    auto grab = [&](size_t bytes) -> void * {
        void *q = nullptr;
        if (cudaMallocAsync(&q, bytes, h->stream) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        tmp.push_back(q);
        return q;
    };
    dc = static_cast<double2 *>(grab(sizeof(double2) * chunk * K * M));
    ddt = static_cast<double *>(grab(sizeof(double) * chunk * K));
    dq = static_cast<double *>(grab(sizeof(double) * chunk));
    int rc = (dc && ddt && dq) ? RIFT_OK : RIFT_ENOMEM;
    for (int64_t i0 = 0; i0 < n && rc == RIFT_OK; i0 += chunk) {
        const int64_t m = std::min(chunk, n - i0);
        if (cudaMemcpyAsync(h->theta, theta + 6 * i0, sizeof(double) * 6 * m, cudaMemcpyHostToDevice, h->stream) ||
            launch_coeffs(h->prob, fp64, h->theta, m, c ? dc : nullptr, dt ? ddt : nullptr, quad ? dq : nullptr,
                          h->stream) ||
            (c && cudaMemcpyAsync(c + 2 * i0 * K * M, dc, sizeof(double2) * m * K * M, cudaMemcpyDeviceToHost,
                                  h->stream)) ||
            (dt && cudaMemcpyAsync(dt + i0 * K, ddt, sizeof(double) * m * K, cudaMemcpyDeviceToHost, h->stream)) ||
            (quad && cudaMemcpyAsync(quad + i0, dq, sizeof(double) * m, cudaMemcpyDeviceToHost, h->stream)))
            rc = RIFT_ECUDA;
    }
    for (void *q : tmp)
        cudaFreeAsync(q, h->stream);
    cudaStreamSynchronize(h->stream);
    h->last_n = 0;
    cudaGetLastError();
    return rc;
}

int rift_ile_marginalize(rift_ile_t *h, int64_t n_samples, rift_ile_result *out)
{
    if (!h || n_samples < 1 || n_samples > h->cap)
        return RIFT_EINVAL;
    if (!h->have_overlaps)
        return RIFT_ESTATE;
    RK(choose_plan(h, n_samples));
    RK(ensure_events(h, 1));
    h->timed = true;
    CK(cudaMemsetAsync(h->err, 0, sizeof(int), h->stream));
    RK(run_iteration(h, n_samples, 0, false, true));
    CK(launch_pooled_final(h->pooled, h->final_out, h->iter_dev, 1, h->stream));
    h->launches += 1;
    h->iteration += 1;
    h->last_n = n_samples;
    return collect_result(h, 1, out);
}

int rift_ile_adapt(rift_ile_t *h, int32_t n_iter, int64_t n_per_iter, rift_ile_result *out)
{
    if (!h || n_iter < 1 || n_iter > RIFT_MAX_ITER || n_per_iter < 1 || n_per_iter > h->cap)
        return RIFT_EINVAL;
    if (!h->have_overlaps)
        return RIFT_ESTATE;
    RK(choose_plan(h, n_per_iter));
    RK(ensure_events(h, n_iter));
    h->timed = true;
    const bool same_graph = h->graph && h->graph_iter == n_iter && h->graph_n == n_per_iter &&
                            h->graph_plan == h->plan;
    const bool repeat = h->last_shape_iter == n_iter && h->last_shape_n == n_per_iter;
    if (graphs_enabled() && (same_graph || repeat)) {
        // a repeated shape: capture once, then replay
        if (!same_graph)
            RK(capture_adapt(h, n_iter, n_per_iter));
        CK(cudaGraphLaunch(h->graph, h->stream));
        h->launches += h->graph_launches;
    } else {
        RK(enqueue_adapt(h, n_iter, n_per_iter));
    }
    h->last_shape_iter = n_iter;
    h->last_shape_n = n_per_iter;
    h->iteration += (uint32_t)n_iter;
    h->last_n = n_per_iter;
    return collect_result(h, n_iter, out);
}

int rift_ile_last_batch(rift_ile_t *h, int mem, double *theta, double *lnp_minus_lnps, double *lnL_tmarg, double *lnw,
                        int64_t *n_out)
{
    if (!h || (mem != RIFT_MEM_HOST && mem != RIFT_MEM_DEVICE))
        return RIFT_EINVAL;
    const int64_t n = h->last_n;
    if (n_out)
        *n_out = n;
    if (n == 0)
        return RIFT_ESTATE;
    const cudaMemcpyKind kind = mem == RIFT_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    if (theta)
        CK(cudaMemcpyAsync(theta, h->theta, sizeof(double) * 6 * n, kind, h->stream));
    if (lnp_minus_lnps)
        CK(cudaMemcpyAsync(lnp_minus_lnps, h->lnpw, sizeof(double) * n, kind, h->stream));
    if (lnL_tmarg)
        CK(cudaMemcpyAsync(lnL_tmarg, h->lnL, sizeof(double) * n, kind, h->stream));
    if (lnw)
        CK(cudaMemcpyAsync(lnw, h->lnw, sizeof(double) * n, kind, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    return RIFT_OK;
}

int rift_ile_fair_draws(rift_ile_t *h, int64_t n_draws, uint64_t seed, int mem, double *theta, double *t,
                        int64_t *index)
{
    if (!h || n_draws < 0 || (mem != RIFT_MEM_HOST && mem != RIFT_MEM_DEVICE) || h->cfg.distance_marg)
        return RIFT_EINVAL;
    if (n_draws == 0)
        return RIFT_OK;
    if (!theta && !t && !index)
        return RIFT_EINVAL;
    const int64_t n = h->last_n;
    if (n == 0)
        return RIFT_ESTATE;
    const int nt = h->prob.n_t;
    int64_t chunk = std::max<int64_t>(1, std::min<int64_t>(n_draws, (int64_t)(16 << 20) / nt));
    const bool plain = !use_tc64(h) || (chunk > h->cap && !pays_in_chunks(h));
    if (!plain)
        chunk = std::min(chunk, h->cap);   // the sort's buffers hold cap samples
    std::vector<void *> tmp;
    auto grab = [&](size_t bytes) -> void * {
        void *q = nullptr;
        if (cudaMallocAsync(&q, bytes, h->stream) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        tmp.push_back(q);
        return q;
    };
    auto W = static_cast<uint64_t *>(grab(sizeof(uint64_t) * n));
    auto E = static_cast<uint64_t *>(grab(sizeof(uint64_t) * n));
    auto scan = static_cast<uint64_t *>(grab(sizeof(uint64_t) * scan_scratch_words(n)));
    auto idx = static_cast<int64_t *>(grab(sizeof(int64_t) * n_draws));
    auto th = static_cast<double *>(grab(sizeof(double) * 6 * n_draws));
    auto Ut = static_cast<uint64_t *>(grab(sizeof(uint64_t) * n_draws));
    auto tt = static_cast<double *>(grab(sizeof(double) * n_draws));
    auto jj = static_cast<int32_t *>(grab(sizeof(int32_t) * n_draws));
    auto bins = static_cast<double *>(grab(sizeof(double) * chunk * nt));
    auto lt = static_cast<double *>(grab(sizeof(double) * chunk));
    int rc = (W && E && scan && idx && th && Ut && tt && jj && bins && lt) ? RIFT_OK : RIFT_ENOMEM;
    const cudaMemcpyKind kind = mem == RIFT_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    auto run = [&]() -> int {
        CK(cudaMemsetAsync(h->err, 0, sizeof(int), h->stream));
        // the batch's largest ln w (checks every ln w is finite)
        CK(launch_reduce(h->lnw, h->lnL, n, h->red_partial, h->stats, kScratchSlot, h->pooled_scratch, 1, h->err,
                         h->stream));
        int k = 0;
        CK(launch_fair_select(h->lnw, n, h->stats, kScratchSlot, W, E, scan, seed, n_draws, h->theta, idx, th, Ut,
                              h->stream, &k));
        h->launches += 2 + k;
        // time bins from each drawn sample's per-bin ln L, in float64 (the draws are few)
        for (int64_t c0 = 0; c0 < n_draws; c0 += chunk) {
            const int64_t m = std::min(chunk, n_draws - c0);
            if (plain) {
                CK(launch_lnl_fp64(h->prob, th + 6 * c0, m, lt, bins, nullptr, nullptr, h->err, h->stream));
                h->launches += 1;
            } else {
                RK(lnl_float64(h, th + 6 * c0, m, false, lt, bins, nullptr, nullptr));
            }
            CK(launch_fair_time(bins, m, nt, Ut + c0, h->prob.t_lo, h->prob.t_step, jj + c0, tt + c0, h->stream));
            h->launches += 1;
        }
        if (theta)
            CK(cudaMemcpyAsync(theta, th, sizeof(double) * 6 * n_draws, kind, h->stream));
        if (t)
            CK(cudaMemcpyAsync(t, tt, sizeof(double) * n_draws, kind, h->stream));
        if (index)
            CK(cudaMemcpyAsync(index, idx, sizeof(int64_t) * n_draws, kind, h->stream));
        return RIFT_OK;
    };
    if (rc == RIFT_OK)
        rc = run();
    for (void *q : tmp)
        cudaFreeAsync(q, h->stream);
    const int rc2 = sync_and_err(h);
    return rc != RIFT_OK ? rc : rc2;
}

int rift_ile_get_sampler(const rift_ile_t *h, double *P)
{
    if (!h || !P)
        return RIFT_EINVAL;
    CK(cudaMemcpyAsync(P, h->P, sizeof(double) * 6 * h->cfg.n_bins, cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    return RIFT_OK;
}

int rift_ile_get_state(const rift_ile_t *h, void *buf, size_t *len)
{
    if (!h || !len)
        return RIFT_EINVAL;
    const size_t need = sizeof(StateHeader) + sizeof(double) * 6 * h->cfg.n_bins;
    if (!buf) {
        *len = need;
        return RIFT_OK;
    }
    if (*len < need)
        return RIFT_EINVAL;
    StateHeader hd{kStateMagic, kStateVersion, (uint32_t)h->cfg.n_bins, h->cfg.seed, h->iteration, 0};
    std::memcpy(buf, &hd, sizeof(hd));
    int rc = rift_ile_get_sampler(h, reinterpret_cast<double *>(static_cast<char *>(buf) + sizeof(hd)));
    if (rc != RIFT_OK)
        return rc;
    *len = need;
    return RIFT_OK;
}

int rift_ile_set_state(rift_ile_t *h, const void *buf, size_t len)
{
    if (!h || !buf)
        return RIFT_EINVAL;
    const size_t need = sizeof(StateHeader) + sizeof(double) * 6 * h->cfg.n_bins;
    if (len != need)
        return RIFT_ESTATE;
    StateHeader hd;
    std::memcpy(&hd, buf, sizeof(hd));
    if (hd.magic != kStateMagic || hd.version != kStateVersion || hd.n_bins != (uint32_t)h->cfg.n_bins)
        return RIFT_ESTATE;
    const double *P = reinterpret_cast<const double *>(static_cast<const char *>(buf) + sizeof(hd));
    for (int e = 0; e < 6 * h->cfg.n_bins; ++e)
        if (!(P[e] >= 0.0) || !std::isfinite(P[e]))
            return RIFT_ESTATE;
    drop_graph(h);   // the seed is a kernel argument of the captured draws
    h->cfg.seed = hd.seed;
    h->iteration = hd.iteration;
    CK(cudaMemcpyAsync(h->iter_dev, &h->iteration, sizeof(uint32_t), cudaMemcpyHostToDevice, h->stream));
    CK(cudaMemcpyAsync(h->P, P, sizeof(double) * 6 * h->cfg.n_bins, cudaMemcpyHostToDevice, h->stream));
    CK(launch_build_cdf(sampler_of(h), h->stream));
    CK(cudaStreamSynchronize(h->stream));
    h->last_n = 0;
    return RIFT_OK;
}

}  // extern "C"
