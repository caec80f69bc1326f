// Float32 likelihood kernel on the CUDA cores (arXiv:2505.11655 Sec. II A,
// Eq. (def:lnL:Decomposed), time-marginalised on a uniform grid).
//
// A block owns 8 samples (4 when there are few), a warp each:
//   1. prologue: float64 sky trigonometry and arrival delays, float32 responses F_k and
//      harmonics Y_lm, coefficients c_k,lm = x F_k Y_lm as real components C[r, s]
//      (r = 2m: Re, 2m+1: Im), template term;
//   2. for each chunk of up to 1024 time bins and each detector, on the Q sample grid
//         R[s, c] = sum_r C[r, s] Qr[r, base + c]     (= Re sum_lm conj(c_lm) Q_lm)
//      over all columns that the chunk's bins reach at any of the block's samples (a thread
//      contracts 4 columns for 8 samples, Q straight from L2), then R is interpolated linearly
//      at every bin's shifted time (interpolation commutes with the mode sum) and summed over
//      detectors in registers: lane l of the sample's warp has the bins l, l + 32, ...;
//   3. each chunk is folded into the sample's online log-sum-exp; ln L_tmarg = max + ln(sum) -
//      quad - ln n_t in float64.
// Samples whose delays differ by more than the R tile holds are contracted in turn.
//
// What bounds it is the float32 multiply-adds of the contraction (2M per column and sample); a
// sample's time bins are one chunk, so a column is contracted once, whatever the delays of its
// neighbours in the sort: unsorted or thinly spread samples cost the union of their windows
// (at most 1.4 times one window at 16384 Hz).  Tiles of 64 samples over 256-column windows, which
// this replaces, needed compact tiles: a call with 256 samples of 3 detectors, 21 modes, 1001 bins at
// 16384 Hz took 2.2 ms, now 0.16 ms; 10,000 of 2 detectors and 9 modes 0.62 ms, now 0.22 ms.
// Eight samples a block, two blocks per SM: with sixteen, Q is read half as often, but the
// prologue's latency has one other block less to hide behind (5-8% slower).
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>

#include "ile_kernels.h"

namespace rift {

namespace {

constexpr int kLanesBins = 32;          // time bins per lane and chunk
constexpr int kChunkBins = 32 * kLanesBins;
constexpr int kPowStride = 16;          // >= kMaxPow + 1
constexpr int kFewSamples = 4, kSamples = 8;
static_assert(kPowStride >= kMaxPow + 1, "power table too short");
static_assert(kMaxModes <= 32 && kMaxDet * kSamples <= 64, "prologue items");

struct BlockLayout {
    size_t r, cs, trig, par, pw, fx, qpart, i0, f0, quad, gid, end;
};

__host__ __device__ inline size_t al16(size_t o) { return (o + 15) & ~(size_t)15; }

__host__ __device__ inline BlockLayout block_layout(int S, int K, int M, int wcap)
{
    BlockLayout L;
    size_t o = 0;
    L.r = o;     o = al16(o + (size_t)S * wcap * 4);
    L.cs = o;    o = al16(o + (size_t)K * 2 * M * S * 4);
    // per-sample tables are sample-minor ([row][S])
    L.trig = o;  o = al16(o + (size_t)4 * S * 8);                // sin, cos of h, of delta
    L.par = o;   o = al16(o + (size_t)6 * S * 4);                // c2psi, s2psi, cos, sin of iota/2, x, phi
    L.pw = o;    o = al16(o + (size_t)2 * kPowStride * S * 4);   // cos(i/2)^p, sin(i/2)^p
    L.fx = o;    o = al16(o + (size_t)K * S * 8);                // x F_k
    L.qpart = o; o = al16(o + (size_t)32 * S * 4);
    L.i0 = o;    o = al16(o + (size_t)K * S * 4);
    L.f0 = o;    o = al16(o + (size_t)K * S * 4);
    L.quad = o;  o = al16(o + (size_t)S * 4);
    L.gid = o;   o = al16(o + (size_t)S * 4);
    L.end = o;
    return L;
}

// Bins per chunk and columns of the R tile (a multiple of 4).
struct BlockPlan {
    int chunk, wcap;
};

BlockPlan block_plan(const Problem &P, int S, int64_t n, bool sorted, int max_smem)
{
    const double beta = P.t_step * P.fs;
    double span = 0.0;   // largest distance between two samples' windows at one detector
    for (int k = 0; k < P.K; ++k) {
        double r2 = 0.0;
        for (int i = 0; i < 3; ++i)
            r2 += P.xpos[k][i] * P.xpos[k][i];
        span = std::max(span, 2.0 * std::sqrt(r2) * P.fs);
    }
    // neighbours of a sorted batch share a patch of the sky; those that do not fit the
    // allowance are contracted in turn
    const double allow = sorted ? std::min(span, 16.0 + 4.0 * span * std::sqrt((double)S / (double)n)) : span;
    const int64_t room = ((int64_t)max_smem - 1024 - (int64_t)block_layout(S, P.K, P.M, 0).end) / (4 * S) / 4 * 4;
    BlockPlan B;
    const double bins = beta > 0.0 ? std::floor(((double)room - std::min(allow, 0.5 * (double)room) - 12.0) / beta) + 1.0
                                   : (double)kChunkBins;
    const int most = (int)std::max(1.0, std::min(bins, (double)kChunkBins));
    const int chunks = (P.n_t + most - 1) / most;
    B.chunk = (P.n_t + chunks - 1) / chunks;
    const double want = std::ceil((B.chunk - 1) * beta) + std::ceil(allow) + 12.0;
    B.wcap = ((int)std::min((double)room, want) + 3) / 4 * 4;
    if (B.wcap > room)
        B.wcap = (int)room;
    return B;
}

template <int S, bool kDM>
__global__ void __launch_bounds__(32 * S, 512 / (32 * S))
lnl_block_kernel(Problem P, BinTable bt, const double *__restrict__ theta, const uint32_t *__restrict__ perm, int64_t n,
                 int chunk, int wcap, double *__restrict__ lnL_tmarg, double *__restrict__ lnL_t,
                 const double *__restrict__ lnpw, double *__restrict__ lnw, int *err, PeakOut po)
{
    constexpr int kThreads = 32 * S;
    constexpr int kSG = S < 8 ? S : 8;                 // samples a thread contracts
    constexpr int kCG = kThreads / (S / kSG);          // column groups of four
    extern __shared__ __align__(16) unsigned char smraw[];
    const int K = P.K, M = P.M, R2 = 2 * M, NT = P.n_t;
    const BlockLayout L = block_layout(S, K, M, wcap);
    float *Rs = reinterpret_cast<float *>(smraw + L.r);          // [S][wcap]
    float *Cs = reinterpret_cast<float *>(smraw + L.cs);         // [K][2M][S]
    double *trig = reinterpret_cast<double *>(smraw + L.trig);
    float *par = reinterpret_cast<float *>(smraw + L.par);
    float *pw = reinterpret_cast<float *>(smraw + L.pw);
    float2 *fx = reinterpret_cast<float2 *>(smraw + L.fx);
    float *qpart = reinterpret_cast<float *>(smraw + L.qpart);   // [32][S]
    int *i0s = reinterpret_cast<int *>(smraw + L.i0);
    float *f0s = reinterpret_cast<float *>(smraw + L.f0);
    float *qds = reinterpret_cast<float *>(smraw + L.quad);
    uint32_t *gid = reinterpret_cast<uint32_t *>(smraw + L.gid);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s_of = tid % S, grp = tid / S;           // prologue items: sample, one of 32 groups

    // ---------------- prologue A: the five angles of a sample, a thread each (float64 for the
    // sky position, which the delays need)
    if (grp < 6) {
        const int64_t si = (int64_t)blockIdx.x * S + s_of;
        uint32_t g = si < n ? (perm ? perm[si] : (uint32_t)si) : 0xffffffffu;
        const bool valid = (int64_t)g < n;
        const double *th = theta + 6 * (int64_t)g;
        if (grp < 2) {
            const double a = !valid ? 0.0 : grp == 0 ? th[0] - P.gmst : th[1];
            double sn, cs;
            sincos(a, &sn, &cs);
            trig[(2 * grp) * S + s_of] = sn;
            trig[(2 * grp + 1) * S + s_of] = cs;
        } else if (grp < 4) {
            float sn, cs;
            sincosf(!valid ? 0.f : grp == 2 ? (float)(2.0 * th[2]) : (float)(0.5 * th[4]), &sn, &cs);
            par[(2 * grp - 4) * S + s_of] = cs;
            par[(2 * grp - 3) * S + s_of] = sn;
        } else if (grp == 4) {
            par[4 * S + s_of] = !valid ? 0.f : kDM ? 1.f : (float)P.d_ref / (float)th[5];
            par[5 * S + s_of] = valid ? (float)th[3] : 0.f;
        } else {
            gid[s_of] = valid ? g : 0xffffffffu;
        }
    }
    __syncthreads();
    // ---------------- B: delays and x F_k; powers of the half-angle functions
    if (grp < K) {
        const int k = grp;
        const double sh = trig[s_of], ch = trig[S + s_of], sd = trig[2 * S + s_of], cd = trig[3 * S + s_of];
        // Q-sample position of the first bin, (t_lo + dt_k - q_t0_k) fs
        const double u0 = fma(P.xfs[k][0], cd * ch, fma(P.xfs[k][1], cd * sh, fma(P.xfs[k][2], sd, P.ufs0[k])));
        // (of finite angles: the problem's Q window covers every sky position.  Other samples have
        // no Q index: they are flagged and take column 0, and no address is formed from them)
        const bool ok = isfinite(u0);
        if (!ok)
            atomicOr(err, kErrRange);
        const double fl = ok ? floor(u0) : 0.0;
        i0s[k * S + s_of] = (int)fl;
        f0s[k * S + s_of] = (float)(u0 - fl);
        const Cx<float> F = response_f(P.Dten_f[k], (float)(-sh), (float)ch, (float)(-sd * ch), (float)(-sd * sh),
                                       (float)cd, par[s_of], par[S + s_of]);
        const float amp = par[4 * S + s_of];
        fx[k * S + s_of] = make_float2(amp * F.re, amp * F.im);
    } else if (grp >= 8 && grp < 10) {
        const float x = par[(grp - 6) * S + s_of];   // cos, sin of iota/2
        float v = 1.f;
        for (int q = 0; q <= kMaxPow; ++q) {
            pw[((grp - 8) * kPowStride + q) * S + s_of] = v;
            v *= x;
        }
    }
    __syncthreads();
    // ---------------- C: harmonics and coefficients, a mode per group
    if (grp < M) {
        const int m = grp;
        float d = 0.f;
        for (int t = 0; t < P.wn[m]; ++t)
            d += P.wcoef_f[m][t] * pw[P.wpc[m][t] * S + s_of] * pw[(kPowStride + P.wps[m][t]) * S + s_of];
        float sy, cy;
        sincosf(-(float)P.mode_m[m] * par[5 * S + s_of], &sy, &cy);
        const float yr = d * cy, yi = d * sy;
        for (int k = 0; k < K; ++k) {
            const float2 f = fx[k * S + s_of];
            Cs[(k * R2 + 2 * m) * S + s_of] = f.x * yr - f.y * yi;
            Cs[(k * R2 + 2 * m + 1) * S + s_of] = f.x * yi + f.y * yr;
        }
    }
    __syncthreads();
    // ---------------- D: template term, row a of every detector per group, with U^H = U, V^T = V:
    //   c^H U c = sum_a [U_aa |c_a|^2 + 2 Re(conj(c_a) sum_{b>a} U_ab c_b)]
    //   c^T V c = sum_a [V_aa c_a^2   + 2 c_a sum_{b>a} V_ab c_b]
    {
        float acc = 0.f;
        const int a = grp;
        if (a < M)
            for (int k = 0; k < K; ++k) {
                const float *Ck = Cs + (size_t)k * R2 * S + s_of;
                const float2 *Ur = P.U32 + ((size_t)k * M + a) * M;
                const float2 *Vr = P.V32 + ((size_t)k * M + a) * M;
                const float ar = Ck[(2 * a) * S], ai = Ck[(2 * a + 1) * S];
                float ur = 0.f, ui = 0.f, vr = 0.f, vi = 0.f;
#pragma unroll 4
                for (int b = a + 1; b < M; ++b) {
                    const float cr = Ck[(2 * b) * S], ci = Ck[(2 * b + 1) * S];
                    const float2 u = __ldg(Ur + b), v = __ldg(Vr + b);
                    ur = fmaf(u.x, cr, fmaf(-u.y, ci, ur));
                    ui = fmaf(u.x, ci, fmaf(u.y, cr, ui));
                    vr = fmaf(v.x, cr, fmaf(-v.y, ci, vr));
                    vi = fmaf(v.x, ci, fmaf(v.y, cr, vi));
                }
                const float2 ud = __ldg(Ur + a), vd = __ldg(Vr + a);
                const float a2r = ar * ar - ai * ai, a2i = 2.f * ar * ai;
                acc += ud.x * (ar * ar + ai * ai) + 2.f * (ar * ur + ai * ui);
                acc += (vd.x * a2r - vd.y * a2i) + 2.f * (ar * vr - ai * vi);
            }
        qpart[grp * S + s_of] = acc;
    }
    __syncthreads();
    if (grp == 0) {
        float q = 0.f;
        for (int a = 0; a < M; ++a)
            q += qpart[a * S + s_of];
        qds[s_of] = (float)P.kappa * q;
    }
    __syncthreads();

    // ---------------- the sample of this warp
    const uint32_t g = gid[warp];
    const float qd = qds[warp];
    unsigned valid = 0;   // samples of the block
#pragma unroll
    for (int s = 0; s < S; ++s)
        valid |= gid[s] != 0xffffffffu ? 1u << s : 0u;
    const int sg = (tid / kCG) * kSG, cg = tid % kCG;
    float run_mx = -INFINITY, run_sum = 0.f;
    int run_j = 0;
    for (int j0 = 0; j0 < NT; j0 += chunk) {
        const int J = min(chunk, NT - j0), jl = j0 + J - 1;
        float lin[kLanesBins];
#pragma unroll
        for (int q = 0; q < kLanesBins; ++q)
            lin[q] = 0.f;
        const int b0 = __ldg(bt.bin_i + j0), span = __ldg(bt.bin_i + jl) - b0 + 3;   // columns of one sample
        for (int k = 0; k < K; ++k) {
            const float *Qk = P.Qr32 + (size_t)k * R2 * P.n_q_pad;
            const float *Ck = Cs + (size_t)k * R2 * S + sg;
            for (unsigned rem = valid; rem;) {
                // the samples whose windows fit the R tile from the lowest one on
                int lo = INT_MAX, hi = INT_MIN;
#pragma unroll
                for (int s = 0; s < S; ++s)
                    if ((rem >> s) & 1u)
                        lo = min(lo, i0s[k * S + s]);
                const int base = max(lo + b0, 0) & ~3;
                unsigned now = 0;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const int i0 = i0s[k * S + s];
                    if (((rem >> s) & 1u) && i0 + b0 - base + span <= wcap) {
                        now |= 1u << s;
                        hi = max(hi, i0);
                    }
                }
                if (!now) {   // cannot be: a single window fits by the choice of the chunk
                    if (tid == 0)
                        atomicOr(err, kErrRange);
                    break;
                }
                rem &= ~now;
                const int ncols = hi + b0 - base + span;
                for (int c = 4 * cg; c < ncols; c += 4 * kCG) {
                    const float *q = Qk + base + c;
                    float2 acc[4][kSG / 2];   // columns, pairs of samples
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int p = 0; p < kSG / 2; ++p)
                            acc[i][p] = make_float2(0.f, 0.f);
#pragma unroll 2
                    for (int r = 0; r < R2; ++r) {
                        const float4 qv = __ldg(reinterpret_cast<const float4 *>(q + (size_t)r * P.n_q_pad));
                        const float qa[4] = {qv.x, qv.y, qv.z, qv.w};
                        float2 cv[kSG / 2];
#pragma unroll
                        for (int p = 0; p < kSG / 4; ++p) {
                            const float4 x = *reinterpret_cast<const float4 *>(Ck + r * S + 4 * p);
                            cv[2 * p] = make_float2(x.x, x.y);
                            cv[2 * p + 1] = make_float2(x.z, x.w);
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int p = 0; p < kSG / 2; ++p)
                                acc[i][p] = __ffma2_rn(make_float2(qa[i], qa[i]), cv[p], acc[i][p]);
                    }
#pragma unroll
                    for (int p = 0; p < kSG / 2; ++p) {
                        float *out = Rs + (size_t)(sg + 2 * p) * wcap + c;
                        *reinterpret_cast<float4 *>(out) = make_float4(acc[0][p].x, acc[1][p].x, acc[2][p].x, acc[3][p].x);
                        *reinterpret_cast<float4 *>(out + wcap) =
                            make_float4(acc[0][p].y, acc[1][p].y, acc[2][p].y, acc[3][p].y);
                    }
                }
                __syncthreads();   // R complete
                if ((now >> warp) & 1u) {
                    const float *row = Rs + (size_t)warp * wcap + (i0s[k * S + warp] - base);
                    const float f0 = f0s[k * S + warp];
#pragma unroll
                    for (int q0 = 0; q0 < kLanesBins; q0 += 4)
                        if (32 * q0 < J) {   // (uniform)
#pragma unroll
                            for (int q = q0; q < q0 + 4; ++q) {
                                const int j = min(j0 + lane + 32 * q, jl);
                                const float sf = f0 + __ldg(bt.bin_f + j);
                                const int carry = sf >= 1.f;
                                const float fr = sf - (float)carry;
                                const float *rr = row + __ldg(bt.bin_i + j) + carry;
                                const float r0 = rr[0], r1 = rr[1];
                                lin[q] += fmaf(fr, r1 - r0, r0);
                            }
                        }
                }
                __syncthreads();   // R read
            }
        }
        if (g == 0xffffffffu)
            continue;
        // ---- fold the chunk (of the data term alone: the template term enters at the end)
        const int jv = J - lane;   // bin 32 q + lane exists: 32 q < jv
        float cmx = -INFINITY;
        if (kDM) {
            // distance marginal per bin: upper bounds first; the bin with the highest bound is
            // evaluated (by the lane holding it), and bins whose bound lies more than 40 below
            // the larger of that value and the running maximum cannot move the marginal (< e^-40):
            // left out
            float bl = -INFINITY, al = 0.f;
#pragma unroll
            for (int q = 0; q < kLanesBins; ++q) {
                const float b = 32 * q < jv ? dm_bound32(P, lin[q], qd) : -INFINITY;
                if (b > bl) {
                    bl = b;
                    al = lin[q];
                }
            }
            float bmax = bl;
#pragma unroll
            for (int o = 16; o; o >>= 1)
                bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
            const unsigned holds = __ballot_sync(0xffffffffu, bl == bmax);
            const int owner = holds ? __ffs(holds) - 1 : 0;
            float vbest = -INFINITY;
            if (lane == owner && bmax > -INFINITY)
                vbest = ln_dist_marg32(P, al, qd);
            vbest = __shfl_sync(0xffffffffu, vbest, owner);
            const float thr = lnL_t ? -INFINITY : fmaxf(run_mx, vbest) - 40.f;
            unsigned need = 0;
#pragma unroll
            for (int q = 0; q < kLanesBins; ++q) {
                if (32 * q < jv && dm_bound32(P, lin[q], qd) >= thr)
                    need |= 1u << q;
                else
                    lin[q] = -INFINITY;
            }
            // one copy of the quadrature, its bin picked from and put back to its register by
            // selects
            for (unsigned any = __reduce_or_sync(0xffffffffu, need); any; any &= any - 1u) {
                const int q = __ffs(any) - 1;
                float x = -INFINITY;
#pragma unroll
                for (int u = 0; u < kLanesBins; ++u)
                    x = u == q ? lin[u] : x;
                if ((need >> q) & 1u)
                    x = ln_dist_marg32(P, x, qd);
                cmx = fmaxf(cmx, x);
#pragma unroll
                for (int u = 0; u < kLanesBins; ++u)
                    lin[u] = u == q ? x : lin[u];
            }
        } else {
#pragma unroll
            for (int q = 0; q < kLanesBins; ++q)
                if (32 * q < jv)
                    cmx = fmaxf(cmx, lin[q]);
        }
        if (lnL_t)
#pragma unroll
            for (int q = 0; q < kLanesBins; ++q)
                if (32 * q < jv)
                    lnL_t[(int64_t)g * NT + j0 + lane + 32 * q] = kDM ? (double)lin[q] : (double)lin[q] - (double)qd;
#pragma unroll
        for (int o = 16; o; o >>= 1)
            cmx = fmaxf(cmx, __shfl_xor_sync(0xffffffffu, cmx, o));
        if (cmx > run_mx) {   // a new running maximum: its bin, the lowest holding it
            int jc = INT_MAX;
#pragma unroll
            for (int q = 0; q < kLanesBins; ++q)
                if (32 * q < jv && lin[q] == cmx)
                    jc = min(jc, j0 + lane + 32 * q);
            run_j = __reduce_min_sync(0xffffffffu, jc);
        }
        const float nm = fmaxf(run_mx, cmx);
        float cs = 0.f;
#pragma unroll
        for (int q = 0; q < kLanesBins; ++q)
            if (32 * q < jv)
                cs += __expf(lin[q] - nm);
#pragma unroll
        for (int o = 16; o; o >>= 1)
            cs += __shfl_xor_sync(0xffffffffu, cs, o);
        run_sum = (run_mx == -INFINITY ? 0.f : run_sum * __expf(run_mx - nm)) + cs;
        run_mx = nm;
    }
    if (lane == 0 && g != 0xffffffffu) {
        // the log-sum-exp in float32 like the terms (run_sum >= 1); the template term
        // subtracted in float64, so that the difference of two large terms is not rounded to
        // float32
        const double r = (double)run_mx + (double)__logf(run_sum) - (kDM ? 0.0 : (double)qd) - bt.ln_nt;
        if (!kDM && po.q) {
            po.q[g] = qd;
            po.m[g] = run_mx;
            po.j[g] = run_j;
        }
        if (!isfinite(r))
            atomicOr(err, kErrNonFinite);
        lnL_tmarg[g] = r;
        if (lnw && lnpw)
            lnw[g] = r + lnpw[g];
    }
}

}  // namespace

cudaError_t launch_lnl_fp32(const Problem &P, BinTable bt, const double *theta, const uint32_t *perm, int64_t n,
                            double *lnL_tmarg, double *lnL_t, const double *lnpw, double *lnw, int *err,
                            cudaStream_t st, PeakOut po)
{
    if (n <= 0)
        return cudaSuccess;
    int dev = 0, sms = 0, max_smem = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    // four samples a block while eight would leave SMs without one
    const bool few = n <= (int64_t)kSamples * sms;
    const int S = few ? kFewSamples : kSamples;
    const BlockPlan B = block_plan(P, S, n, perm != nullptr, max_smem);
    const size_t smem = block_layout(S, P.K, P.M, B.wcap).end;
    if (B.wcap < 16 || smem > (size_t)max_smem)
        return cudaErrorInvalidConfiguration;
    auto kern = few ? (P.dist_marg ? lnl_block_kernel<kFewSamples, true> : lnl_block_kernel<kFewSamples, false>)
                    : (P.dist_marg ? lnl_block_kernel<kSamples, true> : lnl_block_kernel<kSamples, false>);
    cudaError_t e = allow_max_dynamic_smem(kern);
    if (e != cudaSuccess)
        return e;
    kern<<<(unsigned)((n + S - 1) / S), 32 * S, smem, st>>>(P, bt, theta, perm, n, B.chunk, B.wcap, lnL_tmarg, lnL_t,
                                                           lnpw, lnw, err, po);
    return cudaGetLastError();
}

cudaError_t prepare_tile_kernels()
{
    cudaError_t e = allow_max_dynamic_smem(lnl_block_kernel<kFewSamples, false>);
    if (e == cudaSuccess)
        e = allow_max_dynamic_smem(lnl_block_kernel<kFewSamples, true>);
    if (e == cudaSuccess)
        e = allow_max_dynamic_smem(lnl_block_kernel<kSamples, false>);
    return e != cudaSuccess ? e : allow_max_dynamic_smem(lnl_block_kernel<kSamples, true>);
}

}  // namespace rift
