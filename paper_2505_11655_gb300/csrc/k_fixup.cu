// Large-term correction of the float32 likelihood path.
//
// ln L_j = lin_j - quad is the difference of the data term and the template term of
// arXiv:2505.11655 Eq. (def:lnL:Decomposed).  For a sample near the lower distance bound
// both terms reach 1e3..1e4 while their difference is a large negative number, and float32
// rounding of the coefficients c_k,lm = (D_ref/D) F_k Y_lm and of the template term moves
// ln L by ~3e-7 (|lnL| + 2 quad): up to ~1e-2.  Nearly all of that error is common to
// every time bin of the sample (the template term, and the scale of the coefficients), so
// it is removed per sample rather than per bin:
//
//   1. the float32 kernel writes, beside ln L_tmarg = LSE_j(lin_j) - quad32 - ln n_t (the
//      difference taken in float64), the float32 template term quad32, the largest float32
//      data term m32 and a block of bins holding the bin of m32;
//   2. samples with quad32 + |m32| above a threshold (the float32 error can exceed the
//      parity bar there) are listed;
//   3. for each listed sample, with the coefficients from float64 geometry:
//        the template term in double-float (~44 bits), written through the symmetry of
//        U (Hermitian) and the form Y_lm = d_lm(iota) exp(-i m phi):
//          c^H U_k c = |s_k|^2 sum_D exp(i D phi) G_k,D,  G_k,D = sum_{m_a - m_b = D} d_a d_b U_k,ab
//          c^T V_k c = s_k^2  sum_S exp(-i S phi) H_k,S,  H_k,S = sum_{m_a + m_b = S} d_a d_b V_k,ab
//        with s_k = (D_ref/D) F_k.  The d_lm are trigonometric polynomials of degree l in iota,
//        so every G_k,D and H_k,S is one of degree 2 l_max, in cosines for even D, S and in
//        sines for odd; their coefficients are summed once per problem in float64 (21 modes up
//        to l = 4: 9 x 9 + 17 x 9 complex coefficients a detector in place of 2 x 231 mode pairs
//        with a product d_a d_b each: a loud solve's 250,000 corrections 1.07 -> 0.79 ms);
//        the bin of the block with the largest data term (a float32 search when the block
//        holds several bins), and the data term there in double-float, from a double-float
//        copy of Q;
//      and ln L_tmarg moves by (quad32 - quad) + (lin(j*) - m32): the error of the float32
//      data term is the same at every bin near the maximum (a scale error of the
//      coefficients), and the bins far below it do not move the log-sum-exp.
// The per-bin values (when requested) move by the same amount.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>

#include "df.cuh"
#include "ile_kernels.h"

namespace rift {

constexpr int kFixMaxWarps = 16;   // warps per block: as many as the shared memory holds, up to this

// --------------------------------------------------------------- double-float copies

__device__ __forceinline__ float4 df4(double re, double im)
{
    const df a = df_of(re), b = df_of(im);
    return make_float4(a.hi, a.lo, b.hi, b.lo);
}

__global__ void fix_prep_q_kernel(const double2 *__restrict__ Q64, int64_t nq, float4 *__restrict__ qdf)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nq; e += (int64_t)gridDim.x * blockDim.x) {
        const double2 v = Q64[e];
        qdf[e] = df4(v.x, v.y);
    }
}

// Coefficient n of the product of two polar functions with Fourier coefficients A, B (sine
// series where odd): cosines of n iota when both or neither are odd, else sines.
__device__ __forceinline__ double product_coef(const double *A, bool odd_a, const double *B, bool odd_b, int n)
{
    double v = 0.0;
    for (int u = 0; u <= kMaxL; ++u) {
        const int sum = n - u, lower = u - n, upper = u + n;   // partners with u + w = n, u - w = n, w - u = n
        double t = 0.0;
        if (sum >= 0 && sum <= kMaxL)
            t += odd_a && odd_b ? -B[sum] : B[sum];
        if (lower >= 0)
            t += !odd_a && odd_b ? -B[lower] : B[lower];
        if (n > 0 && upper <= kMaxL)
            t += odd_a && !odd_b ? -B[upper] : B[upper];
        v += A[u] * t;
    }
    return 0.5 * v;
}

// One warp per (detector, D or S, n).
__global__ void fix_prep_template_kernel(Problem P, FixTables T)
{
    const int lane = threadIdx.x & 31, M = P.M, na = T.dmax + 1, ns = 2 * T.dmax + 1;
    const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), per = (na + ns) * T.nf;
    if (e >= P.K * per)
        return;
    const int k = e / per, row = (e - k * per) / T.nf, n = e - k * per - row * T.nf;
    const bool u_term = row < na;
    const int want = u_term ? row : row - na - T.dmax;   // D or S
    const double2 *G = (u_term ? P.U64 : P.V64) + (size_t)k * M * M;
    double re = 0.0, im = 0.0;
    for (int p = lane; p < M * M; p += 32) {
        const int a = p / M, b = p - a * M, ma = P.mode_m[a], mb = P.mode_m[b];
        if ((u_term ? ma - mb : ma + mb) != want)
            continue;
        const double c = product_coef(T.alpha + a * (kMaxL + 1), ma & 1, T.alpha + b * (kMaxL + 1), mb & 1, n);
        const double2 g = G[p];
        re += c * g.x;
        im += c * g.y;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (lane == 0) {
        if (u_term)
            T.ga[((size_t)k * na + row) * T.nf + n] = df4(re, im);
        else
            T.hb[((size_t)k * ns + row - na) * T.nf + n] = df4(re, im);
    }
}

// --------------------------------------------------------------- selection

__global__ void fix_select_kernel(const float *__restrict__ aq, const float *__restrict__ am, int64_t n, float thr,
                                  uint32_t *__restrict__ idx, uint32_t *__restrict__ count)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool take = false;
    if (i < n)
        take = aq[i] + fabsf(am[i]) > thr;   // a non-finite value is flagged by the kernel that wrote it
    const unsigned mask = __ballot_sync(0xffffffffu, take);
    if (!mask)
        return;
    const int lane = threadIdx.x & 31, leader = __ffs(mask) - 1;
    uint32_t base = 0;
    if (lane == leader)
        base = atomicAdd(count, (uint32_t)__popc(mask));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (take)
        idx[base + __popc(mask & ((1u << lane) - 1u))] = (uint32_t)i;
}

// --------------------------------------------------------------- correction

// Per-warp shared memory: float64 rows [K + 1][32] (the Q position u0_k of the first bin,
// then the template term), float rows [..][32] (double-float s_k, d_lm, exp(-i n phi), cos and
// sin of n iota), and [32] the bin at which each sample's data term is evaluated.
__host__ __device__ inline int fix_float_rows(int K, int M, int dmax, int nf)
{
    return 4 * K + 2 * M + 4 * (dmax + 1) + 4 * nf;
}

__host__ __device__ inline size_t fix_warp_bytes(int K, int M, int dmax, int nf)
{
    return (size_t)(K + 1) * 32 * 8 + (size_t)fix_float_rows(K, M, dmax, nf) * 32 * 4 + 32 * 4;
}

__global__ void __launch_bounds__(32 * kFixMaxWarps)
fix_kernel(Problem P, BinTable bt, FixTables T, const double *__restrict__ theta, const uint32_t *__restrict__ idx,
           const uint32_t *__restrict__ count, PeakOut po, int blen, double *__restrict__ lnL_tmarg,
           double *__restrict__ lnL_t, const double *__restrict__ lnpw, double *__restrict__ lnw, int *err)
{
    extern __shared__ __align__(16) unsigned char fsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int K = P.K, M = P.M, NT = P.n_t;
    const int nph = T.dmax + 1;
    unsigned char *wb = fsm + fix_warp_bytes(K, M, T.dmax, T.nf) * warp;
    double *rd = reinterpret_cast<double *>(wb);                 // [K + 1][32]
    float *rf = reinterpret_cast<float *>(rd + (K + 1) * 32);     // [nf][32]
    float *c32 = rf + fix_float_rows(K, M, T.dmax, T.nf) * 32;
    // rows of rf: s_k (re.hi, re.lo, im.hi, im.lo) at 4k; d_lm (hi, lo) at 4K + 2m;
    // exp(-i n phi) (re.hi, re.lo, im.hi, im.lo) at 4K + 2M + 4n; cos(n iota) (hi, lo), then sin
    const int rs = 0, rdl = 4 * K, rph = 4 * K + 2 * M, rtr = rph + 4 * nph, NF = T.nf;
    const double beta = P.t_step * P.fs;
    const uint32_t cnt = *count;
    const int nw = (int)(blockDim.x >> 5);
    // A lane corrects a sample of its own, or eight lanes share one when the list fits the grid
    // that way: they split the angles, detectors, modes and azimuthal orders, and a short list
    // takes the latency of a few of these instead of all (256 samples of the plain problem 45 us,
    // now 28).
    const int gsh = (int64_t)cnt <= (int64_t)gridDim.x * nw * 4 ? 3 : 0, G = 1 << gsh, spw = 32 >> gsh;
    const int col = lane >> gsh, sub = lane & (G - 1);
    // batch b of spw listed samples goes to block b % gridDim.x, warp b / gridDim.x (round
    // robin over the blocks first, so that a short list still spreads over every SM)
    if ((int64_t)blockIdx.x * spw >= (int64_t)cnt)
        return;   // no listed sample for this block (the grid is sized for every sample)
    // the template coefficients of every detector, staged once per block
    const int na = nph, ns = 2 * T.dmax + 1;
    float4 *sga = reinterpret_cast<float4 *>(fsm + fix_warp_bytes(K, M, T.dmax, T.nf) * nw);
    float4 *shb = sga + K * na * NF;
    for (int e = threadIdx.x; e < K * na * NF; e += blockDim.x)
        sga[e] = T.ga[e];
    for (int e = threadIdx.x; e < K * ns * NF; e += blockDim.x)
        shb[e] = T.hb[e];
    __syncthreads();
    // this lane's sample: the double-float value at rows (row, row + 1)
    auto ld = [&](int row) { return df{rf[row * 32 + col], rf[(row + 1) * 32 + col]}; };
    // (the lanes of a sample write the same value, or each its own row)
    auto put = [&](int row, df d) {
        rf[row * 32 + col] = d.hi;
        rf[(row + 1) * 32 + col] = d.lo;
    };
    // sums over the lanes of a sample
    auto join = [&](df v) {
        for (int o = 1; o < G; o <<= 1)
            v = df_add(v, df_shfl_xor(v, o));
        return v;
    };

    for (int64_t base = ((int64_t)warp * gridDim.x + blockIdx.x) * spw; base < (int64_t)cnt;
         base += (int64_t)gridDim.x * nw * spw) {
        const int64_t e = base + col;
        const bool active = e < (int64_t)cnt;
        const uint32_t g = active ? idx[e] : 0u;

        // ---- phase A: geometry in float64, rounded to double-float
        {
            double th[6] = {0.0, 0.0, 0.0, 0.0, 0.0, P.d_ref};   // inert values on idle lanes
            if (active)
                for (int d = 0; d < 6; ++d)
                    th[d] = theta[6 * (int64_t)g + d];
            Sky sky;
            double s2p, c2p, si, ci, sp, cp;
            if (G == 1) {
                sky = sky_of(th[0], th[1], P.gmst);
                sincos(2.0 * th[2], &s2p, &c2p);
                sincos(th[4], &si, &ci);
                sincos(th[3], &sp, &cp);
            } else {   // an angle per lane
                double sn, cs;
                sincos(sub == 0 ? th[1] : sub == 1 ? th[0] - P.gmst : sub == 2 ? 2.0 * th[2] : sub == 3 ? th[4] : th[3], &sn, &cs);
                const int l0 = lane & ~7;
                sky.sd = __shfl_sync(0xffffffffu, sn, l0);
                sky.cd = __shfl_sync(0xffffffffu, cs, l0);
                sky.sh = __shfl_sync(0xffffffffu, sn, l0 + 1);
                sky.ch = __shfl_sync(0xffffffffu, cs, l0 + 1);
                s2p = __shfl_sync(0xffffffffu, sn, l0 + 2);
                c2p = __shfl_sync(0xffffffffu, cs, l0 + 2);
                si = __shfl_sync(0xffffffffu, sn, l0 + 3);
                ci = __shfl_sync(0xffffffffu, cs, l0 + 3);
                sp = __shfl_sync(0xffffffffu, sn, l0 + 4);
                cp = __shfl_sync(0xffffffffu, cs, l0 + 4);
            }
            const double n0 = sky.cd * sky.ch, n1 = sky.cd * sky.sh, n2 = sky.sd;
            const double x = P.d_ref / th[5];
            for (int k = sub; k < K; k += G) {
                rd[k * 32 + col] = fma(P.xfs[k][0], n0, fma(P.xfs[k][1], n1, fma(P.xfs[k][2], n2, P.ufs0[k])));
                const Cx<double> F = response<double>(P, k, sky, c2p, s2p);
                put(rs + 4 * k, df_of(x * F.re));
                put(rs + 4 * k + 2, df_of(x * F.im));
            }
            // cos and sin of n iota by powers of exp(i iota), exp(-i n phi), and the polar functions
            // from their Fourier coefficients, in double-float (in float64, with a conversion per
            // value, they were half of the kernel's float64 operations; the corrected values' rms
            // errors, 1.7e-5 to 1.2e-4 at SNR 40 and 150, are the same to five digits, nearly
            // face-on and face-off samples included)
            dfc r{{1.f, 0.f}, {0.f, 0.f}};
            const dfc r1{df_of(ci), df_of(si)};
            for (int nn = 0; nn < NF; ++nn) {
                put(rtr + 2 * nn, r.re);
                put(rtr + 2 * NF + 2 * nn, r.im);
                r = dfc_mul(r, r1);
            }
            r = {{1.f, 0.f}, {0.f, 0.f}};
            const dfc e1{df_of(cp), df_of(-sp)};
            for (int nn = 0; nn < nph; ++nn) {
                put(rph + 4 * nn, r.re);
                put(rph + 4 * nn + 2, r.im);
                r = dfc_mul(r, e1);
            }
            __syncwarp();
            for (int m = sub; m < M; m += G) {
                const float2 *al = T.alpha32 + m * (kMaxL + 1);
                const int tb = rtr + ((P.mode_m[m] & 1) ? 2 * NF : 0);
                df d{0.f, 0.f};
#pragma unroll
                for (int u = 0; u <= kMaxL; ++u)
                    if (2 * u < NF)
                        df_acc(d, ld(tb + 2 * u), {al[u].x, al[u].y});
                put(rdl + 2 * m, df_norm(d));
            }
        }
        __syncwarp();

        // ---- the template term in double-float
        {
            df A[kMaxDet];
            dfc B[kMaxDet];
#pragma unroll
            for (int k = 0; k < kMaxDet; ++k) {
                A[k] = {0.f, 0.f};
                B[k] = {{0.f, 0.f}, {0.f, 0.f}};
            }
            for (int D = sub; D <= T.dmax; D += G) {
                dfc G[kMaxDet];
#pragma unroll
                for (int k = 0; k < kMaxDet; ++k)
                    G[k] = {{0.f, 0.f}, {0.f, 0.f}};
                const int tb = rtr + ((D & 1) ? 2 * NF : 0);
#pragma unroll 3
                for (int n = D & 1; n < NF; ++n) {
                    const df t = ld(tb + 2 * n);
#pragma unroll
                    for (int k = 0; k < kMaxDet; ++k)
                        if (k < K) {
                            const float4 u = sga[(k * na + D) * NF + n];
                            df_acc(G[k].re, t, {u.x, u.y});
                            df_acc(G[k].im, t, {u.z, u.w});
                        }
                }
#pragma unroll
                for (int k = 0; k < kMaxDet; ++k)
                    G[k] = {df_norm(G[k].re), df_norm(G[k].im)};
                // A_k += G_0, or 2 Re(exp(i D phi) G_D) = 2 (Re e Re G + Im e Im G), e = exp(-i D phi)
                const df er = ld(rph + 4 * D), ei = ld(rph + 4 * D + 2);
#pragma unroll
                for (int k = 0; k < kMaxDet; ++k)
                    if (k < K) {
                        if (D == 0) {
                            A[k] = df_add(A[k], G[k].re);
                        } else {
                            const df t = df_add(df_mul(er, G[k].re), df_mul(ei, G[k].im));
                            A[k] = df_add(A[k], df_add(t, t));
                        }
                    }
            }
            for (int S = sub - T.dmax; S <= T.dmax; S += G) {
                dfc H[kMaxDet];
#pragma unroll
                for (int k = 0; k < kMaxDet; ++k)
                    H[k] = {{0.f, 0.f}, {0.f, 0.f}};
                const int tb = rtr + ((S & 1) ? 2 * NF : 0);
#pragma unroll 3
                for (int n = S & 1; n < NF; ++n) {
                    const df t = ld(tb + 2 * n);
#pragma unroll
                    for (int k = 0; k < kMaxDet; ++k)
                        if (k < K) {
                            const float4 v = shb[(k * ns + S + T.dmax) * NF + n];
                            df_acc(H[k].re, t, {v.x, v.y});
                            df_acc(H[k].im, t, {v.z, v.w});
                        }
                }
#pragma unroll
                for (int k = 0; k < kMaxDet; ++k)
                    H[k] = {df_norm(H[k].re), df_norm(H[k].im)};
                // exp(-i S phi): the table entry for S >= 0, its conjugate for S < 0
                const int a = S < 0 ? -S : S;
                dfc e{ld(rph + 4 * a), ld(rph + 4 * a + 2)};
                if (S < 0)
                    e.im = {-e.im.hi, -e.im.lo};
#pragma unroll
                for (int k = 0; k < kMaxDet; ++k)
                    if (k < K) {
                        const dfc t = dfc_mul(e, H[k]);
                        B[k].re = df_add(B[k].re, t.re);
                        B[k].im = df_add(B[k].im, t.im);
                    }
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < kMaxDet; ++k)
                if (k < K) {
                    A[k] = join(A[k]);
                    B[k] = {join(B[k].re), join(B[k].im)};
                }
            // quad = kappa sum_k |s_k|^2 A_k + Re(s_k^2 B_k)
            df q = {0.f, 0.f};
#pragma unroll
            for (int k = 0; k < kMaxDet; ++k)
                if (k < K) {
                    const df sr = ld(rs + 4 * k), si = ld(rs + 4 * k + 2);
                    const df rr = df_mul(sr, sr), ii = df_mul(si, si), ri = df_mul(sr, si);
                    const df abs2 = df_add(rr, ii), s2r = df_sub(rr, ii), s2i = df_add(ri, ri);
                    q = df_add(q, df_mul(abs2, A[k]));
                    q = df_add(q, df_sub(df_mul(s2r, B[k].re), df_mul(s2i, B[k].im)));
                }
            rd[K * 32 + col] = P.kappa * df_to_double(q);
        }
        __syncwarp();

        // ---- phase B: the bin of the largest data term in the kernel's block (float32
        // search; lanes = (sample, bin of the block) pairs), then the data term there in
        // double-float, one sample per lane
        const int nb = (int)((int64_t)cnt - base < spw ? (int64_t)cnt - base : spw);
        int *jbest = reinterpret_cast<int *>(c32);   // [32] the bin each sample is evaluated at
        if (blen <= 1) {
            if (col < nb && sub == 0)
                jbest[col] = po.j[g];
        } else {
            int lps = 1;   // lanes per sample: the block length rounded up to a power of two
            while (lps < blen)
                lps <<= 1;
            const int spr = 32 / lps;   // samples per round
            for (int r0 = 0; r0 < nb; r0 += spr) {
                const int t = r0 + lane / lps, b = lane % lps;
                const uint32_t gt = __shfl_sync(0xffffffffu, g, (t << gsh) & 31);
                float best = -INFINITY;
                int bj = INT_MAX;
                if (t < nb && b < blen) {
                    const int jb = po.j[gt], j = jb + b;
                    if (jb >= 0 && j < NT) {
                        float lin = 0.f;
                        bool ok = true;
                        for (int k = 0; k < K && ok; ++k) {
                            const double u0 = rd[k * 32 + t];
                            const double fl = floor(u0);
                            const float sf = (float)(u0 - fl) + bt.bin_f[j];
                            const int carry = sf >= 1.f;
                            const float fr = sf - (float)carry;
                            const int c = (int)fl + bt.bin_i[j] + carry;
                            if (c < 0 || c + 1 >= P.n_q) {
                                ok = false;
                                break;
                            }
                            const float sr = rf[(rs + 4 * k) * 32 + t], si = rf[(rs + 4 * k + 2) * 32 + t];
                            const float *Qk = P.Qr32 + (size_t)k * 2 * M * P.n_q_pad + c;
#pragma unroll 7
                            for (int m = 0; m < M; ++m) {
                                const int mm = P.mode_m[m], a = mm < 0 ? -mm : mm;
                                const float d = rf[(rdl + 2 * m) * 32 + t];
                                const float er = rf[(rph + 4 * a) * 32 + t];
                                const float ei = mm < 0 ? -rf[(rph + 4 * a + 2) * 32 + t] : rf[(rph + 4 * a + 2) * 32 + t];
                                const float yr = d * er, yi = d * ei;
                                const float cr = sr * yr - si * yi, ci = sr * yi + si * yr;
                                const float *qr = Qk + (size_t)(2 * m) * P.n_q_pad, *qi = qr + P.n_q_pad;
                                const float vr = fmaf(fr, qr[1] - qr[0], qr[0]), vi = fmaf(fr, qi[1] - qi[0], qi[0]);
                                lin = fmaf(cr, vr, fmaf(ci, vi, lin));
                            }
                        }
                        if (ok) {
                            best = lin;
                            bj = j;
                        }
                    }
                }
                // the largest value of the sample's bins, the lowest bin among equals
                for (int o = 1; o < lps; o <<= 1) {
                    const float ov = __shfl_xor_sync(0xffffffffu, best, o);
                    const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
                    if (ov > best || (ov == best && oj < bj)) {
                        best = ov;
                        bj = oj;
                    }
                }
                if (b == 0 && t < nb)
                    jbest[t] = bj;
            }
        }
        __syncwarp();
        double corr = 0.0;
        bool good = false;
        {
            const int j = col < nb ? jbest[col] : INT_MAX;
            dfc w[kMaxDet];
#pragma unroll
            for (int k = 0; k < kMaxDet; ++k)
                w[k] = {{0.f, 0.f}, {0.f, 0.f}};
            if (j != INT_MAX) {
                // lin = sum_k Re(conj(s_k) sum_m conj(Y_m) Q_k,m), Q interpolated at the bin
                good = true;
                df f[kMaxDet];
                int i[kMaxDet];
#pragma unroll
                for (int k = 0; k < kMaxDet; ++k) {
                    f[k] = {0.f, 0.f};
                    i[k] = 0;
                    if (k < K) {
                        const double u = rd[k * 32 + col] + (double)j * beta;
                        const double fl = floor(u);
                        if (!(fl >= 0.0) || fl + 1.0 > (double)(P.n_q - 1)) {
                            good = false;
                        } else {
                            i[k] = (int)fl;
                            f[k] = df_of(u - fl);
                        }
                    }
                }
                for (int m = sub; m < M && good; m += G) {
                    // Y_lm = d_lm exp(-i m phi): the table entry for m >= 0, its conjugate for m < 0
                    const int mm = P.mode_m[m], a = mm < 0 ? -mm : mm;
                    const df d = ld(rdl + 2 * m);
                    df yi = df_mul(d, ld(rph + 4 * a + 2));
                    const df yr = df_mul(d, ld(rph + 4 * a));
                    if (mm < 0)
                        yi = {-yi.hi, -yi.lo};
#pragma unroll
                    for (int k = 0; k < kMaxDet; ++k)
                        if (k < K) {
                            const float4 *qk = T.qdf + ((size_t)k * M + m) * P.n_q + i[k];
                            const float4 q0 = qk[0], q1 = qk[1];
                            const df r0{q0.x, q0.y}, r1{q1.x, q1.y}, i0{q0.z, q0.w}, i1{q1.z, q1.w};
                            const df qre = df_add(r0, df_mul(f[k], df_sub(r1, r0)));
                            const df qim = df_add(i0, df_mul(f[k], df_sub(i1, i0)));
                            df_acc(w[k].re, yr, qre);
                            df_acc(w[k].re, yi, qim);
                            df_acc(w[k].im, yr, qim);
                            df_acc(w[k].im, {-yi.hi, -yi.lo}, qre);
                        }
                }
            }
            __syncwarp();
            df acc = {0.f, 0.f};
#pragma unroll
            for (int k = 0; k < kMaxDet; ++k)
                if (k < K)
                    acc = df_add(acc, df_add(df_mul(ld(rs + 4 * k), join(df_norm(w[k].re))),
                                             df_mul(ld(rs + 4 * k + 2), join(df_norm(w[k].im)))));
            if (good)
                corr = ((double)po.q[g] - rd[K * 32 + col]) + (df_to_double(acc) - (double)po.m[g]);
            if (col < nb && !good) {
                atomicOr(err, kErrRange);
            } else if (col < nb && sub == 0) {
                const double r = lnL_tmarg[g] + corr;
                if (!isfinite(r))
                    atomicOr(err, kErrNonFinite);
                lnL_tmarg[g] = r;
                if (lnw && lnpw)
                    lnw[g] = r + lnpw[g];
            }
        }
        if (lnL_t) {
            // the per-bin values of the warp's samples move by the same amount
            for (int t = 0; t < nb; ++t) {
                const uint32_t gt = __shfl_sync(0xffffffffu, g, t << gsh);
                const double ct = __shfl_sync(0xffffffffu, corr, t << gsh);
                if (__shfl_sync(0xffffffffu, good ? 1 : 0, t << gsh))
                    for (int j = lane; j < NT; j += 32)
                        lnL_t[(int64_t)gt * NT + j] += ct;
            }
        }
        __syncwarp();
    }
}

cudaError_t launch_fix_prep(const Problem &P, FixTables T, cudaStream_t st)
{
    const int64_t nq = (int64_t)P.K * P.M * P.n_q;
    fix_prep_q_kernel<<<(int)std::min<int64_t>((nq + 255) / 256, 4096), 256, 0, st>>>(P.Q64, nq, T.qdf);
    const int rows = P.K * (3 * T.dmax + 2) * T.nf;
    fix_prep_template_kernel<<<(rows + 7) / 8, 256, 0, st>>>(P, T);
    return cudaGetLastError();
}

cudaError_t launch_fix(const Problem &P, BinTable bt, FixTables T, const double *theta, int64_t n, PeakOut po,
                       int blen, float thr, uint32_t *idx, uint32_t *count, double *lnL_tmarg, double *lnL_t,
                       const double *lnpw, double *lnw, int *err, cudaStream_t st, int *launched)
{
    if (n <= 0)
        return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(uint32_t), st);
    if (e != cudaSuccess)
        return e;
    fix_select_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(po.q, po.m, n, thr, idx, count);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // one block per SM with as many warps as its shared memory holds (the coefficients are
    // staged once per block, the per-warp scratch grows with the warps): latency-bound
    // double-float chains want the warps
    int max_smem = 0;
    cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const size_t wbytes = fix_warp_bytes(P.K, P.M, T.dmax, T.nf);
    const size_t tbytes = (size_t)P.K * (3 * T.dmax + 2) * T.nf * 16;
    int nw = kFixMaxWarps;
    while (nw > 1 && wbytes * nw + tbytes > (size_t)max_smem)
        --nw;
    const int grid = (int)std::min<int64_t>((n + 3) / 4, (int64_t)sms);
    const size_t smem = wbytes * nw + tbytes;
    fix_kernel<<<grid, 32 * nw, smem, st>>>(P, bt, T, theta, idx, count, po, blen, lnL_tmarg, lnL_t, lnpw,
                                                    lnw, err);
    if (launched)
        *launched = 2;
    return cudaGetLastError();
}

cudaError_t prepare_fix_kernels() { return allow_max_dynamic_smem(fix_kernel); }

}  // namespace rift
