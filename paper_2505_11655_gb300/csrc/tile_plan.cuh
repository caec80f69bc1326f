// What the kernels that plan the tensor-core likelihoods' work share (internal): the Q columns of
// a tile's samples, one warp per tile, and work items filed in four classes by cost.
//
// The delays are float32 here (the likelihood kernels place their samples themselves, from float64
// delays).  A planning kernel is one short pass at the latency of its loads and its instruction
// fetch, so it takes a small parameter block instead of the problem's and loops instead of unrolled
// code, and a block's items go to the global lists with one atomic per class (one warp per tile
// filing for itself, unrolled over samples and detectors: 27 us for 235 tiles, 61 us for 7813).
#pragma once

#include <climits>

#include "ile_common.cuh"

namespace rift {

constexpr int kPlanSamples = 128;   // per tile
constexpr int kPlanWarps = 8;       // tiles per block
constexpr int kPlanClasses = 4;

struct PlanProblem {
    int K, n_t;
    float beta;                          // Q samples per time bin
    double gmst;
    float x[kMaxDet][3], u0[kMaxDet];    // Q position of the first bin: u0 + x . n
};

inline PlanProblem plan_problem(const Problem &P)
{
    PlanProblem R{};
    R.K = P.K;
    R.n_t = P.n_t;
    R.beta = (float)(P.t_step * P.fs);
    R.gmst = P.gmst;
    for (int k = 0; k < P.K; ++k) {
        for (int i = 0; i < 3; ++i)
            R.x[k][i] = (float)P.xfs[k][i];
        R.u0[k] = (float)P.ufs0[k];
    }
    return R;
}

// Columns of the tile's samples: i0[k][e], INT_MIN where sample e does not exist (an index
// 0xffffffff, or one at n_theta <= 0xffffffff or beyond, is never read).  Lane k < K
// gets the lowest and highest of detector k (INT_MAX, INT_MIN without samples).
__device__ __forceinline__ void plan_columns(const PlanProblem &P, const double *__restrict__ theta,
                                             const uint32_t *__restrict__ perm, int64_t tile, int64_t n_use,
                                             int64_t n_theta, int (*i0)[kPlanSamples], int &lo, int &hi)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int e = lane; e < kPlanSamples; e += 32) {
        const int64_t si = tile * kPlanSamples + e;
        const uint32_t g = si < n_use ? (perm ? perm[si] : (uint32_t)si) : 0xffffffffu;
        const bool ok = g != 0xffffffffu && (int64_t)g < n_theta;
        float n0 = 0.f, n1 = 0.f, n2 = 0.f;
        if (ok) {
            const double *th = theta + 6 * (int64_t)g;
            const float h = (float)(th[0] - P.gmst), d = (float)th[1];
            float sa, ca, sd, cd;
            sincosf(h, &sa, &ca);
            sincosf(d, &sd, &cd);
            n0 = cd * ca;
            n1 = cd * sa;
            n2 = sd;
        }
#pragma unroll 1
        for (int k = 0; k < P.K; ++k) {
            const float u = fmaf(P.x[k][0], n0, fmaf(P.x[k][1], n1, fmaf(P.x[k][2], n2, P.u0[k])));
            i0[k][e] = ok ? (int)floorf(u) : INT_MIN;
        }
    }
    __syncwarp();
    lo = INT_MAX;
    hi = INT_MIN;
#pragma unroll 1
    for (int k = 0; k < P.K; ++k) {
        int a = INT_MAX, b = INT_MIN;
#pragma unroll
        for (int q = 0; q < kPlanSamples / 32; ++q) {
            const int v = i0[k][32 * q + lane];
            if (v != INT_MIN)
                a = min(a, v);
            b = max(b, v);
        }
        a = __reduce_min_sync(0xffffffffu, a);
        b = __reduce_max_sync(0xffffffffu, b);
        if (lane == k) {
            lo = a;
            hi = b;
        }
    }
}

// A block's items by class, filed together: list halves of `cap` items, classes 0 and 1 from the
// fronts, 3 and 2 from the backs.
template <typename T, int kItems> struct PlanFiles {
    T item[kItems];
    short cls[kItems], at[kItems];
    int n, count[kPlanClasses], base[kPlanClasses];
};

template <typename T, int kItems> __device__ __forceinline__ void plan_reset(PlanFiles<T, kItems> &F)
{
    if (threadIdx.x < kPlanClasses)
        F.count[threadIdx.x] = 0;
    if (threadIdx.x == 0)
        F.n = 0;
    __syncthreads();
}

template <typename T, int kItems> __device__ __forceinline__ void plan_file(PlanFiles<T, kItems> &F, T v, int cls)
{
    const int i = atomicAdd(&F.n, 1);
    F.item[i] = v;
    F.cls[i] = (short)cls;
    F.at[i] = (short)atomicAdd(&F.count[cls], 1);
}

// by every thread of the block
template <typename T, int kItems>
__device__ __forceinline__ void plan_write(PlanFiles<T, kItems> &F, T *__restrict__ list, int64_t cap,
                                           int *__restrict__ counts)
{
    __syncthreads();
    if (threadIdx.x < kPlanClasses && F.count[threadIdx.x])
        F.base[threadIdx.x] = atomicAdd(counts + threadIdx.x, F.count[threadIdx.x]);
    __syncthreads();
    for (int i = threadIdx.x; i < F.n; i += blockDim.x) {
        const int c = F.cls[i];
        const int64_t at = F.base[c] + F.at[i];
        list[((c == 1 || c == 2) ? cap : 0) + (c < 2 ? at : cap - 1 - at)] = F.item[i];
    }
}

// Item u of the classes in order; false beyond the last.
template <typename T>
__device__ __forceinline__ bool plan_item(const T *__restrict__ list, int64_t cap, const int *__restrict__ counts, int u,
                                          T &v)
{
    int c = 0;
    for (; c < kPlanClasses && u >= counts[c]; ++c)
        u -= counts[c];
    if (c == kPlanClasses)
        return false;
    v = list[((c == 1 || c == 2) ? cap : 0) + (c < 2 ? u : cap - 1 - u)];
    return true;
}

}  // namespace rift
