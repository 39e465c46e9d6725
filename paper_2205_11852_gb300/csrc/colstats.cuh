// Column means and extrema of [n_mock][nbin] matrices in two steps: partials
// over COL_CHUNKS row ranges (column_partials_kernel), closed by each block of
// the kernel that centres and splits the columns (column_stats).  Together
// they replace one block per 32 columns reading all rows, whose 21 blocks (a
// 3500 x 200 LC covariance) took 39 us.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace tpcf {
namespace {

constexpr int COL_WARPS = 8;      // warps per block, interleaved over the rows; lane = column
constexpr int COL_CHUNKS = 32;    // row ranges per column block

// The extrema are kept as order-preserving integer keys of the doubles
// (integer minima: the float64 pipe, two operations per clock and SM, is left
// to the sums).  All 64 bits: a column's scatter can be far below its mean,
// and extrema known to 2^-20 of their value only would bound the residuals of
// such a column by 2^-20 of the mean.
struct ColPartial {
    double sum;
    long long lo, hi;
};
constexpr long long KEY_MAX = 0x7fffffffffffffffll;

__device__ __forceinline__ long long key_of(double v)
{
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & KEY_MAX);
}

// the double with the key
__device__ __forceinline__ double of_key(long long key) { return __longlong_as_double(key ^ ((key >> 63) & KEY_MAX)); }

// part[v][chunk][b] of the rows [chunk * per, (chunk + 1) * per); zero (may be null): [v][n_zero][nbin] to clear
__global__ void __launch_bounds__(32 * COL_WARPS)
    column_partials_kernel(const double *__restrict__ x0, const double *__restrict__ x1,
                           const double *__restrict__ x2, int n_mock, int nbin, ColPartial *__restrict__ part,
                           uint32_t *__restrict__ zero, int n_zero)
{
    __shared__ ColPartial sh[COL_WARPS][32];
    const int v = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double *x = v == 0 ? x0 : (v == 1 ? x1 : x2);
    const int b = blockIdx.x * 32 + lane;
    if (zero && blockIdx.y == 0 && b < nbin)
        for (int k = warp; k < n_zero; k += COL_WARPS) zero[((size_t)v * n_zero + k) * nbin + b] = 0u;
    const int per = (n_mock + COL_CHUNKS - 1) / COL_CHUNKS;
    const int m0 = min(n_mock, (int)blockIdx.y * per), m1 = min(n_mock, m0 + per);
    double s[2] = {0.0, 0.0};
    long long lo = KEY_MAX, hi = -KEY_MAX - 1;
    if (b < nbin) {
        int m = m0 + warp;
        constexpr int U = 8;
        for (; m + (U - 1) * COL_WARPS < m1; m += U * COL_WARPS) {
            double t[U];
#pragma unroll
            for (int k = 0; k < U; k++) t[k] = x[(size_t)(m + k * COL_WARPS) * nbin + b];
#pragma unroll
            for (int k = 0; k < U; k++) {
                const long long key = key_of(t[k]);
                s[k & 1] += t[k];
                lo = min(lo, key);
                hi = max(hi, key);
            }
        }
#pragma unroll 4
        for (; m < m1; m += COL_WARPS) {
            const double t = x[(size_t)m * nbin + b];
            const long long key = key_of(t);
            s[0] += t;
            lo = min(lo, key);
            hi = max(hi, key);
        }
    }
    sh[warp][lane] = ColPartial{s[0] + s[1], lo, hi};
    __syncthreads();
    if (warp == 0 && b < nbin) {
        ColPartial p = sh[0][lane];
#pragma unroll
        for (int w = 1; w < COL_WARPS; w++) {
            p.sum += sh[w][lane].sum;
            p.lo = min(p.lo, sh[w][lane].lo);
            p.hi = max(p.hi, sh[w][lane].hi);
        }
        part[((size_t)v * COL_CHUNKS + blockIdx.y) * nbin + b] = p;
    }
}

// Mean, smallest and largest entry of column b (this thread's lane) of variant
// v, from all partials in a fixed order; called by every thread of a block of
// 32 x COL_WARPS.  A column with a NaN has a NaN mean (its extrema need not be
// numbers).
__device__ __forceinline__ void column_stats(const ColPartial *__restrict__ part, int v, int n_mock, int nbin, int b,
                                             double &mean, double &lo, double &hi)
{
    __shared__ ColPartial sh[COL_WARPS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int Q = COL_CHUNKS / COL_WARPS;
    static_assert(COL_CHUNKS % COL_WARPS == 0, "whole partials per warp");
    if (b < nbin) {
        ColPartial p[Q];
#pragma unroll
        for (int k = 0; k < Q; k++) p[k] = part[((size_t)v * COL_CHUNKS + warp * Q + k) * nbin + b];
#pragma unroll
        for (int k = 1; k < Q; k++) {
            p[0].sum += p[k].sum;
            p[0].lo = min(p[0].lo, p[k].lo);
            p[0].hi = max(p[0].hi, p[k].hi);
        }
        sh[warp][lane] = p[0];
    }
    __syncthreads();
    // one warp closes the columns: float64 operations run one to two per clock and SM
    __shared__ double smean[32], slo[32], shi[32];
    if (warp == 0 && b < nbin) {
        ColPartial p = sh[0][lane];
#pragma unroll
        for (int w = 1; w < COL_WARPS; w++) {
            p.sum += sh[w][lane].sum;
            p.lo = min(p.lo, sh[w][lane].lo);
            p.hi = max(p.hi, sh[w][lane].hi);
        }
        smean[lane] = p.sum / (double)n_mock;
        slo[lane] = of_key(p.lo);
        shi[lane] = of_key(p.hi);
    }
    __syncthreads();
    mean = smean[lane];
    lo = slo[lane];
    hi = shi[lane];
}

inline cudaError_t launch_column_partials(const double *x0, const double *x1, const double *x2, int n_var, int n_mock,
                                          int nbin, ColPartial *part, cudaStream_t s, uint32_t *zero = nullptr,
                                          int n_zero = 0)
{
    column_partials_kernel<<<dim3((nbin + 31) / 32, COL_CHUNKS, n_var), 32 * COL_WARPS, 0, s>>>(x0, x1, x2, n_mock,
                                                                                               nbin, part, zero, n_zero);
    return cudaGetLastError();
}

}  // namespace
}  // namespace tpcf
