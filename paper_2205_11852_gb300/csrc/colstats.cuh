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
constexpr long long KEY_MAX = 0x7fffffffffffffffll;

__device__ __forceinline__ long long key_of(double v)
{
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & KEY_MAX);
}

// the double with the key
__device__ __forceinline__ double of_key(long long key) { return __longlong_as_double(key ^ ((key >> 63) & KEY_MAX)); }

// What is known of some rows of a column: the sum, or the sum and the extrema's
// keys.  (The extrema's integer operations and stores took 2 us of the 54 of a
// 1201 x 333 split-precision covariance, which has no use for them.)
struct ColSum {
    double sum;
    static __device__ __forceinline__ ColSum none() { return ColSum{0.0}; }
    __device__ __forceinline__ void see(double) {}
    __device__ __forceinline__ void join(const ColSum &o) { sum += o.sum; }
};
struct ColRange {
    double sum;
    long long lo, hi;
    static __device__ __forceinline__ ColRange none() { return ColRange{0.0, KEY_MAX, -KEY_MAX - 1}; }
    __device__ __forceinline__ void see(double v)
    {
        const long long key = key_of(v);
        lo = min(lo, key);
        hi = max(hi, key);
    }
    __device__ __forceinline__ void join(const ColRange &o)
    {
        sum += o.sum;
        lo = min(lo, o.lo);
        hi = max(hi, o.hi);
    }
};

// part[v][chunk][b] of the rows [chunk * per, (chunk + 1) * per); clear[v][n_clear][nbin] is set to zero for a kernel
// that follows
template <class P>
__global__ void __launch_bounds__(32 * COL_WARPS)
    column_partials_kernel(const double *__restrict__ x0, const double *__restrict__ x1,
                           const double *__restrict__ x2, int n_mock, int nbin, P *__restrict__ part,
                           uint32_t *__restrict__ clear, int n_clear)
{
    __shared__ P sh[COL_WARPS][32];
    const int v = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double *x = v == 0 ? x0 : (v == 1 ? x1 : x2);
    const int b = blockIdx.x * 32 + lane;
    const int per = (n_mock + COL_CHUNKS - 1) / COL_CHUNKS;
    const int m0 = min(n_mock, (int)blockIdx.y * per), m1 = min(n_mock, m0 + per);
    double s[2] = {0.0, 0.0};
    P mine = P::none();
    if (b < nbin) {
        int m = m0 + warp;
        constexpr int U = 8;
        for (; m + (U - 1) * COL_WARPS < m1; m += U * COL_WARPS) {
            double t[U];
#pragma unroll
            for (int k = 0; k < U; k++) t[k] = x[(size_t)(m + k * COL_WARPS) * nbin + b];
#pragma unroll
            for (int k = 0; k < U; k++) {
                s[k & 1] += t[k];
                mine.see(t[k]);
            }
        }
#pragma unroll 4
        for (; m < m1; m += COL_WARPS) {
            const double t = x[(size_t)m * nbin + b];
            s[0] += t;
            mine.see(t);
        }
    }
    mine.sum = s[0] + s[1];
    sh[warp][lane] = mine;
    __syncthreads();
    if (warp == 0 && b < nbin) {
#pragma unroll
        for (int w = 1; w < COL_WARPS; w++) mine.join(sh[w][lane]);
        part[((size_t)v * COL_CHUNKS + blockIdx.y) * nbin + b] = mine;
    }
    if (blockIdx.y == COL_CHUNKS - 1 && b < nbin)   // (the row range with the fewest rows)
        for (int k = warp; k < n_clear; k += COL_WARPS) clear[((size_t)v * n_clear + k) * nbin + b] = 0u;
}

// Mean, and what is known of all rows, of column b (this thread's lane) of
// variant v, from all partials in a fixed order; called by every thread of a
// block of 32 x COL_WARPS.  A column with a NaN has a NaN mean (its extrema
// need not be numbers).
template <class P>
__device__ __forceinline__ P column_stats(const P *__restrict__ part, int v, int n_mock, int nbin, int b, double &mean)
{
    __shared__ P sh[COL_WARPS][32];
    __shared__ double smean[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int Q = COL_CHUNKS / COL_WARPS;
    static_assert(COL_CHUNKS % COL_WARPS == 0, "whole partials per warp");
    if (b < nbin) {
        P p[Q];
#pragma unroll
        for (int k = 0; k < Q; k++) p[k] = part[((size_t)v * COL_CHUNKS + warp * Q + k) * nbin + b];
#pragma unroll
        for (int k = 1; k < Q; k++) p[0].join(p[k]);
        sh[warp][lane] = p[0];
    }
    __syncthreads();
    // one warp closes the columns: float64 operations run one to two per clock and SM
    if (warp == 0 && b < nbin) {
        P p = sh[0][lane];
#pragma unroll
        for (int w = 1; w < COL_WARPS; w++) p.join(sh[w][lane]);
        smean[lane] = p.sum / (double)n_mock;
        sh[0][lane] = p;
    }
    __syncthreads();
    mean = smean[lane];
    return sh[0][lane];
}

template <class P>
inline cudaError_t launch_column_partials(const double *x0, const double *x1, const double *x2, int n_var, int n_mock,
                                          int nbin, P *part, uint32_t *clear, int n_clear, cudaStream_t s)
{
    column_partials_kernel<P><<<dim3((nbin + 31) / 32, COL_CHUNKS, n_var), 32 * COL_WARPS, 0, s>>>(
        x0, x1, x2, n_mock, nbin, part, clear, n_clear);
    return cudaGetLastError();
}

}  // namespace
}  // namespace tpcf
