// Accuracy of the covariance estimates (Sect. 3): the covariance of the
// sample and LC covariances for Gaussian xi (Eqs. covcov, covcov_brute,
// covcov_fast), the chi^2 accuracy measure of Eq. (chi2) and its predicted
// value, and the eigenvalues of a symmetric matrix, used to check whether an
// LC covariance is positive definite before it is inverted (Sect. 3.4).
#include <algorithm>
#include <cmath>

#include "tpcf_internal.h"

namespace tpcf {
namespace {

// Variance of each covariance element, Eq. (covcov_fast) at k = i, l = j:
//   (N-1) Var(C_ij) = D_ii D_jj + D_ij^2 + c^2 (B_ii B_jj + B_ij^2)
// D = A + w B.  LC: w = 1/(2 M_a), c = 1/(2 M_a) - 1/M.  Sample covariance,
// Eq. (covcov_brute): B absent (c = 0) and A = C.
__device__ __forceinline__ double covcov_term(const double *A, const double *B, int n, int i, int j, double w,
                                              double c2)
{
    const size_t ii = (size_t)i * n + i, jj = (size_t)j * n + j, ij = (size_t)i * n + j;
    double dii = A[ii], djj = A[jj], dij = A[ij];
    double t = 0.0;
    if (B) {
        const double bii = B[ii], bjj = B[jj], bij = B[ij];
        dii = fma(w, bii, dii);
        djj = fma(w, bjj, djj);
        dij = fma(w, bij, dij);
        t = c2 * fma(bii, bjj, bij * bij);
    }
    return fma(dii, djj, dij * dij) + t;
}

__global__ void covcov_kernel(const double *__restrict__ A, const double *__restrict__ B, int n, double w, double c2,
                              double inv_nm1, double *__restrict__ var)
{
    const size_t nn = (size_t)n * n;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < nn; t += (size_t)gridDim.x * blockDim.x)
        var[t] = covcov_term(A, B, n, (int)(t / n), (int)(t % n), w, c2) * inv_nm1;
}

constexpr int RED_BLOCKS = 152 * 2, RED_THREADS = 256;

// sum over the block (blockDim.x a multiple of 32, at most 1024), in a fixed
// order; the result is valid in thread 0
__device__ double block_sum(double v)
{
    __shared__ double part[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < (int)(blockDim.x >> 5); k++) s += part[k];
    __syncthreads();
    return s;
}

// per-block partial sums over (i, j) of a normalised term:
//   mode 0: covcov_term / (R_ii R_jj)                 (predicted chi^2_2)
//   mode 1: (X_ij - Y_ij)^2 / (R_ii R_jj)             (measured chi^2, Eq. chi2)
__global__ void __launch_bounds__(RED_THREADS) chi2_partial(int mode, const double *__restrict__ X,
                                                            const double *__restrict__ Y, const double *__restrict__ R,
                                                            int n, double w, double c2, double *__restrict__ part)
{
    const size_t nn = (size_t)n * n;
    double s = 0.0;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < nn; t += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / n), j = (int)(t % n);
        const double norm = R[(size_t)i * n + i] * R[(size_t)j * n + j];
        double v;
        if (mode == 0) {
            v = covcov_term(X, Y, n, i, j, w, c2);
        } else {
            const double d = X[t] - Y[t];
            v = d * d;
        }
        s += v / norm;
    }
    s = block_sum(s);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

__global__ void __launch_bounds__(RED_THREADS) chi2_final(const double *__restrict__ part, int n_part, double scale,
                                                          double *__restrict__ out)
{
    double s = 0.0;
    for (int k = threadIdx.x; k < n_part; k += blockDim.x) s += part[k];
    s = block_sum(s);
    if (threadIdx.x == 0) *out = s * scale;
}

// ---- eigenvalues of a symmetric matrix ----
constexpr int TRI_CTAS = 8, TRI_THREADS = 512;

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// all threads of the cluster; orders this cluster's global-memory writes
// before the barrier ahead of its reads after it
__device__ __forceinline__ void cluster_sync_all()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Householder reduction of the symmetric matrix a[n][n] (overwritten) to
// tridiagonal form d[n], e[n-1] by one cluster of TRI_CTAS blocks: for each
// column k the reflector H = I - beta v v^T zeroes a[k+2.., k] and the
// trailing block B becomes H B H = B - v w^T - w v^T with p = beta B v,
// w = p - (beta p.v / 2) v.  Block r owns the rows i = r mod TRI_CTAS: it
// forms p_i for them (to pg in global memory), and after a cluster barrier
// every block forms w from all of p and updates its own rows; a second
// barrier ends the column.  v, beta and w are computed by every block alike
// (the same data and operation order), so every block takes the same branch
// at each barrier.
__global__ void __cluster_dims__(TRI_CTAS, 1, 1) __launch_bounds__(TRI_THREADS)
    tridiag_kernel(double *__restrict__ a, int n, double *__restrict__ d, double *__restrict__ e,
                   double *__restrict__ pg)
{
    extern __shared__ double sh[];
    double *v = sh;            // [n]
    double *w = sh + n;        // [n]
    __shared__ double s_alpha, s_beta, s_k;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const int rank = (int)cluster_rank();
    for (int k = 0; k + 2 < n; k++) {
        const int m0 = k + 1;   // the reflector acts on rows/cols m0..n-1
        // x = a[m0.., k] = a[k, m0..] (symmetric); alpha = -sign(x0) |x|
        const double *rk = a + (size_t)k * n;
        double ss = 0.0;
        for (int i = m0 + 1 + tid; i < n; i += blockDim.x) ss = fma(rk[i], rk[i], ss);
        const double tail = block_sum(ss);
        if (tid == 0) {
            const double x0 = rk[m0];
            if (tail == 0.0) {
                s_alpha = x0;      // column already reduced: H = I
                s_beta = 0.0;
            } else {
                const double nx = sqrt(fma(x0, x0, tail));
                const double alpha = x0 > 0.0 ? -nx : nx;
                const double v0 = x0 - alpha;
                s_alpha = alpha;
                s_beta = 2.0 / fma(v0, v0, tail);   // 2 / (v.v)
                v[m0] = v0;
            }
            if (rank == 0) {
                d[k] = rk[k];
                e[k] = s_alpha;
            }
        }
        __syncthreads();
        const double beta = s_beta;
        if (beta == 0.0) continue;   // nothing written in this column: no barrier needed
        for (int i = m0 + 1 + tid; i < n; i += blockDim.x) v[i] = rk[i];
        __syncthreads();
        // p_i = beta (B v)_i for this block's rows, one warp per row
        const int r0 = m0 + ((rank - m0) % TRI_CTAS + TRI_CTAS) % TRI_CTAS;   // first own row >= m0
        for (int i = r0 + TRI_CTAS * warp; i < n; i += TRI_CTAS * nw) {
            const double *row = a + (size_t)i * n;
            double t = 0.0;
            for (int j = m0 + lane; j < n; j += 32) t = fma(row[j], v[j], t);
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) pg[i] = beta * t;
        }
        cluster_sync_all();
        double pv = 0.0;
        for (int i = m0 + tid; i < n; i += blockDim.x) pv = fma(pg[i], v[i], pv);
        pv = block_sum(pv);
        if (tid == 0) s_k = 0.5 * beta * pv;
        __syncthreads();
        const double K = s_k;
        for (int i = m0 + tid; i < n; i += blockDim.x) w[i] = fma(-K, v[i], pg[i]);
        __syncthreads();
        // this block's rows of B - v w^T - w v^T
        const int m = n - m0, nr = (n - r0 + TRI_CTAS - 1) / TRI_CTAS;
        for (int t = tid; t < nr * m; t += blockDim.x) {
            const int i = r0 + TRI_CTAS * (t / m), j = m0 + t % m;
            double *x = a + (size_t)i * n + j;
            *x = fma(-v[i], w[j], fma(-w[i], v[j], *x));
        }
        cluster_sync_all();
    }
    if (rank == 0 && tid == 0) {
        if (n >= 2) {
            d[n - 2] = a[(size_t)(n - 2) * n + (n - 2)];
            e[n - 2] = a[(size_t)(n - 1) * n + (n - 2)];
        }
        d[n - 1] = a[(size_t)(n - 1) * n + (n - 1)];
    }
}

// v into block `rank`'s shared memory at the offset of `p` in this block's
__device__ __forceinline__ void st_cluster(double *p, uint32_t rank, double v)
{
    const uint32_t la = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(la), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}

// sum over the warp, in every lane
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

constexpr int TS_WARPS = 8;

// Shared-memory bytes of tridiag_smem_kernel<C> for order n: block r's rows
// (ceil(n / C) of n doubles) and six vectors.
size_t tri_smem_bytes(int n, int C)
{
    const size_t R = ((size_t)n + C - 1) / C;
    return (R * (size_t)n + 6 * (size_t)n) * sizeof(double);
}

// The same reduction with the matrix held in the shared memory of a cluster of
// C blocks, block r with the rows i = r mod C, and one cluster barrier per
// column.  What the other blocks need is written into their shared memory as
// soon as it is known: p_i = beta (B v)_i by the row's owner, and the row that
// the next column but one starts from.  At column k every block holds row k
// (all updates applied: it gives the reflector) and, from its owner, row k + 1
// as it was before column k; after the barrier, when all of p is there, every
// block applies column k's update to row k + 1 itself, which is column k + 1's
// start, while the owners update their rows.  Row i of B - v w^T - w v^T with
// w = p - K v (K = beta p.v / 2) is b_i - v_i p - (p_i - 2 K v_i) v, so no
// block forms w.  Warp 0 forms the next reflector while the other warps
// update.  Inboxes and v are double-buffered: a block writes slot k mod 2
// again only after a barrier that every block reaches past its last use.
//
// What bounds it: a column's chain of three reductions over a warp (0.26 us
// each: 109 clocks per step), a square root and a division (0.33 us each) and
// the barrier (0.18 us), and the float64 work, n^3 / C multiply-adds per SM at
// two per clock.  n = 120: 759 -> 465 us against two barriers, reads of remote
// rows and four block-wide reductions per column.
template <int C>
__global__ void __launch_bounds__(32 * TS_WARPS)
    tridiag_smem_kernel(const double *__restrict__ A, int n, double *__restrict__ d, double *__restrict__ e)
{
    extern __shared__ double sh[];
    const int R = (n + C - 1) / C;
    double *rows = sh;                         // [R][n]
    double *vb = rows + (size_t)R * n;         // [2][n] reflectors
    double *pb = vb + 2 * (size_t)n;           // [2][n] inbox: p
    double *xb = pb + 2 * (size_t)n;           // [2][n] inbox: row k + 1 before column k
    __shared__ double s_beta[2], s_k;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)cluster_rank();
    const int nown = (n - rank + C - 1) / C;   // rows of this block
    for (int idx = tid; idx < nown * n; idx += blockDim.x) {
        const int t = idx / n, j = idx % n;
        rows[(size_t)t * n + j] = A[(size_t)(rank + C * t) * n + j];
    }
    for (int j = tid; j < n; j += blockDim.x) xb[n + j] = A[(size_t)n + j];   // row 1

    // one warp: the reflector of column k from row k, x(j) for j >= k
    auto reflector = [&](int k, auto x) {
        const int m0 = k + 1;
        double *v = vb + (k & 1) * (size_t)n;
        double ss = 0.0, x0 = 0.0;
        for (int j = m0 + lane; j < n; j += 32) {
            const double xj = x(j);
            v[j] = xj;
            if (j == m0) x0 = xj; else ss = fma(xj, xj, ss);
        }
        const double xk = lane == 0 ? x(k) : 0.0;
        const double tail = warp_sum(ss);
        if (lane == 0) {
            double alpha = x0, beta = 0.0;   // tail = 0: already reduced, H = I
            if (tail != 0.0) {
                const double nx = sqrt(fma(x0, x0, tail));
                alpha = x0 > 0.0 ? -nx : nx;
                const double v0 = x0 - alpha;
                beta = 2.0 / fma(v0, v0, tail);   // 2 / (v.v)
                v[m0] = v0;
            }
            s_beta[k & 1] = beta;
            if (rank == 0) {
                d[k] = xk;
                e[k] = alpha;
            }
        }
        __syncwarp();
    };
    if (warp == 0) reflector(0, [&](int j) { return A[j]; });
    __syncthreads();
    cluster_sync_all();   // every block has started: its shared memory may be written

    for (int k = 0; k + 2 < n; k++) {
        const int m0 = k + 1;
        const double *v = vb + (k & 1) * (size_t)n;
        double *p = pb + (k & 1) * (size_t)n;
        const double beta = s_beta[k & 1];
        const int t0 = (m0 - rank + C - 1) / C > 0 ? (m0 - rank + C - 1) / C : 0;
        if (beta != 0.0) {
            // p_i for this block's rows i >= m0, two rows per warp at a time
            for (int t = t0 + 2 * warp; t < nown; t += 2 * TS_WARPS) {
                const bool two = t + 1 < nown;
                const double *r0 = rows + (size_t)t * n, *r1 = two ? r0 + n : r0;
                double a0 = 0.0, a1 = 0.0;
#pragma unroll 4
                for (int j = m0 + lane; j < n; j += 32) {
                    const double vj = v[j];
                    a0 = fma(r0[j], vj, a0);
                    a1 = fma(r1[j], vj, a1);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    a0 += __shfl_xor_sync(0xffffffffu, a0, o);
                    a1 += __shfl_xor_sync(0xffffffffu, a1, o);
                }
                if (lane < C) st_cluster(p + rank + C * t, (uint32_t)lane, beta * a0);
                if (two && lane < C) st_cluster(p + rank + C * (t + 1), (uint32_t)lane, beta * a1);
            }
        }
        cluster_sync_all();
        double K = 0.0;
        if (beta != 0.0) {
            if (warp == 0) {
                double pv = 0.0;
#pragma unroll 4
                for (int i = m0 + lane; i < n; i += 32) pv = fma(p[i], v[i], pv);
                pv = warp_sum(pv);
                if (lane == 0) s_k = 0.5 * beta * pv;
            }
            __syncthreads();
            K = s_k;
        }
        if (warp == 0) {
            // row k + 1 after this column's update: column k + 1's start
            const double *y = xb + ((k + 1) & 1) * (size_t)n;
            if (k + 3 < n) {
                if (beta != 0.0) {
                    const double vi = -v[m0], ui = -fma(-2.0 * K, v[m0], p[m0]);
                    reflector(k + 1, [&](int j) { return fma(vi, p[j], fma(ui, v[j], y[j])); });
                } else {
                    reflector(k + 1, [&](int j) { return y[j]; });
                }
            } else if (rank == 0) {   // the last column: d and e of the remaining 2 x 2 block's first row
                const double vi = -v[m0], ui = beta != 0.0 ? -fma(-2.0 * K, v[m0], p[m0]) : 0.0;
                if (lane < 2) {
                    const int j = n - 2 + lane;
                    (lane ? e : d)[n - 2] = beta != 0.0 ? fma(vi, p[j], fma(ui, v[j], y[j])) : y[j];
                }
            }
        } else {
            // this block's rows i > k + 1, one warp per row; row k + 2 also goes to every block
            for (int t = t0 + warp - 1; t < nown; t += TS_WARPS - 1) {
                const int i = rank + C * t;
                if (i == m0) continue;
                double *r = rows + (size_t)t * n;
                const double vi = beta != 0.0 ? -v[i] : 0.0, ui = beta != 0.0 ? -fma(-2.0 * K, v[i], p[i]) : 0.0;
                double *out = xb + (k & 1) * (size_t)n;
#pragma unroll 4
                for (int j = m0 + lane; j < n; j += 32) {
                    const double x = beta != 0.0 ? fma(vi, p[j], fma(ui, v[j], r[j])) : r[j];
                    r[j] = x;
                    if (i == k + 2 && k + 3 < n)
#pragma unroll
                        for (int q = 0; q < C; q++) st_cluster(out + j, (uint32_t)q, x);
                }
            }
        }
        __syncthreads();
    }
    cluster_sync_all();   // no block leaves while another may still write its shared memory
    if ((n - 1) % C == rank && tid == 0) d[n - 1] = rows[(size_t)((n - 1) / C) * n + n - 1];
}

// The continuants p_i of T - x I (leading principal minors: p_{-1} = 1, p_i =
// (d_i - x) p_{i-1} - e2_{i-1} p_{i-2}) of the tridiagonal T = (d, e) scaled so
// that its norm lies in [1, 2): the number of sign changes is the number of
// eigenvalues below x, without a division per step, and each step rounds like
// the ratio form of the Sturm sequence, so the count is that of a matrix
// within a few ulps of T.  t[i] = (d_i, e2_{i-1}), e2 at least 2^-180.  An
// exact zero becomes a tiny value of the opposite sign of p_{i-1}, which no
// later comparison can tell from it.  The pair (p_i, p_{i-1}) is rescaled by a
// power of two (exactly) every four steps: its larger member changes by 2^-183
// to 2^3 per step, so it stays within 2^+-950 in between.  Returns the count;
// (m, ex): the last continuant as m 2^ex.
__device__ __forceinline__ int sturm_count(const double2 *t, int n, double x, double &m, int &ex)
{
    double pm = 0.0, p = 1.0;
    int c = 0, shift = 0;
    auto step = [&](double2 q) {
        double pn = fma(q.x - x, p, -(q.y * pm));
        const int hp = __double2hiint(p);
        int hn = __double2hiint(pn);
        if (((hn & 0x7fffffff) | __double2loint(pn)) == 0) {
            hn = 0x01700000 | (~hp & (int)0x80000000);   // 2^-1000, sign opposite to p
            pn = __hiloint2double(hn, 0);
        }
        c += (int)((uint32_t)(hn ^ hp) >> 31);
        pm = p;
        p = pn;
    };
    int i = 0;
    for (; i + 4 <= n; i += 4) {
        const double2 q0 = t[i], q1 = t[i + 1], q2 = t[i + 2], q3 = t[i + 3];
        step(q0);
        step(q1);
        step(q2);
        step(q3);
        const int eb = max(__double2hiint(p) & 0x7ff00000, __double2hiint(pm) & 0x7ff00000) >> 20;
        if (eb > 1023 + 200 || eb < 1023 - 200) {
            const double f = __hiloint2double((2046 - eb) << 20, 0);
            p *= f;
            pm *= f;
            shift += eb - 1023;
        }
    }
    for (; i < n; i++) step(t[i]);
    m = p;
    ex = shift;
    return c;
}

// The same for a T with smaller off-diagonals, down to exact zeros (a diagonal
// matrix, blocks that do not couple): p_i alone may fall by any factor in a
// step, so the pair is rescaled whenever p_i leaves [2^-300, 2^300], and an
// exact zero becomes -2^-400 p_{i-1}.
__device__ __noinline__ int sturm_count_apart(const double2 *t, int n, double x, double &m, int &ex)
{
    double pm = 0.0, p = 1.0;
    int c = 0, shift = 0;
#pragma unroll 1
    for (int i = 0; i < n; i++) {
        double pn = fma(t[i].x - x, p, -(t[i].y * pm));
        if (pn == 0.0) pn = -0x1p-400 * p;
        c += (int)((uint32_t)(__double2hiint(pn) ^ __double2hiint(p)) >> 31);
        pm = p;
        p = pn;
        const int eb = (__double2hiint(p) >> 20) & 0x7ff;
        if (eb > 1023 + 300 || eb < 1023 - 300) {
            p = scalbn(p, 1023 - eb);
            pm = scalbn(pm, 1023 - eb);
            shift += eb - 1023;
        }
    }
    m = p;
    ex = shift;
    return c;
}

// eigenvalue i (ascending), one warp each, by multisection on the Sturm count
// from the Gershgorin interval: every round the lanes' 31 points shrink the
// bracket [lo, hi] (count(lo) <= i < count(hi)).  While the bracket holds
// other eigenvalues the points divide it evenly (5 bits a round).  Once it
// holds this one alone, the determinant changes sign in it, and sixteen of the
// points close in geometrically on the secant's root (whose error falls with
// the square of the bracket) while fifteen still divide it evenly: about
// seven rounds instead of twelve.  Ends when the bracket is down to two of its
// last places or a round no longer shrinks it.  The block stages T scaled by a
// power of two (exactly) to a norm in [1, 2).  Bound by the float64 pipe and
// the chain of n dependent multiply-adds per round; one warp per block, so
// that no two share an SM while there are SMs left (n = 120: 361 -> 175 us).
__global__ void __launch_bounds__(32) multisect_kernel(const double *__restrict__ d, const double *__restrict__ e,
                                                       int n, double *__restrict__ w)
{
    extern __shared__ double2 st[];   // [n]
    const int lane = threadIdx.x & 31, i = blockIdx.x;
    double lo = INFINITY, hi = -INFINITY, nrm = 0.0;
    bool nan = false;
    for (int k = lane; k < n; k += 32) {
        const double r = (k > 0 ? fabs(e[k - 1]) : 0.0) + (k + 1 < n ? fabs(e[k]) : 0.0);
        lo = fmin(lo, d[k] - r);
        hi = fmax(hi, d[k] + r);
        nrm = fmax(nrm, fabs(d[k]) + r);
        nan |= !(fabs(d[k]) + r < INFINITY);
    }
    if (__any_sync(0xffffffffu, nan)) {   // fmin and fmax pass over NaNs, and an infinite bracket does not close
        if (lane == 0) w[i] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        nrm = fmax(nrm, __shfl_xor_sync(0xffffffffu, nrm, o));
    }
    if (nrm == 0.0) {   // T = 0
        if (lane == 0) w[i] = 0.0;
        return;
    }
    const int ks = ilogb(nrm);   // T / 2^ks has its norm in [1, 2)
    bool small = false;
    for (int k = lane; k < n; k += 32) {
        const double ek = k > 0 ? scalbn(e[k - 1], -ks) : 0.0;
        st[k] = make_double2(scalbn(d[k], -ks), ek * ek);
        small |= k > 0 && ek * ek < 0x1p-180;
    }
    const bool apart = __any_sync(0xffffffffu, small);
    __syncwarp();
    const double pad = 4e-16 * n;
    lo = scalbn(lo, -ks) - pad;
    hi = scalbn(hi, -ks) + pad;
    // Everything but the counts runs on the integer and FP32 pipes: a float64 operation holds a warp's issue for 64
    // clocks.  Ends of the bracket by order-preserving integer keys; a point is lo + (hi - lo) frac with an FP32 frac.
    auto key = [](double v) -> long long {
        const long long b = __double_as_longlong(v);
        return b ^ ((b >> 63) & 0x7fffffffffffffffll);
    };
    auto expo = [](double v) -> int { return (__double2hiint(v) >> 20) & 0x7ff; };
    const float geo = (lane & 1 ? 1.0f : -1.0f) * __int_as_float((127 - 5 - 2 * ((lane - 15) >> 1)) << 23);
    int clo = 0, chi = n, exlo = 0, exhi = 0;   // counts and determinants at the bracket's ends
    double mlo = 0.0, mhi = 0.0;                // 0: not known
    for (int it = 0; it < 96; it++) {
        const double h = hi - lo;
        // done: the bracket is 2 last places of its ends, or empty
        if (h <= 0.0 || expo(h) <= max(1023 - 320, max(expo(lo), expo(hi)) - 51)) break;
        float frac = (float)(lane + 1) * (1.0f / 32.0f);
        if (clo == i && chi == i + 1 && mlo != 0.0 && mhi != 0.0) {
            if (lane < 15) {
                frac = (float)(lane + 1) * (1.0f / 16.0f);
            } else {   // the secant's root a / (a + b), a and b the determinants at lo and hi
                const float fa = __int_as_float((__double2hiint(mlo) & 0xfffff) << 3 | 0x3f800000);
                const float fb = __int_as_float((__double2hiint(mhi) & 0xfffff) << 3 | 0x3f800000);
                const int dx = max(-60, min(60, expo(mhi) + exhi - expo(mlo) - exlo));
                const float ratio = __fdividef(fb, fa) * __int_as_float((127 + dx) << 23);
                frac = fminf(fmaxf(__fdividef(1.0f, 1.0f + ratio) + geo, 0.0f), 1.0f);
            }
        }
        const double x = fma(h, (double)frac, lo);
        double m;
        int ex;
        const int c = apart ? sturm_count_apart(st, n, x, m, ex) : sturm_count(st, n, x, m, ex);
        const bool above = c > i;
        // the highest point that is not above and the lowest that is (lane 31's point takes part in neither)
        const long long kx = key(x), none = 0x7fffffffffffffffll;
        long long bl = lane < 31 && !above ? kx : -none, bh = lane < 31 && above ? kx : none;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            bl = max(bl, __shfl_xor_sync(0xffffffffu, bl, o));
            bh = min(bh, __shfl_xor_sync(0xffffffffu, bh, o));
        }
        bool moved = false;
        if (bl > key(lo)) {
            const int l = __ffs(__ballot_sync(0xffffffffu, lane < 31 && !above && kx == bl)) - 1;
            lo = __shfl_sync(0xffffffffu, x, l);
            clo = __shfl_sync(0xffffffffu, c, l);
            mlo = __shfl_sync(0xffffffffu, m, l);
            exlo = __shfl_sync(0xffffffffu, ex, l);
            moved = true;
        }
        if (bh < key(hi)) {
            const int l = __ffs(__ballot_sync(0xffffffffu, lane < 31 && above && kx == bh)) - 1;
            hi = __shfl_sync(0xffffffffu, x, l);
            chi = __shfl_sync(0xffffffffu, c, l);
            mhi = __shfl_sync(0xffffffffu, m, l);
            exhi = __shfl_sync(0xffffffffu, ex, l);
            moved = true;
        }
        if (!moved) break;
    }
    if (lane == 0) w[i] = scalbn(0.5 * (lo + hi), ks);
}

int blocks_for(size_t n, int threads) { return (int)std::max<size_t>(1, std::min<size_t>((n + threads - 1) / threads, 152 * 16)); }

// Launch shape of the shared-memory reduction in a cluster of C blocks
template <int C>
struct ClusterLaunch {
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = {};
    ClusterLaunch(int n, cudaStream_t s)
    {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = C;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3(32 * TS_WARPS);
        cfg.dynamicSmemBytes = tri_smem_bytes(n, C);
        cfg.stream = s;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
    ClusterLaunch(const ClusterLaunch &) = delete;
};

// The matrix fits in the shared memory of C blocks and the device runs clusters of that size and footprint (more than 8
// blocks is not guaranteed: a partition may hold fewer SMs of one cluster's reach).  max_cluster > 0 (tests) stands in
// for the device's answer.
template <int C>
bool cluster_fits(int n, int max_cluster)
{
    constexpr size_t room = (size_t)226 << 10;
    ClusterLaunch<C> l(n, nullptr);
    const size_t sb = l.cfg.dynamicSmemBytes;
    if (sb > room || (max_cluster > 0 && C > max_cluster)) return false;
    int held = 0;
    bool ok = cudaFuncSetAttribute(tridiag_smem_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sb) == cudaSuccess;
    if (ok && C > 8)
        ok = cudaFuncSetAttribute(tridiag_smem_kernel<C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    ok = ok && cudaOccupancyMaxActiveClusters(&held, tridiag_smem_kernel<C>, &l.cfg) == cudaSuccess && held > 0;
    if (!ok) cudaGetLastError();
    return ok;
}

template <int C>
cudaError_t launch_tridiag_smem(const double *A, int n, double *d, double *e, cudaStream_t s)
{
    ClusterLaunch<C> l(n, s);
    return cudaLaunchKernelEx(&l.cfg, tridiag_smem_kernel<C>, A, n, d, e);
}

// The cluster size of the shared-memory reduction for order n: 16 blocks (an
// opt-in size) from n = 96, below which 8 do as well, else 8; 0 when neither
// holds the matrix (n > 628) or the device has no room for such a cluster.
// Whole call with 16 / with 8 / before: n = 96
// 497 / 497 / 874 us, 120 675 / 698 / 1134, 200 1224 / 1434 / 2125, 420 4132 /
// 5930 / 6794, 600 8458 / - / 16750.
int pick_cluster(int n, int max_cluster)
{
    if (n >= 96 && cluster_fits<16>(n, max_cluster)) return 16;
    return cluster_fits<8>(n, max_cluster) ? 8 : 0;
}

}  // namespace

cudaError_t launch_covcov(const double *A, const double *B, int nbin, int M_a, double M, int n_mock, double *var,
                          cudaStream_t s)
{
    const double w = B ? 0.5 / M_a : 0.0;
    const double c = B ? 0.5 / M_a - 1.0 / M : 0.0;
    covcov_kernel<<<blocks_for((size_t)nbin * nbin, 256), 256, 0, s>>>(A, B, nbin, w, c * c,
                                                                        1.0 / (double)(n_mock - 1), var);
    return cudaGetLastError();
}

size_t chi2_work_bytes() { return RED_BLOCKS * sizeof(double); }

cudaError_t launch_chi2(int mode, const double *X, const double *Y, const double *R, int nbin, int M_a, double M,
                        double *work, double *out, cudaStream_t s)
{
    double w = 0.0, c = 0.0;
    if (mode == 0 && Y) {
        w = 0.5 / M_a;
        c = 0.5 / M_a - 1.0 / M;
    }
    const int nb = std::min(RED_BLOCKS, blocks_for((size_t)nbin * nbin, RED_THREADS));
    chi2_partial<<<nb, RED_THREADS, 0, s>>>(mode, X, Y, R, nbin, w, c * c, work);
    chi2_final<<<1, RED_THREADS, 0, s>>>(work, nb, 1.0 / ((double)nbin * nbin), out);
    return cudaGetLastError();
}

size_t eig_work_bytes(int n) { return ((size_t)n * n + 3 * (size_t)n) * sizeof(double); }

cudaError_t launch_eigvalsh(const double *C, int n, double *work, double *w, int max_cluster, cudaStream_t s)
{
    double *a = work, *d = work + (size_t)n * n, *e = d + n, *pg = e + n;
    cudaError_t err;
    int cl = 0;   // blocks of the cluster whose shared memory holds the matrix; 0: none does
    if (n >= 3) cl = pick_cluster(n, max_cluster);
    if (cl == 16) {
        err = launch_tridiag_smem<16>(C, n, d, e, s);
        if (err != cudaSuccess) return err;
    } else if (cl == 8) {
        err = launch_tridiag_smem<8>(C, n, d, e, s);
        if (err != cudaSuccess) return err;
    } else {
        err = cudaMemcpyAsync(a, C, (size_t)n * n * sizeof(double), cudaMemcpyDeviceToDevice, s);
        if (err != cudaSuccess) return err;
        tridiag_kernel<<<TRI_CTAS, TRI_THREADS, 2 * (size_t)n * sizeof(double), s>>>(a, n, d, e, pg);
    }
    multisect_kernel<<<n, 32, (size_t)n * sizeof(double2), s>>>(d, e, n, w);
    return cudaGetLastError();
}

}  // namespace tpcf
