// Float64 covariances on the 5th-generation tensor cores (tcgen05): the Gram
// products G = Y^T Y of the centred correlation functions (Eqs. bruteforce,
// R1R2, LCdef) from error-free digit splits of Y (the scheme of Ozaki, Ogita,
// Oishi and Rump 2012, on a low-precision matrix unit as Ootomo, Ozaki and
// Yokota 2024 do it on integer ones).
//
// GB300's float64 pipe runs about two fused multiply-adds per clock and SM, so
// a 3500 x 200 LC covariance spent 1.29 of its 1.36 ms in a tiled float64
// kernel.  Here every residual y of column i becomes a 56-bit fixed-point
// number f = round(y 2^(55 - e_i)), 2^e_i > max |y| of the column, and f eight
// balanced digits of 7 bits (|d| <= 64), which bf16 holds exactly.  A product
// of two digits is at most 2^12 and the FP32 accumulators of the tensor cores
// add integers below 2^24 exactly, so the products of digits p and q with
// p + q = l ("level" l, weight 2^-7l) of up to 28 slices of 16 mocks (448 x 7
// x 2^12 < 2^24) add up in one accumulator without any rounding.  Levels 0..6
// are kept exactly; level 8 (the digits carry their weight 2^-7p, so it lands
// 7 bits lower) joins level 7 in one accumulator, whose rounding lies below
// the fixed-point resolution of y; levels from 9 on are dropped.  Eight
// accumulators of 64 columns fill tensor memory.  A CTA writes its tile as
// pairs of 64-bit integers, and the combining kernel adds the K-segments as
// integers and rounds to float64 once, so the result does not depend on an
// order of summation.
//
// Which columns are split.  A fixed-point residual is exact from an eighth of
// its column's largest one on (often from less) and off by up to 2^(e_i - 56)
// below, whatever its own size, where a float64 product keeps 53 bits.  That
// is nothing against the sum of |y_i y_j| of ordinary columns (0.01 to 0.08 of
// 2^-53 of it, root mean square, on normal ones; the products' own float64
// sums 0.5 to 1.2), but not of columns whose large residuals are few and meet
// small ones of other columns: with two pairs of +-10^6 in different mocks of
// columns of unit scatter it would be 4 x 10^4.  So the octaves of a column's
// residuals are counted, and it is split when, with a the mean of |y| and r
// its root mean square,
//   2^e_i r <= 2 sqrt(n) a^2    (the products' error against a sum of
//                                independent |y_i| |y_j|, 0.1 x 2^-53), and
//   3/4 of its residuals lie above a / 6 (to a factor of two: any two such
//                                columns have half their mocks in common).
// Over normal, Student t, lognormal, rare-event and two-scale columns, among
// them ones made so that the large residuals of one column meet the small ones
// of the next, at 4 to 3500 mocks, the split columns' error stayed below half
// of the float64 sums'.  Elements of the others (and of columns whose residuals
// are not finite or lie outside 2^+-400) are summed in float64 by the combining
// kernel, in two levels, over tiles of 8 x 8 elements.
//
// What bounds it: the operand tiles' way into the SMs, 48 KB per slice and CTA
// (about 5.7 TB/s over 144 CTAs; a tile of 8 columns, with a quarter of the
// multiplications, takes 85 % of a full tile's loop).  The digits of B are
// stacked along N, so that 20 MMAs of up to 256 columns cover a slice's 43
// products and A is read from shared memory once per 256 columns.  Measured
// (3500 x 200 LC covariance): Gram 44 us, digits 19, column statistics 10,
// combination 8.5; 1356 -> 79 us per call, 82 with the octave counts.  Columns
// that are not split: 3500 x 200 with one of them 112 -> 415 us of device and
// host time, with all 941, by the tiled float64 kernel 1393.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "colstats.cuh"
#include "tc_ptx.cuh"
#include "tpcf_internal.h"

namespace tpcf {
namespace {

constexpr int NDIG = 8;                        // digits of 7 bits
constexpr int DKS = 16;                        // mocks per slice (K of one bf16 MMA)
constexpr int DTM = 128, DTN = 64;             // tile rows and columns (at most)
constexpr int DIG_BYTES = DTM * DKS * 2;       // one digit of 128 rows and one slice
constexpr int SLICE_BYTES = NDIG * DIG_BYTES;  // all digits
constexpr int DSBO = (DKS * 2 / 16) * 128;     // bytes between 8-row groups (as the K-major tiles of gram_split.cu)
constexpr int SEG_SLICES = 28;                 // slices whose level sums stay exact (448 x 7 x 2^12 < 2^24)
constexpr int DSTAGE = 4;                      // slices in flight
constexpr int STAGE_BYTES = SLICE_BYTES + SLICE_BYTES / 2;
constexpr int D_EPI_WARPS = 8;
constexpr int D_THREADS = 32 * (D_EPI_WARPS + 2);
constexpr int EXP_BAD = 1 << 20;               // "exponent" of a column that is not split
constexpr int OCT = 16;                        // octaves of |y| below 2^e that are counted, the last with all below

static_assert(SEG_SLICES * DKS * 7 * 4096 < (1 << 24), "level sums must stay exact in FP32");

// round(y 2^(55 - e)) for |y| < 2^e
__device__ __forceinline__ long long to_fixed(double y, int e)
{
    const long long bits = __double_as_longlong(y);
    const int ex = (int)((bits >> 52) & 0x7ff);
    if (ex == 0) return 0;
    const long long m = (bits & 0xfffffffffffffll) | (1ll << 52);
    const int sh = ex - 1023 - e + 3;          // <= 2
    long long f;
    if (sh >= 0) f = m << sh;
    else f = sh < -54 ? 0 : (m + (1ll << (-sh - 1))) >> -sh;
    return bits < 0 ? -f : f;
}

// Centred residuals as digits.  Tile layout: digits[v][row block of 128
// bins][slice][digit][128 x 16], each digit in the K-major, non-swizzled
// layout of the tensor-core descriptors (8 rows x 16 bytes core matrices).
// A block takes 32 columns (one per lane) and one of COL_CHUNKS row ranges of
// one variant; it first closes the column statistics of all row ranges
// (column_partials_kernel).  ecol[v][b]: the column's exponent; mean[v][b];
// oct[v][k][b]: residuals with 2^(e-1-k) <= |y| < 2^(e-k) (k = 15: all below).
// Rows past nbin are left unwritten (an output element depends on its own two
// operand rows only), mocks past n_mock are zeros.  Two float64 additions per
// element (the sum and the residual) bound the two kernels.
__global__ void __launch_bounds__(32 * COL_WARPS)
    digits_kernel(const double *__restrict__ x0, const double *__restrict__ x1, const double *__restrict__ x2,
                  const ColRange *__restrict__ part, int n_mock, int nbin, int n_rb, int n_ks,
                  unsigned char *__restrict__ tiles, int *__restrict__ ecol, double *__restrict__ mean,
                  uint32_t *__restrict__ oct)
{
    __shared__ uint32_t cnt[OCT][32];
    const int v = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double *x = v == 0 ? x0 : (v == 1 ? x1 : x2);
    const int b = blockIdx.x * 32 + lane;
    double mu;
    for (int k = threadIdx.x; k < OCT * 32; k += blockDim.x) cnt[k / 32][k % 32] = 0u;
    const ColRange range = column_stats(part, v, n_mock, nbin, b, mu);   // (has block barriers)
    // |x - mean| is largest at an extremum (rounding is monotone); NaN and infinities fail the tests
    const double top = fmax(of_key(range.hi) - mu, mu - of_key(range.lo));
    const bool bad = !(mu == mu) || !(top < 0x1p400) || (top != 0.0 && !(top > 0x1p-400));
    const int e = bad || top == 0.0 ? 0 : ilogb(top) + 1;
    if (blockIdx.y == 0 && warp == 0 && b < nbin) {
        ecol[(size_t)v * nbin + b] = bad ? EXP_BAD : e;
        mean[(size_t)v * nbin + b] = mu;
    }
    const int r = b % DTM;
    unsigned char *col = tiles + ((size_t)v * n_rb + b / DTM) * n_ks * SLICE_BYTES + (r >> 3) * DSBO + (r & 7) * 16;
    constexpr long long BIAS = 0x40ll * (1ll + (1ll << 7) + (1ll << 14) + (1ll << 21) + (1ll << 28) + (1ll << 35) +
                                         (1ll << 42) + (1ll << 49));
    // groups of 8 mocks: one 16-byte chunk per digit
    const int n_g = 2 * n_ks, per = (n_g + gridDim.y - 1) / gridDim.y;
    const int g1 = b < nbin ? min(n_g, ((int)blockIdx.y + 1) * per) : 0;
    for (int g = (int)blockIdx.y * per + warp; g < g1; g += COL_WARPS) {
        double y[8];
#pragma unroll
        for (int k = 0; k < 8; k++) y[k] = g * 8 + k < n_mock ? x[(size_t)(g * 8 + k) * nbin + b] : mu;
        long long t[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const double d = y[k] - mu;
            t[k] = (bad ? 0ll : to_fixed(d, e)) + BIAS;
            if (g * 8 + k < n_mock) atomicAdd(&cnt[min(OCT - 1, e + 1022 - ((__double2hiint(d) >> 20) & 0x7ff)) & (OCT - 1)][lane], 1u);
        }
        unsigned char *dst = col + (size_t)(g >> 1) * SLICE_BYTES + (g & 1) * 128;
#pragma unroll
        for (int d = 0; d < NDIG; d++) {
            // digit d (0: the leading one) times 2^-7d: (2^23 + u) 2^-7d - (2^23 + 64) 2^-7d, exact
            const int sft = 7 * (NDIG - 1 - d);
            const uint32_t mg = 0x4B000000u - ((uint32_t)(7 * d) << 23);
            const float off = __uint_as_float(mg | 64u);
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                uint32_t u0 = (uint32_t)(t[2 * k] >> sft), u1 = (uint32_t)(t[2 * k + 1] >> sft);
                if (d > 0) {
                    u0 &= 127u;
                    u1 &= 127u;
                }
                const __nv_bfloat162 p = __floats2bfloat162_rn(__uint_as_float(mg | u0) - off,
                                                               __uint_as_float(mg | u1) - off);
                w[k] = *reinterpret_cast<const uint32_t *>(&p);
            }
            *(uint4 *)(dst + d * DIG_BYTES) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
    __syncthreads();
    if (b < nbin)
        for (int k = warp; k < OCT; k += COL_WARPS)
            if (cnt[k][lane]) atomicAdd(&oct[((size_t)v * OCT + k) * nbin + b], cnt[k][lane]);
}

// Whether a column of n residuals with these octave counts is split (see the top); o[k * stride]
__device__ __forceinline__ bool column_fits(const uint32_t *__restrict__ o, int stride, int n)
{
    float a = 0.0f, q = 0.0f, w = 1.0f;   // mean |y| and mean square over 2^e, residuals spread evenly in an octave
    uint32_t c[OCT];
#pragma unroll
    for (int k = 0; k < OCT; k++) c[k] = o[(size_t)k * stride];
#pragma unroll
    for (int k = 0; k < OCT - 1; k++) {
        w *= 0.5f;
        a += 1.5f * w * (float)c[k];
        q += 7.0f / 3.0f * w * w * (float)c[k];
    }
    if (a == 0.0f) return true;   // all residuals are zero
    a /= (float)n;
    q /= (float)n;
    if (!(q <= 4.0f * a * a * a * a * (float)n)) return false;
    uint32_t above = 0;
    w = 1.0f;
#pragma unroll
    for (int k = 0; k < OCT - 1; k++) {
        if (w > a * (1.0f / 6.0f)) above += c[k];
        w *= 0.5f;
    }
    return 4ull * ((uint32_t)n - above) <= (uint32_t)n;
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

// eight columns of all eight levels (cw columns apart), complete on return
__device__ __forceinline__ void tmem_ld8x8(uint32_t t, uint32_t cw, uint32_t (&r)[8][8])
{
#define O8(i) "=r"(r[i][0]), "=r"(r[i][1]), "=r"(r[i][2]), "=r"(r[i][3]), "=r"(r[i][4]), "=r"(r[i][5]), "=r"(r[i][6]), "=r"(r[i][7])
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%64];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8, %9, %10, %11, %12, %13, %14, %15}, [%65];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16, %17, %18, %19, %20, %21, %22, %23}, [%66];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24, %25, %26, %27, %28, %29, %30, %31}, [%67];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%32, %33, %34, %35, %36, %37, %38, %39}, [%68];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%40, %41, %42, %43, %44, %45, %46, %47}, [%69];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%48, %49, %50, %51, %52, %53, %54, %55}, [%70];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%56, %57, %58, %59, %60, %61, %62, %63}, [%71];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : O8(0), O8(1), O8(2), O8(3), O8(4), O8(5), O8(6), O8(7)
        : "r"(t), "r"(t + cw), "r"(t + 2 * cw), "r"(t + 3 * cw), "r"(t + 4 * cw), "r"(t + 5 * cw), "r"(t + 6 * cw),
          "r"(t + 7 * cw)
        : "memory");
#undef O8
}

constexpr int digits_smem_bytes() { return DSTAGE * STAGE_BYTES + 8 * (2 * DSTAGE + 1) + 16; }

// Tile pairs: rows [128 bi, +128) (operand A), columns [64 bj, +64) (operand
// B, narrowed to the last multiple of 16 that holds bins), bj >= 2 bi: every
// element j >= i of the upper triangle.  One CTA per (pair, variant, segment
// of at most SEG_SLICES slices).  Warp 9 streams the segment's slices through
// DSTAGE stages (bulk copies), one thread of warp 8 issues the MMAs, and warps
// 0-7 read the eight accumulators back once and write T[segment][v][j][i],
// consecutive i per warp.
//
// The first CTA of each variant also decides which columns the combining
// kernel takes from the products (its warps 0-7 would wait for them).
//
// Every wait is bounded.  The MMA thread commits `done` also when a wait gave
// up, so the epilogue's wait always ends; a wait that gave up sets
// STATUS_TIMEOUT and nothing of the tile is written.
__global__ void __launch_bounds__(D_THREADS, 1)
    gram_digits_kernel(const unsigned char *__restrict__ tiles, int nbin, int n_rb, int n_cb, int n_ks, int spc,
                       longlong2 *__restrict__ T, const uint32_t *__restrict__ oct, int n_mock,
                       int *__restrict__ ecol, int *__restrict__ status)
{
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *full = (uint64_t *)(smem + DSTAGE * STAGE_BYTES);
    uint64_t *empty = full + DSTAGE;
    uint64_t *done = empty + DSTAGE;
    uint32_t *slot = (uint32_t *)(done + 1);
    int *ok_mma = (int *)(slot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int bi = 0, rest = (int)blockIdx.x;
    while (rest >= n_cb - 2 * bi) {
        rest -= n_cb - 2 * bi;
        bi++;
    }
    const int bj = 2 * bi + rest;
    const int v = blockIdx.y, kc = blockIdx.z;
    const int k0 = kc * spc, n = min(n_ks, k0 + spc) - k0;   // n >= 1 by the host's chunking
    const int cw = min(DTN, ((nbin - bj * DTN) + 15) & ~15);  // columns of the tile, a multiple of 16
    if (warp == 0) tmem_alloc(slot, 8 * DTN);
    if (tid == 0) {
        for (int i = 0; i < DSTAGE; i++) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        mbar_init(done, 1);
        mbar_fence_init();
        *ok_mma = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *slot;
    if (warp == D_EPI_WARPS + 1) {
        if (lane == 0) {
            const unsigned char *ga = tiles + ((size_t)v * n_rb + bi) * n_ks * SLICE_BYTES;
            const unsigned char *gb = tiles + ((size_t)v * n_rb + (bj >> 1)) * n_ks * SLICE_BYTES +
                                      (bj & 1) * (DIG_BYTES / 2);
            const uint32_t bb = (uint32_t)cw * DKS * 2;   // one digit of B
            int issued = 0;
            bool ok = true;
            for (; issued < n; issued++) {
                const int st = issued % DSTAGE;
                if (issued >= DSTAGE) {
                    ok = mbar_wait(&empty[st], (uint32_t)(issued / DSTAGE - 1) & 1u, SPIN_LIMIT);
                    if (!ok) break;
                }
                unsigned char *sa = smem + st * STAGE_BYTES;
                mbar_expect_tx(&full[st], (uint32_t)SLICE_BYTES + NDIG * bb);
                bulk_g2s(sa, ga + (size_t)(k0 + issued) * SLICE_BYTES, SLICE_BYTES, &full[st]);
                for (int d = 0; d < NDIG; d++)
                    bulk_g2s(sa + SLICE_BYTES + d * bb, gb + (size_t)(k0 + issued) * SLICE_BYTES + d * DIG_BYTES, bb,
                             &full[st]);
            }
            if (!ok) {   // the copies in flight land before the block may leave (bounded)
                atomicOr(status, STATUS_TIMEOUT);
                for (int i = max(0, issued - DSTAGE); i < issued; i++)
                    mbar_wait(&full[i % DSTAGE], (uint32_t)(i / DSTAGE) & 1u, SPIN_LIMIT);
            }
        }
    } else if (warp == D_EPI_WARPS) {
        if (lane == 0) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) |
                                   ((uint32_t)(DTM >> 4) << 24);   // bf16 x bf16 -> FP32, K-major, M = 128
            const int qmax = 256 / cw;                             // digits of B per MMA
            bool ok = true;
            for (int i = 0; i < n; i++) {
                const int st = i % DSTAGE;
                ok = mbar_wait(&full[st], (uint32_t)(i / DSTAGE) & 1u, SPIN_LIMIT);
                if (!ok) break;
                tc_fence_after();
                const uint32_t sa = smem_addr(smem + st * STAGE_BYTES);
                const uint64_t da = smem_desc(sa, 128, DSBO), db = smem_desc(sa + SLICE_BYTES, 128, DSBO);
#pragma unroll 1
                for (int p = 0; p < NDIG; p++) {
                    // digit p of A times the digits 0..7 - p of B, stacked along N: levels p..7, whose
                    // accumulators follow one another in tensor memory like the digits do in shared memory
                    for (int q = 0; q < NDIG - p; q += qmax) {
                        const int nq = min(qmax, NDIG - p - q);
                        mma_bf16(tmem + (uint32_t)((p + q) * cw), da + p * (DIG_BYTES >> 4), db + q * (cw * 2),
                                 idesc | ((uint32_t)(nq * cw >> 3) << 17), (p | i) ? 1u : 0u);
                    }
                    if (p)   // level 8 joins level 7
                        mma_bf16(tmem + (uint32_t)((NDIG - 1) * cw), da + p * (DIG_BYTES >> 4),
                                 db + (NDIG - p) * (cw * 2), idesc | ((uint32_t)(cw >> 3) << 17), 1u);
                }
                mma_commit(&empty[st]);
            }
            *ok_mma = ok ? 1 : 0;
            mma_commit(done);
            if (!ok) atomicOr(status, STATUS_TIMEOUT);
        }
    } else if (blockIdx.x == 0 && kc == 0) {
        for (int b = tid; b < nbin; b += 32 * D_EPI_WARPS)
            if (!column_fits(oct + (size_t)v * OCT * nbin + b, nbin, n_mock)) ecol[(size_t)v * nbin + b] = EXP_BAD;
    }
    __syncthreads();
    // every product has completed (bounded)
    const bool fin = mbar_wait(done, 0, SPIN_LIMIT);
    if (!fin && tid == 0) atomicOr(status, STATUS_TIMEOUT);
    if (fin && *ok_mma && warp < D_EPI_WARPS) {
        tc_fence_after();
        const int i = bi * DTM + (warp & 3) * 32 + lane, c0 = (warp >> 2) * (DTN / 2);
        longlong2 *t = T + ((size_t)kc * gridDim.y + v) * nbin * nbin;
#pragma unroll 1
        for (int c = c0; c < c0 + DTN / 2; c += 8) {
            if (c >= cw) break;   // uniform
            uint32_t r[8][8];
            tmem_ld8x8(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c, (uint32_t)cw, r);
#pragma unroll
            for (int q = 0; q < 8; q++) {
                // level l's accumulator holds its sum times 2^-7l
                long long hi = 0, lo = 0;
#pragma unroll
                for (int l = 0; l < 4; l++)
                    hi = hi * 128 + __float2int_rn(__uint_as_float(r[l][q]) * (float)(1u << (7 * l)));
#pragma unroll
                for (int l = 4; l < 7; l++)
                    lo = lo * 128 + __float2int_rn(__uint_as_float(r[l][q]) * 0x1p28f * (float)(1u << (7 * (l - 4))));
                lo = lo * 128 + __float2ll_rn(__uint_as_float(r[7][q]) * 0x1p49f);
                const int j = bj * DTN + c + q;
                if (i < nbin && j < nbin) t[(size_t)j * nbin + i] = make_longlong2(hi, lo);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 8 * DTN);
}

// Adds the segments of T (integers) and combines: NV = 3 the LC covariance
// (Eqs. R1R2, LCdef), NV = 1 the sample covariance into C_lc.  A block takes a
// 8 x 8 tile of the lower triangle, one variant per layer of threads (all of
// an element's loads in flight), and writes the tile and its mirror.  A tile
// with columns that are not split also sums its elements in float64: residuals
// of CK mocks at a time in shared memory (a quarter of a subtraction per
// multiply-add; the next ones' loads in flight), four chains of CK / 4 terms
// each, then one compensated addition (Knuth's two-sum) to the total, so a
// product goes through CK / 4 + 4 roundings however many mocks there are.
constexpr int CT = 8, CK = 32;
template <int NV>
__global__ void __launch_bounds__(CT *CT *NV)
    combine_digits_kernel(const longlong2 *__restrict__ T, int n_seg, int nbin, int n_mock,
                          const int *__restrict__ ecol, const double *__restrict__ mean,
                          const double *__restrict__ x0, const double *__restrict__ x1,
                          const double *__restrict__ x2, double inv, double two_ma, double M, CovOut out)
{
    __shared__ double sc[NV][CT][CT + 1], sh[5][CT][CT + 1], ys[NV][2][CK][CT];
    __shared__ int some[NV];   // elements of the variant are summed directly
    int tj = (int)((sqrtf(8.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
    while ((long long)tj * (tj + 1) / 2 > (long long)blockIdx.x) tj--;
    while ((long long)(tj + 1) * (tj + 2) / 2 <= (long long)blockIdx.x) tj++;
    const int ti = (int)((long long)blockIdx.x - (long long)tj * (tj + 1) / 2);   // tj >= ti
    const int v = threadIdx.x / (CT * CT), tx = threadIdx.x % CT, ty = threadIdx.x / CT % CT;
    const int i = ti * CT + tx, j = tj * CT + ty;
    const size_t nn = (size_t)nbin * nbin;
    const bool low = i < nbin && j < nbin && j >= i;
    double g = 0.0;
    bool bad = false;
    if (threadIdx.x < NV) some[threadIdx.x] = 0;
    if (low) {
        const int ei = ecol[(size_t)v * nbin + i], ej = ecol[(size_t)v * nbin + j];
        const longlong2 *t = T + (size_t)v * nn + (size_t)j * nbin + i;
        long long hi = 0, lo = 0;   // exact
#pragma unroll 8
        for (int k = 0; k < n_seg; k++) {
            const longlong2 u = t[(size_t)k * NV * nn];
            hi += u.x;
            lo += u.y;
        }
        bad = ei == EXP_BAD || ej == EXP_BAD;
        // hi: levels 0..3, units of 2^(ei + ej - 12 - 21); lo: levels 4..8, units of 2^(ei + ej - 12 - 49)
        if (!bad) g = fma((double)hi, 0x1p28, (double)lo) * __hiloint2double((1023 + ei + ej - 61) << 20, 0);
    }
    if (__syncthreads_or(bad)) {
        if (bad) some[v] = 1;
        __syncthreads();
        const bool mine = some[v] != 0, sums = __any_sync(0xffffffffu, bad);   // by layer, by warp
        const double *x = v == 0 ? x0 : (v == 1 ? x1 : x2);
        const int c0 = ti * CT + tx, c1 = tj * CT + tx;   // this thread's columns of the two sides
        const double m0 = c0 < nbin ? mean[(size_t)v * nbin + c0] : 0.0, m1 = c1 < nbin ? mean[(size_t)v * nbin + c1] : 0.0;
        constexpr int Q = CK / CT;   // mocks per thread and side
        double d0[Q] = {}, d1[Q] = {}, total = 0.0, rest = 0.0;
        auto load = [&](int k0) {
#pragma unroll
            for (int q = 0; q < Q; q++) {
                const int k = k0 + ty + CT * q;
                d0[q] = mine && k < n_mock && c0 < nbin ? x[(size_t)k * nbin + c0] : 0.0;
                d1[q] = mine && k < n_mock && c1 < nbin ? x[(size_t)k * nbin + c1] : 0.0;
            }
        };
        load(0);
        for (int k0 = 0; k0 < n_mock; k0 += CK) {
            if (mine) {
#pragma unroll
                for (int q = 0; q < Q; q++) {   // mocks past the last: zero
                    const bool in = k0 + ty + CT * q < n_mock;
                    ys[v][0][ty + CT * q][tx] = in ? d0[q] - m0 : 0.0;
                    ys[v][1][ty + CT * q][tx] = in ? d1[q] - m1 : 0.0;
                }
            }
            __syncthreads();
            if (k0 + CK < n_mock) load(k0 + CK);
            if (sums) {
                double a[4] = {0.0, 0.0, 0.0, 0.0};
                for (int k = 0; k < min(CK, n_mock - k0); k += 8)
#pragma unroll
                    for (int l = 0; l < 8; l++) a[l & 3] = fma(ys[v][0][k + l][tx], ys[v][1][k + l][ty], a[l & 3]);
                const double p = (a[0] + a[1]) + (a[2] + a[3]), t = total + p, z = t - total;
                rest += (total - (t - z)) + (p - z);
                total = t;
            }
            __syncthreads();
        }
        // (a total that is not finite has no compensation)
        if (bad) g = total - total == 0.0 ? total + rest : total;
    }
    if (low) sc[v][ty][tx] = g * inv;
    __syncthreads();
    if (v == 0 && low) {
        if (NV == 1) {
            sh[0][ty][tx] = sc[0][ty][tx];
        } else {
            const double ca = 0.5 * sc[0][ty][tx] + 0.5 * sc[NV / 3][ty][tx], cb = sc[NV - 1][ty][tx];
            const double a = 2.0 * cb - ca, bb = two_ma * (ca - cb);
            sh[0][ty][tx] = a + bb / M;
            sh[1][ty][tx] = ca;
            sh[2][ty][tx] = cb;
            sh[3][ty][tx] = a;
            sh[4][ty][tx] = bb;
        }
    }
    __syncthreads();
    const int ir = ti * CT + ty, jc = tj * CT + tx;   // the mirrored tile: rows i, columns j
    for (int q = v; q < (NV == 1 ? 1 : 5); q += NV) {
        double *o = out.p[q];
        if (!o) continue;
        if (j < nbin && i < nbin) o[(size_t)j * nbin + i] = j >= i ? sh[q][ty][tx] : sh[q][tx][ty];
        if (ti != tj && ir < nbin && jc < nbin) o[(size_t)ir * nbin + jc] = sh[q][tx][ty];
    }
}

struct DShape {
    int n_rb, n_cb, n_ks, pairs, spc, n_seg;
    size_t o_T, o_part, o_mean, o_e, o_oct, bytes;
};

DShape dshape(int n_mock, int nbin, int n_var, int n_sm)
{
    DShape s;
    s.n_rb = (nbin + DTM - 1) / DTM;
    s.n_cb = (nbin + DTN - 1) / DTN;
    s.n_ks = (n_mock + DKS - 1) / DKS;
    s.pairs = 0;
    for (int i = 0; i < s.n_rb; i++) s.pairs += std::max(0, s.n_cb - 2 * i);
    // segments: at least as many as exactness asks for, and as many as fill one
    // wave of one CTA per SM while a segment keeps at least six slices
    const long long least = (s.n_ks + SEG_SLICES - 1) / SEG_SLICES;
    const long long wave = std::max(1, n_sm) / ((long long)s.pairs * n_var);
    const long long want = std::max(least, std::min<long long>(wave, s.n_ks / 6));
    s.spc = (int)((s.n_ks + want - 1) / want);
    s.n_seg = (s.n_ks + s.spc - 1) / s.spc;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    s.o_T = al((size_t)n_var * s.n_rb * s.n_ks * SLICE_BYTES);
    s.o_part = s.o_T + al((size_t)s.n_seg * n_var * nbin * nbin * sizeof(longlong2));
    s.o_mean = s.o_part + al((size_t)n_var * COL_CHUNKS * nbin * sizeof(ColRange));
    s.o_e = s.o_mean + al((size_t)n_var * nbin * 8);
    s.o_oct = s.o_e + al((size_t)n_var * nbin * 4);
    s.bytes = s.o_oct + al((size_t)n_var * OCT * nbin * 4);
    return s;
}

}  // namespace

size_t cov_digits_work_bytes(int n_mock, int nbin, int n_var, int n_sm) { return dshape(n_mock, nbin, n_var, n_sm).bytes; }

// The faster float64 path (device and host time of an LC / a sample covariance of normal columns, this path against the
// tiled float64 kernel): 2 x 3 53 / 36 us against 67 / 50, 40 x 20 57 / 40 against 97 / 81, 301 x 60 67 / 50 against 144 /
// 127, 3500 x 200 112 / 61 against 1390 / 596, 40 x 1000 142 / 60 against 292 / 143.  Of columns of 3 to about 20 mocks 5 to
// 10 % are not split, which with many bins reaches nearly every tile of the combining kernel: 16 x 1000 168 / 68 against
// 162 / 78, 16 x 2000 441 / 148 against 378 / 120, 4 x 4000 1655 / 481 against 1261 / 318, 24 x 2000 356 / 110 against 557 /
// 184; those stay on the float64 kernel from 1000 bins on.  So do calls that would need more than 4 GiB of the larger
// workspace (16 bytes per residual and per element and segment of the Gram matrices).
bool cov_digits_suits(int n_mock, int nbin, int n_var, int n_sm)
{
    if (n_mock > 2 && n_mock < 20 && nbin > 1000) return false;
    const DShape s = dshape(n_mock, nbin, n_var, n_sm);
    return s.n_seg <= 65535 && s.bytes <= ((size_t)4 << 30);
}

cudaError_t launch_cov_digits(const double *x0, const double *x1, const double *x2, int n_var, int n_mock, int nbin,
                              void *work, int n_sm, int M_a, double M, double *C_lc, double *Ca, double *Cb,
                              double *A, double *B, int *status, cudaStream_t s)
{
    const DShape d = dshape(n_mock, nbin, n_var, n_sm);
    unsigned char *w = (unsigned char *)work;
    longlong2 *T = (longlong2 *)(w + d.o_T);
    double *mean = (double *)(w + d.o_mean);
    int *ecol = (int *)(w + d.o_e);
    ColRange *part = (ColRange *)(w + d.o_part);
    uint32_t *oct = (uint32_t *)(w + d.o_oct);
    cudaError_t e = launch_column_partials(x0, x1, x2, n_var, n_mock, nbin, part, oct, OCT, s);
    if (e != cudaSuccess) return e;
    digits_kernel<<<dim3((nbin + 31) / 32, COL_CHUNKS, n_var), 32 * COL_WARPS, 0, s>>>(x0, x1, x2, part, n_mock, nbin,
                                                                                      d.n_rb, d.n_ks, w, ecol, mean, oct);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int smem = digits_smem_bytes();
    e = cudaFuncSetAttribute(gram_digits_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    gram_digits_kernel<<<dim3(d.pairs, n_var, d.n_seg), D_THREADS, smem, s>>>(w, nbin, d.n_rb, d.n_cb, d.n_ks, d.spc,
                                                                             T, oct, n_mock, ecol, status);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long nt = (nbin + CT - 1) / CT;
    const unsigned nb = (unsigned)(nt * (nt + 1) / 2);
    const double inv = 1.0 / (double)(n_mock - 1), two_ma = 2.0 * (double)M_a;
    const CovOut out{{C_lc, Ca, Cb, A, B}};
    if (n_var == 3)
        combine_digits_kernel<3><<<nb, CT * CT * 3, 0, s>>>(T, d.n_seg, nbin, n_mock, ecol, mean, x0, x1, x2, inv,
                                                            two_ma, M, out);
    else
        combine_digits_kernel<1><<<nb, CT * CT, 0, s>>>(T, d.n_seg, nbin, n_mock, ecol, mean, x0, x1, x2, inv, two_ma,
                                                        M, out);
    return cudaGetLastError();
}

}  // namespace tpcf
