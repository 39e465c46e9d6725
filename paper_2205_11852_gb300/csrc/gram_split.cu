// Split-precision Gram products of the LC covariance on the 5th-generation
// tensor cores (tcgen05), Eqs. (bruteforce), (R1R2), (LCdef).
//
// The sample covariances need G_v = Y_v^T Y_v for the three centred
// correlation-function variants v (R1, R2, R1 u R2), Y_v = xi_v - mean_v of
// shape [n_mock][nbin].  Y is split into pieces that the tensor cores take
// exactly:
//   TF32X3: y = hi + lo (tf32 each), G ~ hi.hi + hi.lo + lo.hi         (3 products)
//   BF16X3: y = h + m + l (bf16 each), G ~ hh + hm + mh + hl + lh + mm  (6 products)
// A CTA (one per SM) owns one 128 x 128 output tile of one variant and a
// chunk of K-slices of 16 mocks: its operand tiles arrive by bulk copies
// (cp.async.bulk, the TMA engine, completing on mbarriers) into four stages,
// one thread issues each slice's tcgen05.mma chains into one of two FP32
// accumulator sets in tensor memory, and eight warps read each finished set
// back with tcgen05.ld and add it into sums in registers by compensated
// (Kahan) summation while the next slice multiplies; the sums become the
// chunk's partial Gram, and the combining kernel adds the chunks in float64,
// in chunk order.  The leading product (hi.hi) and the much smaller
// correction products go to two separate accumulators, so the FP32 rounding of
// an accumulator spans one slice's exact products and the corrections do not
// round against the leading sum.
//
// Operand tiles are written by the split kernel directly in the canonical
// K-major, non-swizzled layout of the tensor-core descriptors: 8-row x
// 16-byte core matrices, LBO = 128 bytes between core matrices along K and
// SBO = (32 * elem / 16) * 128 bytes between 8-row groups.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "colstats.cuh"
#include "tc_ptx.cuh"
#include "tpcf_internal.h"

namespace tpcf {
namespace {

constexpr int TM = 128;          // rows (bins) per tile, M = N of the MMA
constexpr int KS = 16;           // mocks per K-slice
constexpr int TMEM_COLS = 4 * TM; // two accumulator sets of (leading product, corrections)
constexpr int GRAM_EPI_WARPS = 8;  // the epilogue: warp w reads TMEM lanes 32 (w mod 4).. and columns half w / 4
constexpr int GRAM_THREADS = 32 * (GRAM_EPI_WARPS + 2);   // + one warp for the MMAs and one for the loads
static_assert(GRAM_EPI_WARPS == 8 && TM == 128, "two warpgroups split a 128-column tile (drain and store)");
constexpr int NSTAGE = 4;                    // K-slices in flight per CTA

template <int PREC>
struct Split;

template <>
struct Split<TPCF_TF32X3> {
    static constexpr int ELEM = 4;                           // bytes
    static constexpr int PIECES = 2;
    static constexpr int K_MMA = 8;                          // K per tcgen05.mma (kind::tf32)
    static constexpr int N_PROD = 3;
    // products hi.hi, hi.lo, lo.hi: piece of A and of B for product q
    __host__ __device__ static constexpr int pa(int q) { return q == 2 ? 1 : 0; }
    __host__ __device__ static constexpr int pb(int q) { return q == 1 ? 1 : 0; }
    static constexpr uint32_t FMT = 2;                       // TF32 operand format
};
template <>
struct Split<TPCF_BF16X3> {
    static constexpr int ELEM = 2;
    static constexpr int PIECES = 3;
    static constexpr int K_MMA = 16;                         // kind::f16
    static constexpr int N_PROD = 6;
    // products hh, hm, mh, hl, lh, mm
    __host__ __device__ static constexpr int pa(int q) { return q == 2 ? 1 : (q == 4 ? 2 : (q == 5 ? 1 : 0)); }
    __host__ __device__ static constexpr int pb(int q) { return q == 1 ? 1 : (q == 3 ? 2 : (q == 5 ? 1 : 0)); }
    static constexpr uint32_t FMT = 1;                       // BF16 operand format
};

template <int PREC>
__host__ __device__ constexpr int tile_bytes() { return TM * KS * Split<PREC>::ELEM; }

template <int PREC>
__host__ __device__ constexpr int sbo_bytes() { return (KS * Split<PREC>::ELEM / 16) * 128; }

// byte offset of element (row r, k) inside a K-major non-swizzled tile
template <int PREC>
__device__ __forceinline__ uint32_t tile_offset(int r, int k)
{
    constexpr int per = 16 / Split<PREC>::ELEM;              // elements per core-matrix row
    return (uint32_t)((r >> 3) * sbo_bytes<PREC>() + (k / per) * 128 + (r & 7) * 16 + (k % per) * Split<PREC>::ELEM);
}

__device__ __forceinline__ uint32_t tf32_rna(float x)
{
    uint32_t y;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(y) : "f"(x));
    return y;
}

// The splits of a residual, on the integer pipes where its exponent allows
// (|d| in [2^-74, 2^126]; the float64 pipe, one to two operations per clock
// and SM with its conversions, bounded the split kernel: 30 us at 3500 x 200).
// The remainders stay exact integers in units of d's last place, so the pieces
// equal those of float64 subtractions and conversions bit for bit.
struct Int64Parts {
    bool plain;       // the integer path applies
    int sign;         // 0x80000000 for a negative d
    uint32_t ex;      // biased float64 exponent
    long long m;      // 53-bit magnitude
    float ulp;        // weight of m's last bit

    __device__ __forceinline__ explicit Int64Parts(double d)
    {
        const unsigned long long b = (unsigned long long)__double_as_longlong(d);
        ex = (uint32_t)(b >> 52) & 0x7ffu;
        plain = ex - 949u <= 200u;
        sign = (int)((uint32_t)(b >> 32) & 0x80000000u);
        m = (long long)((b & 0xfffffffffffffull) | (1ull << 52));
        ulp = __uint_as_float((ex - 948u) << 23);
    }
};

// hi = rna_tf32((float)d), lo = rna_tf32((float)(d - hi))
__device__ __forceinline__ void split_tf32(double d, uint32_t &hi, uint32_t &lo)
{
    const Int64Parts q(d);
    if (!q.plain) {
        hi = tf32_rna((float)d);
        lo = tf32_rna((float)(d - (double)__uint_as_float(hi)));
        return;
    }
    // the float nearest to |d| (ties to even)
    const unsigned long long u = (unsigned long long)q.m + 0x0fffffffull + (((unsigned long long)q.m >> 29) & 1ull);
    const uint32_t h = tf32_rna(__uint_as_float((uint32_t)(u >> 29) + ((q.ex - 897u) << 23)));
    const long long r = q.m - ((long long)((h & 0x7fffffu) | 0x800000u) << ((h >> 23) - q.ex + 925u));
    hi = h | (uint32_t)q.sign;
    lo = tf32_rna(__ll2float_rn(r) * q.ulp) ^ (uint32_t)q.sign;
}

// three bf16 pieces, each the nearest to the remainder of the ones before
__device__ __forceinline__ void split_bf16(double d, uint16_t (&p)[3])
{
    const Int64Parts q(d);
    if (!q.plain) {
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const __nv_bfloat16 t = __double2bfloat16(d);
            d -= (double)__bfloat162float(t);
            p[k] = __bfloat16_as_ushort(t);
        }
        return;
    }
    long long r = q.m;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        // truncated to a float with a sticky last bit, which bf16 then rounds correctly
        const float f = __ll2float_rz(r);
        const uint32_t sticky = __float2ll_rz(f) != r ? 1u : 0u;
        const float t = __bfloat162float(__float2bfloat16_rn(__uint_as_float(__float_as_uint(f) | sticky)));
        r -= __float2ll_rz(t);   // exact: t has no bits below r's last place
        p[k] = (uint16_t)((__float_as_uint(t * q.ulp) ^ (uint32_t)q.sign) >> 16);
    }
}

// centred residuals, split into pieces, written as operand tiles
// tiles[v][piece][rb][ks].  A block takes 32 columns (one per lane) and one of
// COL_CHUNKS row ranges of one variant, closes the column statistics of all
// row ranges (colstats.cuh) and writes whole 16-byte core-matrix rows: `per`
// consecutive mocks of one bin.  Rows past nbin are left unwritten (an output
// element depends on its own two operand rows only), mocks past n_mock are
// zeros.
template <int PREC>
__global__ void __launch_bounds__(32 * COL_WARPS)
    split_kernel(const double *__restrict__ x0, const double *__restrict__ x1, const double *__restrict__ x2,
                 const ColSum *__restrict__ part, int n_mock, int nbin, int n_rb, int n_ks,
                 unsigned char *__restrict__ tiles)
{
    constexpr int TB = tile_bytes<PREC>();
    constexpr int NP = Split<PREC>::PIECES;
    constexpr int per = 16 / Split<PREC>::ELEM;
    const int v = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double *x = v == 0 ? x0 : (v == 1 ? x1 : x2);
    const int b = blockIdx.x * 32 + lane;
    double mu;
    column_stats(part, v, n_mock, nbin, b, mu);
    if (b >= nbin) return;
    const int rb = b / TM, r = b % TM;
    const int n_g = n_ks * (KS / per), share = (n_g + (int)gridDim.y - 1) / (int)gridDim.y;
    const int g1 = min(n_g, ((int)blockIdx.y + 1) * share);
#pragma unroll 2
    for (int g = (int)blockIdx.y * share + warp; g < g1; g += COL_WARPS) {
        const int m0 = g * per, ks = m0 / KS;
        double y[per];
#pragma unroll
        for (int k = 0; k < per; k++) y[k] = m0 + k < n_mock ? x[(size_t)(m0 + k) * nbin + b] : mu;
        uint32_t w[NP][4];
        if (PREC == TPCF_TF32X3) {
#pragma unroll
            for (int k = 0; k < per; k++) {
                const double d = m0 + k < n_mock ? y[k] - mu : 0.0;
                split_tf32(d, w[0][k], w[1][k]);
            }
        } else {
            uint16_t h[per][3];
#pragma unroll
            for (int k = 0; k < per; k++) split_bf16(m0 + k < n_mock ? y[k] - mu : 0.0, h[k]);
#pragma unroll
            for (int p = 0; p < NP; p++)
#pragma unroll
                for (int k = 0; k < 4; k++)
                    w[p][k] = (uint32_t)h[(2 * k) % per][p] | (uint32_t)h[(2 * k + 1) % per][p] << 16;
        }
        const uint32_t off = tile_offset<PREC>(r, m0 % KS);
#pragma unroll
        for (int p = 0; p < NP; p++)
            *(uint4 *)(tiles + ((((size_t)v * NP + p) * n_rb + rb) * n_ks + ks) * TB + off) =
                make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
    }
}

template <int PREC>
__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    if (PREC == TPCF_TF32X3) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
            "l"(a), "l"(b), "r"(idesc), "r"(acc)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
            "l"(a), "l"(b), "r"(idesc), "r"(acc)
            : "memory");
    }
}

// instruction descriptor: FP32 accumulate, K-major A and B, M = N = 128
template <int PREC>
__host__ __device__ constexpr uint32_t instr_desc()
{
    return (1u << 4)                          // D format: F32
           | (Split<PREC>::FMT << 7)          // A format
           | (Split<PREC>::FMT << 10)         // B format
           | ((uint32_t)(TM >> 3) << 17)      // N / 8
           | ((uint32_t)(TM >> 4) << 24);     // M / 16
}

template <int PREC>
__host__ __device__ constexpr int stage_bytes() { return 2 * Split<PREC>::PIECES * tile_bytes<PREC>(); }

// shared memory: NSTAGE stages | full[NSTAGE], empty[NSTAGE], accf[2], accfree[2], done barriers | TMEM slot | flag
template <int PREC>
constexpr int gram_smem_bytes() { return NSTAGE * stage_bytes<PREC>() + 8 * (2 * NSTAGE + 5) + 16; }

// 16 columns of both accumulators of a set, complete on return
__device__ __forceinline__ void tmem_ld16x2(uint32_t t, uint32_t (&lo)[16], uint32_t (&hi)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, "
        "%29, %30, %31}, [%33];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(lo[0]), "=r"(lo[1]), "=r"(lo[2]), "=r"(lo[3]), "=r"(lo[4]), "=r"(lo[5]), "=r"(lo[6]), "=r"(lo[7]),
          "=r"(lo[8]), "=r"(lo[9]), "=r"(lo[10]), "=r"(lo[11]), "=r"(lo[12]), "=r"(lo[13]), "=r"(lo[14]),
          "=r"(lo[15]), "=r"(hi[0]), "=r"(hi[1]), "=r"(hi[2]), "=r"(hi[3]), "=r"(hi[4]), "=r"(hi[5]), "=r"(hi[6]),
          "=r"(hi[7]), "=r"(hi[8]), "=r"(hi[9]), "=r"(hi[10]), "=r"(hi[11]), "=r"(hi[12]), "=r"(hi[13]),
          "=r"(hi[14]), "=r"(hi[15])
        : "r"(t), "r"(t + TM)
        : "memory");
}

// One CTA (one per SM): output tile (bi, bj) of variant v over the K-slices
// [k0, k0 + n) of chunk kc.  Warp 9 keeps NSTAGE slices of operand tiles in
// flight (bulk copies completing on full[stage]); warp 8 issues each slice's
// MMA chain into accumulator set i % 2 of tensor memory (columns 256 (i % 2) +
// [0, 128): leading product, + [128, 256): corrections), once the epilogue has
// drained that set's previous slice (accfree).  Warps 0-7 (TMEM lanes = tile
// rows, two halves of the columns) read each finished set (accf) and add its
// two accumulators into 64 register sums per thread by compensated (Kahan)
// FP32 summation (the FP64 pipe is too slow for this on the SMs), so the sums
// hold the chunk to about one FP32 rounding while the tensor cores work on
// slice i + 1.  At the end D(row i, column j) goes to P[kc][v][j][i], 32
// consecutive doubles per warp.
//
// The drain bounds it: per slice 2 x 16384 accumulator values against 8
// additions each.  With the sums in shared memory (16 bytes of traffic per
// element and slice) and the loads issued by the MMA thread only after the
// slice's products had finished, the kernel took 46 us (3500 x 200, TF32x3),
// now 31 us; the whole covariance 129 -> 69 us.
//
// Every wait is bounded.  The epilogue's waits for the products give up after
// done_limit polls (a context option); skip_mma (tests only) makes CTA
// (0, 0, 0) wait for its first loads and then issue no MMA and no commit, so
// that this wait runs out with no copy or MMA in flight.
template <int PREC>
__global__ void __launch_bounds__(GRAM_THREADS, 1) gram_tc_kernel(const unsigned char *__restrict__ tiles, int nbin,
                                                                 int n_rb, int n_ks, int spc, double *__restrict__ P,
                                                                 int *__restrict__ status, long long done_limit,
                                                                 int skip_mma)
{
    constexpr int TB = tile_bytes<PREC>();
    constexpr int NP = Split<PREC>::PIECES;
    constexpr int SB = stage_bytes<PREC>();
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *full = (uint64_t *)(smem + NSTAGE * SB);
    uint64_t *empty = full + NSTAGE;
    uint64_t *accf = empty + NSTAGE;
    uint64_t *accfree = accf + 2;
    uint64_t *done = accfree + 2;
    uint32_t *slot = (uint32_t *)(done + 1);
    int *all_in = (int *)(slot + 1);   // every slice was multiplied

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // blockIdx.x enumerates the upper-triangle tile pairs (bi <= bj) row by row
    int bi = 0, rest = (int)blockIdx.x;
    while (rest >= n_rb - bi) {
        rest -= n_rb - bi;
        bi++;
    }
    const int bj = bi + rest;
    const int v = blockIdx.y, kc = blockIdx.z;
    const int k0 = kc * spc, n = min(n_ks, k0 + spc) - k0;   // n >= 1 by the host's chunking
    const bool skip = skip_mma && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;

    if (warp == 0) tmem_alloc(slot, TMEM_COLS);
    if (tid == 0) {
        for (int i = 0; i < NSTAGE; i++) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        for (int k = 0; k < 2; k++) {
            mbar_init(&accf[k], 1);
            mbar_init(&accfree[k], GRAM_EPI_WARPS);
        }
        mbar_init(done, 1);
        mbar_fence_init();
        *all_in = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *slot;
    bool fine = true;
    float sum[TM / 2], cmp[TM / 2];   // the epilogue's column half of this thread's row

    if (warp == GRAM_EPI_WARPS + 1) {
        if (lane == 0) {
            const int n_load = skip ? min(NSTAGE, n) : n;
            int issued = 0;
            bool ok = true;
            for (; issued < n_load; issued++) {   // the operand tiles of slice k0 + issued
                const int st = issued % NSTAGE;
                if (issued >= NSTAGE) {
                    ok = mbar_wait(&empty[st], (uint32_t)(issued / NSTAGE - 1) & 1u, SPIN_LIMIT);
                    if (!ok) break;
                }
                unsigned char *sa = smem + st * SB, *sb = sa + NP * TB;
                mbar_expect_tx(&full[st], (uint32_t)SB);
                for (int p = 0; p < NP; p++) {
                    const size_t base = ((size_t)v * NP + p) * n_rb;
                    bulk_g2s(sa + p * TB, tiles + ((base + bi) * n_ks + k0 + issued) * TB, TB, &full[st]);
                    bulk_g2s(sb + p * TB, tiles + ((base + bj) * n_ks + k0 + issued) * TB, TB, &full[st]);
                }
            }
            if (!ok) {   // the copies in flight land before the block may leave (bounded)
                atomicOr(status, STATUS_TIMEOUT);
                for (int i = max(0, issued - NSTAGE); i < issued; i++)
                    mbar_wait(&full[i % NSTAGE], (uint32_t)(i / NSTAGE) & 1u, SPIN_LIMIT);
            }
        }
    } else if (warp == GRAM_EPI_WARPS) {
        if (lane == 0) {
            bool ok = true;
            for (int i = 0; i < n; i++) {
                if (skip && i == NSTAGE) break;
                ok = mbar_wait(&full[i % NSTAGE], (uint32_t)(i / NSTAGE) & 1u, SPIN_LIMIT);
                if (!ok) break;
                if (skip) continue;
                // accumulator set i % 2 is free once the epilogue has drained slice i - 2
                if (i >= 2) {
                    ok = mbar_wait(&accfree[i % 2], (uint32_t)((i - 2) / 2) & 1u, SPIN_LIMIT);
                    if (!ok) break;
                }
                tc_fence_after();
                constexpr uint32_t idesc = instr_desc<PREC>();
                constexpr int steps = KS / Split<PREC>::K_MMA;
                const uint32_t sa = smem_addr(smem + (i % NSTAGE) * SB), sb = sa + NP * TB;
                const uint32_t set = tmem + (uint32_t)((i % 2) * 2 * TM);
#pragma unroll
                for (int q = 0; q < Split<PREC>::N_PROD; q++) {
                    const uint32_t a0 = sa + Split<PREC>::pa(q) * TB;
                    const uint32_t b0 = sb + Split<PREC>::pb(q) * TB;
#pragma unroll
                    for (int st = 0; st < steps; st++) {
                        // each MMA step covers two core matrices along K (2 x 128 bytes); product 0
                        // accumulates in the set's columns [0, 128), the others in [128, 256); the first
                        // step of each accumulator overwrites it
                        const uint64_t da = smem_desc(a0 + st * 256, 128, sbo_bytes<PREC>());
                        const uint64_t db = smem_desc(b0 + st * 256, 128, sbo_bytes<PREC>());
                        const uint32_t d = set + (q == 0 ? 0u : (uint32_t)TM);
                        const bool init = st == 0 && (q == 0 || q == 1);
                        mma<PREC>(d, da, db, idesc, init ? 0u : 1u);
                    }
                }
                mma_commit(&empty[i % NSTAGE]);
                mma_commit(&accf[i % 2]);
            }
            *all_in = (ok && !skip) ? 1 : 0;
            if (!skip) mma_commit(done);   // also when a wait gave up: what was issued completes before TMEM is freed
            if (!ok) atomicOr(status, STATUS_TIMEOUT);
        }
    } else {
        // epilogue: row = this thread's TMEM lane; the two warpgroups take the
        // columns [0, TM / 2) and [TM / 2, TM) of both accumulators
        const uint32_t lane0 = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * (TM / 2));
#pragma unroll
        for (int c = 0; c < TM / 2; c++) sum[c] = cmp[c] = 0.0f;
        for (int i = 0; i < n && fine; i++) {
            fine = mbar_wait(&accf[i % 2], (uint32_t)(i / 2) & 1u, done_limit);
            if (!fine) {
                fine = mbar_wait(&accf[i % 2], (uint32_t)(i / 2) & 1u, done_limit);
                if (!fine) break;
            }
            tc_fence_after();
#pragma unroll
            for (int c0 = 0; c0 < TM / 2; c0 += 16) {
                uint32_t lo[16], hi[16];
                tmem_ld16x2(lane0 + (uint32_t)((i % 2) * 2 * TM + c0), lo, hi);
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    // two compensated additions (the leading product, then the corrections)
                    float sm = sum[c0 + j], cp = cmp[c0 + j];
                    float y = __fsub_rn(__uint_as_float(lo[j]), cp);
                    float t = __fadd_rn(sm, y);
                    cp = __fsub_rn(__fsub_rn(t, sm), y);
                    sm = t;
                    y = __fsub_rn(__uint_as_float(hi[j]), cp);
                    t = __fadd_rn(sm, y);
                    cmp[c0 + j] = __fsub_rn(__fsub_rn(t, sm), y);
                    sum[c0 + j] = t;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&accfree[i % 2]);
        }
        if (!fine && lane == 0) atomicOr(status, STATUS_TIMEOUT);
    }
    __syncthreads();
    // every product has completed before tensor memory is released (bounded)
    bool good = *all_in != 0;
    if (!skip) {
        bool fin = mbar_wait(done, 0, done_limit);
        if (!fin) fin = mbar_wait(done, 0, done_limit);
        good = good && fin;
    }
    if (!good && tid == 0) atomicOr(status, STATUS_TIMEOUT);
    if (good && fine && warp < GRAM_EPI_WARPS) {
        double *g = P + ((size_t)kc * gridDim.y + v) * nbin * nbin;
        const int row = bi * TM + (warp & 3) * 32 + lane, col0 = bj * TM + (warp >> 2) * (TM / 2);
        if (row < nbin) {
#pragma unroll
            for (int c = 0; c < TM / 2; c++)
                if (col0 + c < nbin) g[(size_t)(col0 + c) * nbin + row] = (double)sum[c] - (double)cmp[c];
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

// Adds the chunks' partials in chunk order (float64, deterministic) and
// combines: NV = 3 the LC covariance (Eqs. R1R2, LCdef), NV = 1 the sample
// covariance into out.p[0].  P[kc][v][j][i] = D(i, j) for the 128-tiles
// (i, j) with i's tile <= j's tile; an element below the diagonal tiles is the
// mirror of the one above.  A block takes an 8 x 8 tile (r in [8 tr, +8), c in
// [8 tc, +8), tc >= tr; with 16 x 16 the 91 blocks of 200 bins left SMs idle
// under the float64 additions: 20 us), one variant per layer of threads, and writes it
// and its mirror.
constexpr int CT = 8;
template <int NV>
__global__ void __launch_bounds__(CT *CT *NV) combine_partials_kernel(const double *__restrict__ P, int n_kc, int nbin,
                                                                     int n_mock, int M_a, double M, CovOut out)
{
    __shared__ double sc[NV][2][CT][CT + 1];
    int tc = (int)((sqrtf(8.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
    while ((long long)tc * (tc + 1) / 2 > (long long)blockIdx.x) tc--;
    while ((long long)(tc + 1) * (tc + 2) / 2 <= (long long)blockIdx.x) tc++;
    const int tr = (int)((long long)blockIdx.x - (long long)tc * (tc + 1) / 2);   // tr <= tc
    const int v = threadIdx.x / (CT * CT), tx = threadIdx.x % CT, ty = threadIdx.x / CT % CT;
    const size_t nn = (size_t)nbin * nbin;
    const double inv = 1.0 / (double)(n_mock - 1);
    const bool same = tr / (TM / CT) == tc / (TM / CT);   // inside a diagonal 128-tile: both triangles are stored
#pragma unroll
    for (int h = 0; h < 2; h++) {   // h = 0: D(row r, column c); 1: D(row c, column r), inside a diagonal tile only
        if (h && (!same || tr == tc)) break;
        const int i = (h ? tc : tr) * CT + tx, j = (h ? tr : tc) * CT + ty;
        double acc = 0.0;
        if (i < nbin && j < nbin) {
            const double *p = P + (size_t)v * nn + (size_t)j * nbin + i;
#pragma unroll 8
            for (int k = 0; k < n_kc; k++) acc += p[(size_t)k * NV * nn];
        }
        sc[v][h][ty][tx] = acc * inv;   // [column][row]
    }
    __syncthreads();
    // out(row, col): tile (tr, tc) from h = 0 transposed; tile (tc, tr) from h = 1 transposed, or the mirror of h = 0
    for (int w = v; w < 2; w += NV) {
        if (w && tr == tc) break;
        const int row = (w ? tc : tr) * CT + ty, col = (w ? tr : tc) * CT + tx;
        if (row >= nbin || col >= nbin) continue;
        double c[3];
#pragma unroll
        for (int q = 0; q < NV; q++) c[q] = w == 0 ? sc[q][0][tx][ty] : (same ? sc[q][1][tx][ty] : sc[q][0][ty][tx]);
        const size_t t = (size_t)row * nbin + col;
        if (NV == 1) {
            out.p[0][t] = c[0];
            continue;
        }
        const double ca = 0.5 * c[0] + 0.5 * c[NV / 3], cb = c[NV - 1];
        const double a = 2.0 * cb - ca;
        const double bb = 2.0 * (double)M_a * (ca - cb);
        out.p[0][t] = a + bb / M;
        if (out.p[1]) out.p[1][t] = ca;
        if (out.p[2]) out.p[2][t] = cb;
        if (out.p[3]) out.p[3][t] = a;
        if (out.p[4]) out.p[4][t] = bb;
    }
}

// K-chunking of the Gram grid: n_kc chunks of spc slices each, as many as fit
// in one wave (one CTA per SM: 512 TMEM columns and ~200 KB of shared memory
// each; one CTA more than the SMs would run a second wave of one CTA and
// double the kernel's time); the FP32 rounding spans one 16-mock slice
// whatever the chunk length.  The partials then take at most about n_sm x 2 TM^2 x 8 bytes
// (n_kc x n_var x nbin^2 doubles with n_kc ~ n_sm / (n_var x tile pairs)).
struct Chunking {
    int spc, n_kc;
};

Chunking chunking(int n_mock, int nbin, int n_var, int n_sm)
{
    const int n_rb = (nbin + TM - 1) / TM, n_ks = (n_mock + KS - 1) / KS;
    const long long np = (long long)n_rb * (n_rb + 1) / 2;
    long long want = std::max<long long>(1, (long long)std::max(1, n_sm) / (np * n_var));
    want = std::min<long long>(want, n_ks);
    const int spc = (int)((n_ks + want - 1) / want);
    return Chunking{spc, (n_ks + spc - 1) / spc};
}

template <int PREC>
size_t tiles_bytes(int n_mock, int nbin, int n_var)
{
    const size_t n_rb = (nbin + TM - 1) / TM, n_ks = (n_mock + KS - 1) / KS;
    return (size_t)n_var * Split<PREC>::PIECES * n_rb * n_ks * tile_bytes<PREC>();
}

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

template <int PREC>
size_t work_bytes_of(int n_mock, int nbin, int n_var, int n_sm)
{
    const Chunking c = chunking(n_mock, nbin, n_var, n_sm);
    const size_t g = (size_t)n_var * nbin * nbin * 8;
    return al256(tiles_bytes<PREC>(n_mock, nbin, n_var)) + al256((size_t)c.n_kc * g) +
           al256((size_t)n_var * COL_CHUNKS * nbin * sizeof(ColSum));
}

// n_var = 3: the LC covariance of (x0, x1, x2); n_var = 1: the sample covariance of x0 into C_lc
template <int PREC>
cudaError_t run(const double *x0, const double *x1, const double *x2, int n_var, int n_mock, int nbin, void *work,
                size_t work_bytes, int M_a, double M, double *C_lc, double *Ca, double *Cb, double *A, double *B,
                int *status, const GramOpts &opt, cudaStream_t s)
{
    const int n_rb = (nbin + TM - 1) / TM, n_ks = (n_mock + KS - 1) / KS;
    if (n_rb > 90) return cudaErrorInvalidValue;
    const Chunking ch = chunking(n_mock, nbin, n_var, opt.n_sm);
    if (ch.n_kc > 65535) return cudaErrorInvalidValue;
    unsigned char *w = (unsigned char *)work;
    unsigned char *tiles = w;
    const size_t g = (size_t)n_var * nbin * nbin;
    size_t o = al256(tiles_bytes<PREC>(n_mock, nbin, n_var));
    double *P = (double *)(w + o);
    o += al256((size_t)ch.n_kc * g * 8);
    ColSum *part = (ColSum *)(w + o);
    o += al256((size_t)n_var * COL_CHUNKS * nbin * sizeof(ColSum));
    if (o > work_bytes) return cudaErrorInvalidValue;
    cudaError_t e = launch_column_partials(x0, x1, x2, n_var, n_mock, nbin, part, nullptr, 0, s);
    if (e != cudaSuccess) return e;
    split_kernel<PREC><<<dim3((nbin + 31) / 32, COL_CHUNKS, n_var), 32 * COL_WARPS, 0, s>>>(x0, x1, x2, part, n_mock,
                                                                                           nbin, n_rb, n_ks, tiles);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int np = n_rb * (n_rb + 1) / 2;   // upper-triangle tile pairs
    const int smem = gram_smem_bytes<PREC>();
    e = cudaFuncSetAttribute(gram_tc_kernel<PREC>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    gram_tc_kernel<PREC><<<dim3(np, n_var, ch.n_kc), GRAM_THREADS, smem, s>>>(
        tiles, nbin, n_rb, n_ks, ch.spc, P, status, opt.wait_limit > 0 ? opt.wait_limit : SPIN_LIMIT,
        opt.test_skip_mma);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long nt = (nbin + CT - 1) / CT;
    const unsigned nb = (unsigned)(nt * (nt + 1) / 2);
    const CovOut out{{C_lc, Ca, Cb, A, B}};
    if (n_var == 3)
        combine_partials_kernel<3><<<nb, CT * CT * 3, 0, s>>>(P, ch.n_kc, nbin, n_mock, M_a, M, out);
    else
        combine_partials_kernel<1><<<nb, CT * CT, 0, s>>>(P, ch.n_kc, nbin, n_mock, M_a, M, out);
    return cudaGetLastError();
}

}  // namespace

size_t lc_split_work_bytes(int n_mock, int nbin, int precision, int n_sm, int n_var)
{
    return precision == TPCF_BF16X3 ? work_bytes_of<TPCF_BF16X3>(n_mock, nbin, n_var, n_sm)
                                    : work_bytes_of<TPCF_TF32X3>(n_mock, nbin, n_var, n_sm);
}

cudaError_t launch_lc_split(const double *xi_a1, const double *xi_a2, const double *xi_b, int n_mock, int nbin,
                            int precision, void *work, size_t work_bytes, int M_a, double M, double *C_lc,
                            double *Ca, double *Cb, double *A, double *B, int *status, const GramOpts &opt,
                            cudaStream_t s)
{
    if (precision == TPCF_TF32X3)
        return run<TPCF_TF32X3>(xi_a1, xi_a2, xi_b, 3, n_mock, nbin, work, work_bytes, M_a, M, C_lc, Ca, Cb, A, B,
                                status, opt, s);
    if (precision == TPCF_BF16X3)
        return run<TPCF_BF16X3>(xi_a1, xi_a2, xi_b, 3, n_mock, nbin, work, work_bytes, M_a, M, C_lc, Ca, Cb, A, B,
                                status, opt, s);
    return cudaErrorNotSupported;
}

cudaError_t launch_cov_split(const double *xi, int n_mock, int nbin, int precision, void *work, size_t work_bytes,
                             double *C, int *status, const GramOpts &opt, cudaStream_t s)
{
    if (precision == TPCF_TF32X3)
        return run<TPCF_TF32X3>(xi, xi, xi, 1, n_mock, nbin, work, work_bytes, 1, 2.0, C, nullptr, nullptr,
                                nullptr, nullptr, status, opt, s);
    if (precision == TPCF_BF16X3)
        return run<TPCF_BF16X3>(xi, xi, xi, 1, n_mock, nbin, work, work_bytes, 1, 2.0, C, nullptr, nullptr,
                                nullptr, nullptr, status, opt, s);
    return cudaErrorNotSupported;
}

}  // namespace tpcf
