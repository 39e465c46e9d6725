// Direct binned pair counting on the chaining mesh (Sect. 2.1: DD, DR_i and
// RR_i counts; Sect. 4.3: bins in separation s and in mu) for linear s bins
// starting at 0: s only, mu with the line of sight along x, or mu with the
// line of sight from the observer to the pair's midpoint (cut-sky mocks); and
// for geometric (logarithmic) s bins: s only, or mu along x.
//
// Work decomposition.  A unit is a chunk of at most 64 sorted points of one
// mesh cell A, or of a few cells in a row along x where the cells hold few
// points, paired with the neighbourhood of A in catalogue b.  Each warp
// owns a unit on its own: it stages the a-chunk in its region of shared
// memory, streams the b-points of the neighbourhood (the self cell of an
// auto count as it is, every other neighbour cell through a filter that
// keeps a point only if its distance to the a-chunk's bounding box is below
// the last edge) into its own buffer, and counts every full tile of 128
// b-points (4 per lane) against the a-chunk as soon as it is there.  The
// warps of a block share one to four histogram tables, one per term, and pass
// from one term to the next without waiting for each other (see
// pairdirect_kernel).  The code that few units need (locks, drains, rechecks)
// keeps its loops rolled: with warps at different places the instruction cache
// is what a larger kernel pays with (104 KB of code instead of 67: 4 % on cut-sky
// mocks, 13 % on small ones).
//
// Arithmetic.  Coordinates are exact integer offsets from A's lower corner,
// converted once to FP32 in units of one s bin, so the s bin of a pair is
// floor(u) with u its FP32 separation.  Two pairs run side by side in packed
// FP32 (f32x2) arithmetic.  Per pair: d2 from the differences, r = rsqrt(d2)
// (MUFU), S = floor(d2 r) by one round-toward-zero FMA onto a power-of-two
// offset, the residual d2 r - floor(d2 r) - 1/2 by one more FMA, and the
// signed mu bin T = floor(n_mu dx r) at both ends of the error interval
// [n_mu dx - m, n_mu dx + m] r.  A pair is certain when its s residual lies
// within cs of 1/2 and both mu floors agree; cs and m come from a rigorous
// bound on the FP32 errors (plan.cpp).  Every pair, certain or not, is added
// to the histogram at (S, T-) with one shared-memory atomic; a pair at or
// beyond the last edge lands in the histogram's spare last row.  The check
// costs two compares per pair, or-ed into one predicate per a-point; an
// a-point with an uncertain pair in any lane takes the rare path, which
// recomputes its pairs with a flag each, takes back the uncertain ones' adds
// and rechecks them exactly from the integer coordinates (64-bit squared
// distances, a 128-bit mu test), 32 at a time, so every count equals the
// integer definition bit for bit.  With the midpoint line of sight the mu
// bin comes from l = a + b - 2 o (o the observer), mu = (l.d) r rl with
// rl = rsqrt(|l|^2), its floor and residual against a per-pair bound
// c2 + c1 r + c3 rl (plan.cpp), the rest as above.
//
// Geometric s bins: coordinates in units of the edge that one more bin below
// the first would have, so that S = floor(A l) with l = log2(d2) (MUFU) and A
// = 1 / (2 log2 of the edges' ratio) is the bin plus one, and row 0 takes the
// pairs below the first edge.  l is held above lmid, where A l is either
// a whole number (a pair below that bin, where FP32 errors are large against
// a bin, is always rechecked) or 1/2 (a pair that far below the first
// edge is certain to miss), whichever leaves fewer pairs to recheck.  Three mocks of
// 100 000 points, 24 bins from 0.75 to 150 Mpc/h: 4.81 ms by the general counter, 2.93 so
// (eight pairs in 10^4 rechecked).
//
// Fine mu bins along x (the signed table of mode 1 would not fit): one copy of a
// table with a column per |mu| bin, T from |n_mu dx|, rows a whole number of
// columns apart.  Two lanes seldom meet in one of so many bins, and the
// banks they fall in are as good as random (about three adds in the fullest).
// T- below column -1 only occurs in row 0 and only for uncertain pairs, whose
// adds are taken back: FOLD_PAD words before the table take them.
// 155 250 points in a slab, 200 x 100 bins: 13.06 ms by the general counter, 6.28 so
// (one table per block; 10 pairs in 10^4 rechecked).
//
// Histogram.  R copies of a (n_s + 1) x C table of 32-bit counters, lane l
// adding to copy l mod R, so the 32 adds of a warp fall in distinct banks
// (R = 32) or at most two (R = 16) or four (R = 8) per bank.  mu is binned by sign, C =
// 2 n_mu + 2 columns from -n_mu - 1 to n_mu, and folded to |mu| when a table is
// drained into the term's int64 histogram: when the block's last warp leaves
// the term, or before its 32-bit counters could wrap.
#include "pair_device.cuh"

namespace tpcf {

namespace {

constexpr int NP = 4;               // b-points per lane
constexpr int NQ = NP / 2;          // packed pairs per lane
constexpr int TB = 32 * NP;         // b-points per tile
constexpr int BUF = TB + 128;       // per-warp b buffer: a tile plus one filter pass
constexpr int XCAP = 96;            // per-warp list of pairs awaiting the exact recheck
constexpr float MAG_S = 8388608.0f;       // 2^23: fma.rz(d2, r, MAG_S) = 2^23 + floor(d2 r) for 0 <= d2 r < 2^23
constexpr uint32_t MAG_S_BITS = 0x4B000000u;
constexpr float MAG_T = 12582912.0f;      // 1.5 * 2^23: = 1.5 * 2^23 + floor(t) for |t| < 2^22
constexpr uint32_t MAG_T_BITS = 0x4B400000u;
constexpr float FAR = 1.0e5f;             // a padding b-point: far beyond every edge, still finite
static_assert(DIRECT_ACHUNK % 32 == 0 && DIRECT_ACHUNK <= 64, "a-chunk load: two points per lane");

__host__ __device__ constexpr uint32_t al16(uint32_t x) { return (x + 15u) & ~15u; }

// How a block's warps share its work and its tables.  `claim` and `n_used`
// change by atomics; the rest is read and written under `lock` (taken by one
// lane of a warp for a few instructions).
constexpr int MAX_NT = DIRECT_TABLES;
struct Sched {
    unsigned long long claim;   // the block's claim: next unit (low word; may pass the end) and end (high word)
    unsigned n_used[MAX_NT];    // units taken for a table since it was last empty
    unsigned lock;
    unsigned short done;        // no unit is left to claim
    unsigned short moves;       // times a table was entered or freed (modulo 2^16)
    int term[MAX_NT];           // the term a table counts, or FREE, or DRAINING
    unsigned ref[MAX_NT];       // warps adding to a table
};
constexpr int FREE = -1, DRAINING = -2;
constexpr int FOLD_PAD = DIRECT_FOLD_PAD;   // words before a table of one copy (mode 5)

// Shared memory: the block's tables (one to four), T, the schedule, then one
// region per warp: a-records (3 float4 per a-point), the b buffer (float4: x, y, z in
// bins and the b index), the unit's runs (first index, offset in the
// concatenation) and the recheck list.
struct DOff {
    uint32_t hist, hstride, T, misc, warp0, wstride;
    uint32_t arec, buf, runs, xl, st;   // offsets inside a warp's region
    uint32_t end;
};
__host__ __device__ inline DOff d_off(int n_s, int rows, int n_rows, int R, int C, int NT, int W)
{
    DOff o;
    o.hist = 0;
    o.hstride = al16(4u * (uint32_t)(rows * C * R + (R == 1 ? FOLD_PAD : 0)));
    o.T = o.hstride * (uint32_t)NT;
    o.misc = al16(o.T + 8u * (uint32_t)(n_s + 1));
    o.warp0 = o.misc + al16((uint32_t)sizeof(Sched));
    o.arec = 0;
    o.buf = o.arec + 48u * DIRECT_ACHUNK;
    o.runs = o.buf + 16u * BUF;
    o.xl = al16(o.runs + 8u * (uint32_t)(2 * n_rows + 1));
    o.st = al16(o.xl + 8u * XCAP);
    o.wstride = o.st + 48u;
    o.end = o.warp0 + o.wstride * (uint32_t)W;
    return o;
}

extern __shared__ __align__(16) unsigned char dsm[];

__device__ __forceinline__ void red_add(uint32_t a, uint32_t v)
{
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// An a-point's record, each value duplicated for the packed operands: -a_x,
// -a_y, -a_z, then with the x line of sight p = m - n_mu a_x, q = -m - n_mu a_x,
// with the midpoint line of sight (p, q, w) = a - 2 o (o: the observer).
struct ARec {
    float2 nax, nay, naz, p, q, w;
};

// Histogram address of a pair with s-row word bits(S) and signed-mu-column
// word bits(T-): (bits(S) << LS) + (bits(T-) << LT) + Kl, with LT = log2(4 R)
// and LS = LT + log2(C), so that the row and column strides are shifts.
// With one copy (mode 5) a row is 4 C bytes, multiplied instead of shifted.
template <int R, int LOGC>
struct Sh {
    static constexpr int LT = R == 32 ? 7 : (R == 16 ? 6 : (R == 8 ? 5 : (R == 1 ? 2 : -1)));
    static constexpr int LS = LT + LOGC;
    static_assert(LT > 0, "R is 1, 8, 16 or 32");
};

__device__ __forceinline__ uint64_t u64of(float2 v) { return *reinterpret_cast<uint64_t *>(&v); }

// Constant operand pairs of the packed arithmetic (tinyl to c05: midpoint
// line of sight only; la and the clamp lmid: geometric s bins only; mm = m and
// the row's bytes rs: mode 5 only).
struct K2 {
    uint64_t tiny, ms, m1, mh, mt, nm, tinyl, mhalf, c1n, c3n, c05, la, mm;
    float lmid;
    uint32_t rs;
};

// The kernel's modes V: 0 s only, 1 mu along x, 2 mu from the midpoint; 3 and
// 4 are 0 and 1 with geometric s bins; 5 is 1 with one column per |mu| bin.
__host__ __device__ constexpr bool has_mu(int V) { return V != 0 && V != 3; }
__host__ __device__ constexpr bool is_geo(int V) { return V == 3 || V == 4; }

// One packed pair of pairs (b_p, a), (b_p', a) in hand-written PTX: the
// packed s floor word S and s residual FS (the tiny addend, r = rsqrt(d2) by
// MUFU) and, with mu bins, the signed mu floor words.  V = 1 (x line of
// sight): TP, TM = the floors at both ends of the error interval.  V = 2
// (midpoint line of sight): l = b + (a - 2 o), mu = (l.d) r rl with
// rl = rsqrt(|l|^2 + tinyl), TM = floor(n_mu mu), TP = its residual
// n_mu mu - TM - 1/2, CB = 1/2 - c2 - c1 r - c3 rl (certain when |TP| <= CB).
template <int V>
__device__ __forceinline__ void pair2_core(uint64_t bx, uint64_t by, uint64_t bz, const ARec &a, const K2 &k,
                                           uint64_t &S, uint64_t &FS, uint64_t &TP, uint64_t &TM, uint64_t &CB)
{
    if (V == 2) {
        asm("{\n\t"
            ".reg .b64 dx, dy, dz, d2, r, h, lx, ly, lz, q, l2, rl, w, mu, ht, cb;\n\t"
            ".reg .f32 d2x, d2y, rx, ry, l2x, l2y, rlx, rly;\n\t"
            "add.rn.f32x2 dx, %5, %8;\n\t"
            "add.rn.f32x2 dy, %6, %9;\n\t"
            "add.rn.f32x2 dz, %7, %10;\n\t"
            "fma.rn.f32x2 d2, dx, dx, %14;\n\t"
            "fma.rn.f32x2 d2, dy, dy, d2;\n\t"
            "fma.rn.f32x2 d2, dz, dz, d2;\n\t"
            "mov.b64 {d2x, d2y}, d2;\n\t"
            "rsqrt.approx.ftz.f32 rx, d2x;\n\t"
            "rsqrt.approx.ftz.f32 ry, d2y;\n\t"
            "mov.b64 r, {rx, ry};\n\t"
            "fma.rz.f32x2 %0, d2, r, %15;\n\t"
            "fma.rn.f32x2 h, %0, %16, %17;\n\t"
            "fma.rn.f32x2 %1, d2, r, h;\n\t"
            "add.rn.f32x2 lx, %5, %11;\n\t"
            "add.rn.f32x2 ly, %6, %12;\n\t"
            "add.rn.f32x2 lz, %7, %13;\n\t"
            "mul.rn.f32x2 q, lx, dx;\n\t"
            "fma.rn.f32x2 q, ly, dy, q;\n\t"
            "fma.rn.f32x2 q, lz, dz, q;\n\t"
            "fma.rn.f32x2 l2, lx, lx, %20;\n\t"
            "fma.rn.f32x2 l2, ly, ly, l2;\n\t"
            "fma.rn.f32x2 l2, lz, lz, l2;\n\t"
            "mov.b64 {l2x, l2y}, l2;\n\t"
            "rsqrt.approx.ftz.f32 rlx, l2x;\n\t"
            "rsqrt.approx.ftz.f32 rly, l2y;\n\t"
            "mov.b64 rl, {rlx, rly};\n\t"
            "mul.rn.f32x2 w, r, rl;\n\t"
            "mul.rn.f32x2 mu, q, w;\n\t"
            "fma.rz.f32x2 %3, mu, %19, %18;\n\t"
            "fma.rn.f32x2 ht, %3, %16, %18;\n\t"
            "fma.rn.f32x2 %2, mu, %19, ht;\n\t"
            "add.rn.f32x2 %2, %2, %21;\n\t"
            "fma.rn.f32x2 cb, %23, rl, %24;\n\t"
            "fma.rn.f32x2 %4, %22, r, cb;\n\t"
            "}"
            : "=&l"(S), "=&l"(FS), "=&l"(TP), "=&l"(TM), "=&l"(CB)
            : "l"(bx), "l"(by), "l"(bz), "l"(u64of(a.nax)), "l"(u64of(a.nay)), "l"(u64of(a.naz)), "l"(u64of(a.p)),
              "l"(u64of(a.q)), "l"(u64of(a.w)), "l"(k.tiny), "l"(k.ms), "l"(k.m1), "l"(k.mh), "l"(k.mt), "l"(k.nm),
              "l"(k.tinyl), "l"(k.mhalf), "l"(k.c1n), "l"(k.c3n), "l"(k.c05));
    } else if (V == 4) {
        asm("{\n\t"
            ".reg .b64 dx, dy, dz, d2, r, l, h, xp, xm;\n\t"
            ".reg .f32 d2x, d2y, rx, ry, ex, ey;\n\t"
            "add.rn.f32x2 dx, %4, %7;\n\t"
            "add.rn.f32x2 dy, %5, %8;\n\t"
            "add.rn.f32x2 dz, %6, %9;\n\t"
            "fma.rn.f32x2 d2, dx, dx, %12;\n\t"
            "fma.rn.f32x2 d2, dy, dy, d2;\n\t"
            "fma.rn.f32x2 d2, dz, dz, d2;\n\t"
            "mov.b64 {d2x, d2y}, d2;\n\t"
            "lg2.approx.ftz.f32 ex, d2x;\n\t"
            "lg2.approx.ftz.f32 ey, d2y;\n\t"
            "max.f32 ex, ex, %19;\n\t"
            "max.f32 ey, ey, %19;\n\t"
            "mov.b64 l, {ex, ey};\n\t"
            "rsqrt.approx.ftz.f32 rx, d2x;\n\t"
            "rsqrt.approx.ftz.f32 ry, d2y;\n\t"
            "mov.b64 r, {rx, ry};\n\t"
            "fma.rz.f32x2 %0, l, %18, %13;\n\t"
            "fma.rn.f32x2 h, %0, %14, %15;\n\t"
            "fma.rn.f32x2 %1, l, %18, h;\n\t"
            "fma.rn.f32x2 xp, %4, %17, %10;\n\t"
            "fma.rn.f32x2 xm, %4, %17, %11;\n\t"
            "fma.rz.f32x2 %2, xp, r, %16;\n\t"
            "fma.rz.f32x2 %3, xm, r, %16;\n\t"
            "}"
            : "=&l"(S), "=&l"(FS), "=&l"(TP), "=&l"(TM)
            : "l"(bx), "l"(by), "l"(bz), "l"(u64of(a.nax)), "l"(u64of(a.nay)), "l"(u64of(a.naz)), "l"(u64of(a.p)),
              "l"(u64of(a.q)), "l"(k.tiny), "l"(k.ms), "l"(k.m1), "l"(k.mh), "l"(k.mt), "l"(k.nm), "l"(k.la),
              "f"(k.lmid));
        CB = 0;
    } else if (V == 5) {
        asm("{\n\t"
            ".reg .b64 dx, dy, dz, d2, r, h, x, xp, xm;\n\t"
            ".reg .f32 d2x, d2y, rx, ry;\n\t"
            "add.rn.f32x2 dx, %4, %7;\n\t"
            "add.rn.f32x2 dy, %5, %8;\n\t"
            "add.rn.f32x2 dz, %6, %9;\n\t"
            "fma.rn.f32x2 d2, dx, dx, %11;\n\t"
            "fma.rn.f32x2 d2, dy, dy, d2;\n\t"
            "fma.rn.f32x2 d2, dz, dz, d2;\n\t"
            "mov.b64 {d2x, d2y}, d2;\n\t"
            "rsqrt.approx.ftz.f32 rx, d2x;\n\t"
            "rsqrt.approx.ftz.f32 ry, d2y;\n\t"
            "mov.b64 r, {rx, ry};\n\t"
            "fma.rz.f32x2 %0, d2, r, %12;\n\t"
            "fma.rn.f32x2 h, %0, %13, %14;\n\t"
            "fma.rn.f32x2 %1, d2, r, h;\n\t"
            "fma.rn.f32x2 x, %4, %16, %10;\n\t"
            "and.b64 x, x, 0x7fffffff7fffffff;\n\t"
            "add.rn.f32x2 xp, x, %17;\n\t"
            "fma.rn.f32x2 xm, %17, %13, x;\n\t"
            "fma.rz.f32x2 %2, xp, r, %15;\n\t"
            "fma.rz.f32x2 %3, xm, r, %15;\n\t"
            "}"
            : "=&l"(S), "=&l"(FS), "=&l"(TP), "=&l"(TM)
            : "l"(bx), "l"(by), "l"(bz), "l"(u64of(a.nax)), "l"(u64of(a.nay)), "l"(u64of(a.naz)), "l"(u64of(a.p)),
              "l"(k.tiny), "l"(k.ms), "l"(k.m1), "l"(k.mh), "l"(k.mt), "l"(k.nm), "l"(k.mm));
        CB = 0;
    } else if (V == 3) {
        asm("{\n\t"
            ".reg .b64 dx, dy, dz, d2, l, h;\n\t"
            ".reg .f32 d2x, d2y, ex, ey;\n\t"
            "add.rn.f32x2 dx, %2, %5;\n\t"
            "add.rn.f32x2 dy, %3, %6;\n\t"
            "add.rn.f32x2 dz, %4, %7;\n\t"
            "fma.rn.f32x2 d2, dx, dx, %8;\n\t"
            "fma.rn.f32x2 d2, dy, dy, d2;\n\t"
            "fma.rn.f32x2 d2, dz, dz, d2;\n\t"
            "mov.b64 {d2x, d2y}, d2;\n\t"
            "lg2.approx.ftz.f32 ex, d2x;\n\t"
            "lg2.approx.ftz.f32 ey, d2y;\n\t"
            "max.f32 ex, ex, %13;\n\t"
            "max.f32 ey, ey, %13;\n\t"
            "mov.b64 l, {ex, ey};\n\t"
            "fma.rz.f32x2 %0, l, %12, %9;\n\t"
            "fma.rn.f32x2 h, %0, %10, %11;\n\t"
            "fma.rn.f32x2 %1, l, %12, h;\n\t"
            "}"
            : "=&l"(S), "=&l"(FS)
            : "l"(bx), "l"(by), "l"(bz), "l"(u64of(a.nax)), "l"(u64of(a.nay)), "l"(u64of(a.naz)), "l"(k.tiny),
              "l"(k.ms), "l"(k.m1), "l"(k.mh), "l"(k.la), "f"(k.lmid));
        TP = TM = CB = 0;
    } else if (V == 1) {
        asm("{\n\t"
            ".reg .b64 dx, dy, dz, d2, r, h, xp, xm;\n\t"
            ".reg .f32 d2x, d2y, rx, ry;\n\t"
            "add.rn.f32x2 dx, %4, %7;\n\t"
            "add.rn.f32x2 dy, %5, %8;\n\t"
            "add.rn.f32x2 dz, %6, %9;\n\t"
            "fma.rn.f32x2 d2, dx, dx, %12;\n\t"
            "fma.rn.f32x2 d2, dy, dy, d2;\n\t"
            "fma.rn.f32x2 d2, dz, dz, d2;\n\t"
            "mov.b64 {d2x, d2y}, d2;\n\t"
            "rsqrt.approx.ftz.f32 rx, d2x;\n\t"
            "rsqrt.approx.ftz.f32 ry, d2y;\n\t"
            "mov.b64 r, {rx, ry};\n\t"
            "fma.rz.f32x2 %0, d2, r, %13;\n\t"
            "fma.rn.f32x2 h, %0, %14, %15;\n\t"
            "fma.rn.f32x2 %1, d2, r, h;\n\t"
            "fma.rn.f32x2 xp, %4, %17, %10;\n\t"
            "fma.rn.f32x2 xm, %4, %17, %11;\n\t"
            "fma.rz.f32x2 %2, xp, r, %16;\n\t"
            "fma.rz.f32x2 %3, xm, r, %16;\n\t"
            "}"
            : "=&l"(S), "=&l"(FS), "=&l"(TP), "=&l"(TM)
            : "l"(bx), "l"(by), "l"(bz), "l"(u64of(a.nax)), "l"(u64of(a.nay)), "l"(u64of(a.naz)), "l"(u64of(a.p)),
              "l"(u64of(a.q)), "l"(k.tiny), "l"(k.ms), "l"(k.m1), "l"(k.mh), "l"(k.mt), "l"(k.nm));
        CB = 0;
    } else {
        asm("{\n\t"
            ".reg .b64 dx, dy, dz, d2, r, h;\n\t"
            ".reg .f32 d2x, d2y, rx, ry;\n\t"
            "add.rn.f32x2 dx, %2, %5;\n\t"
            "add.rn.f32x2 dy, %3, %6;\n\t"
            "add.rn.f32x2 dz, %4, %7;\n\t"
            "fma.rn.f32x2 d2, dx, dx, %8;\n\t"
            "fma.rn.f32x2 d2, dy, dy, d2;\n\t"
            "fma.rn.f32x2 d2, dz, dz, d2;\n\t"
            "mov.b64 {d2x, d2y}, d2;\n\t"
            "rsqrt.approx.ftz.f32 rx, d2x;\n\t"
            "rsqrt.approx.ftz.f32 ry, d2y;\n\t"
            "mov.b64 r, {rx, ry};\n\t"
            "fma.rz.f32x2 %0, d2, r, %9;\n\t"
            "fma.rn.f32x2 h, %0, %10, %11;\n\t"
            "fma.rn.f32x2 %1, d2, r, h;\n\t"
            "}"
            : "=&l"(S), "=&l"(FS)
            : "l"(bx), "l"(by), "l"(bz), "l"(u64of(a.nax)), "l"(u64of(a.nay)), "l"(u64of(a.naz)), "l"(k.tiny),
              "l"(k.ms), "l"(k.m1), "l"(k.mh));
        TP = TM = CB = 0;
    }
}

__device__ __forceinline__ float lo_f(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi_f(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }

// Histogram addresses of the two pairs: the s row (S clamped to the spare
// last row) and, with mu bins, the signed mu column of T-.
template <int V, int LS, int LT>
__device__ __forceinline__ void pair_addr(uint64_t S, uint64_t TM, float stop, uint32_t Kl, uint32_t rs, uint32_t &a0,
                                          uint32_t &a1)
{
    const uint32_t s0 = __float_as_uint(fminf(lo_f(S), stop)), s1 = __float_as_uint(fminf(hi_f(S), stop));
    a0 = Kl + (V == 5 ? s0 * rs : s0 << LS);
    a1 = Kl + (V == 5 ? s1 * rs : s1 << LS);
    if (has_mu(V)) {
        a0 += (uint32_t)TM << LT;
        a1 += (uint32_t)(TM >> 32) << LT;
    }
}

// Rare path: two pairs recomputed with one uncertainty flag each, by the
// same instructions as the hot path's PTX block (so bit for bit the same
// addresses and decisions).
template <int V, int LS, int LT>
__device__ __forceinline__ void pair2_flags(uint64_t bx, uint64_t by, uint64_t bz, const ARec &a, const K2 &k,
                                            float cs, float stop, uint32_t Kl, uint32_t &a0, uint32_t &a1, bool &f0,
                                            bool &f1)
{
    uint64_t S, FS, TP, TM, CB;
    pair2_core<V>(bx, by, bz, a, k, S, FS, TP, TM, CB);
    pair_addr<V, LS, LT>(S, TM, stop, Kl, k.rs, a0, a1);
    f0 = fabsf(lo_f(FS)) > cs;
    f1 = fabsf(hi_f(FS)) > cs;
    if (V == 1 || V == 4 || V == 5) {
        f0 = f0 || lo_f(TP) != lo_f(TM);
        f1 = f1 || hi_f(TP) != hi_f(TM);
    } else if (V == 2) {
        f0 = f0 || fabsf(lo_f(TP)) > lo_f(CB);
        f1 = f1 || fabsf(hi_f(TP)) > hi_f(CB);
    }
}

// One a-point against this lane's four b-points (two packed pairs q = 0, 1),
// in one block of hand-written PTX so that the uncertainty of all four pairs
// accumulates in one predicate (setp with .or): the four histogram adds, and
// whether some pair of this lane is uncertain.  The loop runs two a-points per
// iteration (two independent blocks the scheduler interleaves) under one vote.  CHK (self
// cell): a pair with a >= b goes to the lane's spare word instead.
// Operands: %0 the lane's uncertainty; %1-%6 b (x, y, z) of q = 0, 1; %7-%11 the a-record;
// %12-%17 constants; %18 cs; %19 the s clamp; %20 Kl; %21, %22 LS, LT;
// CHK: %23 a index, %24-%27 b indices of slots 0-3, %28 spare word; geometric bins: A and lmid after these, mode 5: m and
// a row's bytes.
#define PD_D2(BX, BY, BZ)                            \
    "add.rn.f32x2 dx, " BX ", %7;\n\t"                 \
    "add.rn.f32x2 dy, " BY ", %8;\n\t"                 \
    "add.rn.f32x2 dz, " BZ ", %9;\n\t"                 \
    "fma.rn.f32x2 d2, dx, dx, %12;\n\t"                \
    "fma.rn.f32x2 d2, dy, dy, d2;\n\t"                 \
    "fma.rn.f32x2 d2, dz, dz, d2;\n\t"                 \
    "mov.b64 {d2x, d2y}, d2;\n\t"
#define PD_RSQ                                       \
    "rsqrt.approx.ftz.f32 rx, d2x;\n\t"                \
    "rsqrt.approx.ftz.f32 ry, d2y;\n\t"                \
    "mov.b64 r, {rx, ry};\n\t"
#define PD_LG2(LA, LMID)                             \
    "lg2.approx.ftz.f32 sx, d2x;\n\t"                  \
    "lg2.approx.ftz.f32 sy, d2y;\n\t"                  \
    "max.f32 sx, sx, " LMID ";\n\t"                    \
    "max.f32 sy, sy, " LMID ";\n\t"                    \
    "mov.b64 d2, {sx, sy};\n\t"                        \
    "fma.rz.f32x2 s, d2, " LA ", %13;\n\t"             \
    "fma.rn.f32x2 h, s, %14, %15;\n\t"                 \
    "fma.rn.f32x2 fs, d2, " LA ", h;\n\t"
#define PD_LIN                                       \
    "fma.rz.f32x2 s, d2, r, %13;\n\t"                  \
    "fma.rn.f32x2 h, s, %14, %15;\n\t"                 \
    "fma.rn.f32x2 fs, d2, r, h;\n\t"
#define PD_S                                         \
    "mov.b64 {sx, sy}, s;\n\t"                         \
    "mov.b64 {fx, fy}, fs;\n\t"                        \
    "abs.f32 fx, fx;\n\t"                              \
    "abs.f32 fy, fy;\n\t"                              \
    "setp.gtu.or.f32 p, fx, %18, p;\n\t"               \
    "setp.gtu.or.f32 p, fy, %18, p;\n\t"               \
    "min.f32 sx, sx, %19;\n\t"                         \
    "min.f32 sy, sy, %19;\n\t"                         \
    "mov.b32 ux, sx;\n\t"                              \
    "mov.b32 uy, sy;\n\t"
#define PD_ROW                                       \
    "shl.b32 ux, ux, %21;\n\t"                         \
    "shl.b32 uy, uy, %21;\n\t"                         \
    "add.u32 ux, ux, %20;\n\t"                         \
    "add.u32 uy, uy, %20;\n\t"
#define PD_DIFF(BX, BY, BZ) PD_D2(BX, BY, BZ) PD_RSQ PD_LIN PD_S PD_ROW
#define PD_GEO(BX, BY, BZ, LA, LMID) PD_D2(BX, BY, BZ) PD_LG2(LA, LMID) PD_S PD_ROW
#define PD_ABS(BX, BY, BZ, MM, RS)                   \
    PD_D2(BX, BY, BZ) PD_RSQ PD_LIN PD_S               \
    "mad.lo.u32 ux, ux, " RS ", %20;\n\t"              \
    "mad.lo.u32 uy, uy, " RS ", %20;\n\t"              \
    "fma.rn.f32x2 xm, " BX ", %17, %10;\n\t"           \
    "and.b64 xm, xm, 0x7fffffff7fffffff;\n\t"          \
    "add.rn.f32x2 xp, xm, " MM ";\n\t"                 \
    "fma.rn.f32x2 xm, " MM ", %14, xm;\n\t" PD_COL
#define PD_MU(BX)                                    \
    "fma.rn.f32x2 xp, " BX ", %17, %10;\n\t"           \
    "fma.rn.f32x2 xm, " BX ", %17, %11;\n\t" PD_COL
#define PD_COL                                       \
    "fma.rz.f32x2 tp, xp, r, %16;\n\t"                 \
    "fma.rz.f32x2 tm, xm, r, %16;\n\t"                 \
    "mov.b64 {px, py}, tp;\n\t"                        \
    "mov.b64 {mx, my}, tm;\n\t"                        \
    "setp.neu.or.f32 p, px, mx, p;\n\t"                \
    "setp.neu.or.f32 p, py, my, p;\n\t"                \
    "mov.b32 vx, mx;\n\t"                              \
    "mov.b32 vy, my;\n\t"                              \
    "shl.b32 vx, vx, %22;\n\t"                         \
    "shl.b32 vy, vy, %22;\n\t"                         \
    "add.u32 ux, ux, vx;\n\t"                          \
    "add.u32 uy, uy, vy;\n\t"
#define PD_CHK(IB0, IB1)                             \
    "setp.lt.u32 c, %23, " IB0 ";\n\t"                 \
    "selp.b32 ux, ux, %28, c;\n\t"                     \
    "setp.lt.u32 c, %23, " IB1 ";\n\t"                 \
    "selp.b32 uy, uy, %28, c;\n\t"
#define PD_RED                                       \
    "red.shared.add.u32 [ux], 1;\n\t"                  \
    "red.shared.add.u32 [uy], 1;\n\t"
#define PD_HEAD                                                                     \
    "{\n\t"                                                                           \
    ".reg .b64 dx, dy, dz, d2, r, s, h, fs, xp, xm, tp, tm;\n\t"                      \
    ".reg .f32 d2x, d2y, rx, ry, sx, sy, fx, fy, px, py, mx, my;\n\t"                 \
    ".reg .b32 ux, uy, vx, vy;\n\t"                                                   \
    ".reg .pred p, c;\n\t"                                                            \
    "setp.ne.u32 p, %20, %20;\n\t"
#define PD_TAIL                                      \
    "selp.u32 %0, 1, 0, p;\n\t"                        \
    "}"

// Midpoint line of sight.  Operands: %0 the lane's uncertainty; %1-%6 b;
// %7-%9 -a; %10-%12 a - 2 o; %13-%23 constants (tiny, ms, m1, mh, mt, nm,
// tinyl, -1/2, c1n, c3n, c05); %24 cs; %25 the s clamp; %26 Kl; %27, %28 LS,
// LT; self-cell tiles: %29 the a index, %30-%33 b limits, %34 the spare word.
// The mu residual is (n_mu mu - floor(n_mu mu)) - 1/2: 1.5 * 2^23 - 1/2 has no
// FP32 form, so the half is subtracted after the fraction.
#define PM_PAIR(BX, BY, BZ)                          \
    "add.rn.f32x2 dx, " BX ", %7;\n\t"                 \
    "add.rn.f32x2 dy, " BY ", %8;\n\t"                 \
    "add.rn.f32x2 dz, " BZ ", %9;\n\t"                 \
    "fma.rn.f32x2 d2, dx, dx, %13;\n\t"                \
    "fma.rn.f32x2 d2, dy, dy, d2;\n\t"                 \
    "fma.rn.f32x2 d2, dz, dz, d2;\n\t"                 \
    "mov.b64 {d2x, d2y}, d2;\n\t"                      \
    "rsqrt.approx.ftz.f32 rx, d2x;\n\t"                \
    "rsqrt.approx.ftz.f32 ry, d2y;\n\t"                \
    "mov.b64 r, {rx, ry};\n\t"                         \
    "fma.rz.f32x2 s, d2, r, %14;\n\t"                  \
    "fma.rn.f32x2 h, s, %15, %16;\n\t"                 \
    "fma.rn.f32x2 fs, d2, r, h;\n\t"                   \
    "add.rn.f32x2 lx, " BX ", %10;\n\t"                \
    "add.rn.f32x2 ly, " BY ", %11;\n\t"                \
    "add.rn.f32x2 lz, " BZ ", %12;\n\t"                \
    "mul.rn.f32x2 q, lx, dx;\n\t"                      \
    "fma.rn.f32x2 q, ly, dy, q;\n\t"                   \
    "fma.rn.f32x2 q, lz, dz, q;\n\t"                   \
    "fma.rn.f32x2 l2, lx, lx, %19;\n\t"                \
    "fma.rn.f32x2 l2, ly, ly, l2;\n\t"                 \
    "fma.rn.f32x2 l2, lz, lz, l2;\n\t"                 \
    "mov.b64 {l2x, l2y}, l2;\n\t"                      \
    "rsqrt.approx.ftz.f32 rlx, l2x;\n\t"               \
    "rsqrt.approx.ftz.f32 rly, l2y;\n\t"               \
    "mov.b64 rl, {rlx, rly};\n\t"                      \
    "mul.rn.f32x2 w, r, rl;\n\t"                       \
    "mul.rn.f32x2 mu, q, w;\n\t"                       \
    "fma.rz.f32x2 tm, mu, %18, %17;\n\t"               \
    "fma.rn.f32x2 ht, tm, %15, %17;\n\t"               \
    "fma.rn.f32x2 fm, mu, %18, ht;\n\t"                \
    "add.rn.f32x2 fm, fm, %20;\n\t"                    \
    "fma.rn.f32x2 cb, %22, rl, %23;\n\t"               \
    "fma.rn.f32x2 cb, %21, r, cb;\n\t"                 \
    "mov.b64 {sx, sy}, s;\n\t"                         \
    "mov.b64 {fx, fy}, fs;\n\t"                        \
    "mov.b64 {gx, gy}, fm;\n\t"                        \
    "mov.b64 {kx, ky}, cb;\n\t"                        \
    "mov.b64 {mx, my}, tm;\n\t"                        \
    "abs.f32 fx, fx;\n\t"                              \
    "abs.f32 fy, fy;\n\t"                              \
    "abs.f32 gx, gx;\n\t"                              \
    "abs.f32 gy, gy;\n\t"                              \
    "setp.gtu.or.f32 p, fx, %24, p;\n\t"               \
    "setp.gtu.or.f32 p, fy, %24, p;\n\t"               \
    "setp.gtu.or.f32 p, gx, kx, p;\n\t"                \
    "setp.gtu.or.f32 p, gy, ky, p;\n\t"                \
    "min.f32 sx, sx, %25;\n\t"                         \
    "min.f32 sy, sy, %25;\n\t"                         \
    "mov.b32 ux, sx;\n\t"                              \
    "mov.b32 uy, sy;\n\t"                              \
    "shl.b32 ux, ux, %27;\n\t"                         \
    "shl.b32 uy, uy, %27;\n\t"                         \
    "add.u32 ux, ux, %26;\n\t"                         \
    "add.u32 uy, uy, %26;\n\t"                         \
    "mov.b32 vx, mx;\n\t"                              \
    "mov.b32 vy, my;\n\t"                              \
    "shl.b32 vx, vx, %28;\n\t"                         \
    "shl.b32 vy, vy, %28;\n\t"                         \
    "add.u32 ux, ux, vx;\n\t"                          \
    "add.u32 uy, uy, vy;\n\t"
#define PM_CHK(IB0, IB1)                             \
    "setp.lt.u32 c, %29, " IB0 ";\n\t"                 \
    "selp.b32 ux, ux, %34, c;\n\t"                     \
    "setp.lt.u32 c, %29, " IB1 ";\n\t"                 \
    "selp.b32 uy, uy, %34, c;\n\t"
#define PM_RED                                       \
    "red.shared.add.u32 [ux], 1;\n\t"                  \
    "red.shared.add.u32 [uy], 1;\n\t"
#define PM_HEAD                                                                                \
    "{\n\t"                                                                                      \
    ".reg .b64 dx, dy, dz, d2, r, s, h, fs, lx, ly, lz, q, l2, rl, w, mu, tm, ht, fm, cb;\n\t"   \
    ".reg .f32 d2x, d2y, rx, ry, l2x, l2y, rlx, rly, sx, sy, fx, fy, gx, gy, kx, ky, mx, my;\n\t" \
    ".reg .b32 ux, uy, vx, vy;\n\t"                                                              \
    ".reg .pred p, c;\n\t"                                                                       \
    "setp.ne.u32 p, %26, %26;\n\t"

template <int V, bool CHK, int LS, int LT>
__device__ __forceinline__ bool apoint(const float2 (&BX)[NQ], const float2 (&BY)[NQ], const float2 (&BZ)[NQ],
                                       const ARec &a, const K2 &k, float cs, float stop, uint32_t Kl, uint32_t ia,
                                       const uint32_t (&IB)[NP], uint32_t dump)
{
    static_assert(NQ == 2, "the PTX block covers two packed pairs");
    constexpr bool MU = has_mu(V);
    uint32_t any;
    if (V == 2) {
#define PM_IN                                                                                                    \
    "l"(u64of(BX[0])), "l"(u64of(BY[0])), "l"(u64of(BZ[0])), "l"(u64of(BX[1])), "l"(u64of(BY[1])),             \
        "l"(u64of(BZ[1])), "l"(u64of(a.nax)), "l"(u64of(a.nay)), "l"(u64of(a.naz)), "l"(u64of(a.p)),            \
        "l"(u64of(a.q)), "l"(u64of(a.w)), "l"(k.tiny), "l"(k.ms), "l"(k.m1), "l"(k.mh), "l"(k.mt), "l"(k.nm),   \
        "l"(k.tinyl), "l"(k.mhalf), "l"(k.c1n), "l"(k.c3n), "l"(k.c05), "f"(cs), "f"(stop), "r"(Kl), "n"(LS), \
        "n"(LT)
        if (CHK)
            asm volatile(PM_HEAD PM_PAIR("%1", "%2", "%3") PM_CHK("%30", "%31") PM_RED PM_PAIR("%4", "%5", "%6")
                             PM_CHK("%32", "%33") PM_RED "selp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(any)
                         : PM_IN, "r"(ia), "r"(IB[0]), "r"(IB[1]), "r"(IB[2]), "r"(IB[3]), "r"(dump)
                         : "memory");
        else
            asm volatile(PM_HEAD PM_PAIR("%1", "%2", "%3") PM_RED PM_PAIR("%4", "%5", "%6") PM_RED
                         "selp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(any)
                         : PM_IN
                         : "memory");
#undef PM_IN
        return any != 0;
    }
#define PD_IN                                                                                                     \
    "l"(u64of(BX[0])), "l"(u64of(BY[0])), "l"(u64of(BZ[0])), "l"(u64of(BX[1])), "l"(u64of(BY[1])),              \
        "l"(u64of(BZ[1])), "l"(u64of(a.nax)), "l"(u64of(a.nay)), "l"(u64of(a.naz)), "l"(u64of(a.p)),             \
        "l"(u64of(a.q)), "l"(k.tiny), "l"(k.ms), "l"(k.m1), "l"(k.mh), "l"(k.mt), "l"(k.nm), "f"(cs), "f"(stop), \
        "r"(Kl), "n"(LS), "n"(LT)
    if (V == 5 && CHK) {
        asm volatile(PD_HEAD PD_ABS("%1", "%2", "%3", "%29", "%30") PD_CHK("%24", "%25") PD_RED
                         PD_ABS("%4", "%5", "%6", "%29", "%30") PD_CHK("%26", "%27") PD_RED PD_TAIL
                     : "=r"(any)
                     : PD_IN, "r"(ia), "r"(IB[0]), "r"(IB[1]), "r"(IB[2]), "r"(IB[3]), "r"(dump), "l"(k.mm),
                       "r"(k.rs)
                     : "memory");
    } else if (V == 5) {
        asm volatile(PD_HEAD PD_ABS("%1", "%2", "%3", "%23", "%24") PD_RED PD_ABS("%4", "%5", "%6", "%23", "%24")
                         PD_RED PD_TAIL
                     : "=r"(any)
                     : PD_IN, "l"(k.mm), "r"(k.rs)
                     : "memory");
    } else if (V == 4 && CHK) {
        asm volatile(PD_HEAD PD_GEO("%1", "%2", "%3", "%29", "%30") PD_RSQ PD_MU("%1") PD_CHK("%24", "%25") PD_RED
                         PD_GEO("%4", "%5", "%6", "%29", "%30") PD_RSQ PD_MU("%4") PD_CHK("%26", "%27") PD_RED PD_TAIL
                     : "=r"(any)
                     : PD_IN, "r"(ia), "r"(IB[0]), "r"(IB[1]), "r"(IB[2]), "r"(IB[3]), "r"(dump), "l"(k.la),
                       "f"(k.lmid)
                     : "memory");
    } else if (V == 4) {
        asm volatile(PD_HEAD PD_GEO("%1", "%2", "%3", "%23", "%24") PD_RSQ PD_MU("%1") PD_RED
                         PD_GEO("%4", "%5", "%6", "%23", "%24") PD_RSQ PD_MU("%4") PD_RED PD_TAIL
                     : "=r"(any)
                     : PD_IN, "l"(k.la), "f"(k.lmid)
                     : "memory");
    } else if (V == 3 && CHK) {
        asm volatile(PD_HEAD PD_GEO("%1", "%2", "%3", "%29", "%30") PD_CHK("%24", "%25") PD_RED
                         PD_GEO("%4", "%5", "%6", "%29", "%30") PD_CHK("%26", "%27") PD_RED PD_TAIL
                     : "=r"(any)
                     : PD_IN, "r"(ia), "r"(IB[0]), "r"(IB[1]), "r"(IB[2]), "r"(IB[3]), "r"(dump), "l"(k.la),
                       "f"(k.lmid)
                     : "memory");
    } else if (V == 3) {
        asm volatile(PD_HEAD PD_GEO("%1", "%2", "%3", "%23", "%24") PD_RED
                         PD_GEO("%4", "%5", "%6", "%23", "%24") PD_RED PD_TAIL
                     : "=r"(any)
                     : PD_IN, "l"(k.la), "f"(k.lmid)
                     : "memory");
    } else if (MU && CHK) {
        asm volatile(PD_HEAD PD_DIFF("%1", "%2", "%3") PD_MU("%1") PD_CHK("%24", "%25") PD_RED
                         PD_DIFF("%4", "%5", "%6") PD_MU("%4") PD_CHK("%26", "%27") PD_RED PD_TAIL
                     : "=r"(any)
                     : PD_IN, "r"(ia), "r"(IB[0]), "r"(IB[1]), "r"(IB[2]), "r"(IB[3]), "r"(dump)
                     : "memory");
    } else if (MU) {
        asm volatile(PD_HEAD PD_DIFF("%1", "%2", "%3") PD_MU("%1") PD_RED PD_DIFF("%4", "%5", "%6") PD_MU("%4")
                         PD_RED PD_TAIL
                     : "=r"(any)
                     : PD_IN
                     : "memory");
    } else if (CHK) {
        asm volatile(PD_HEAD PD_DIFF("%1", "%2", "%3") PD_CHK("%24", "%25") PD_RED PD_DIFF("%4", "%5", "%6")
                         PD_CHK("%26", "%27") PD_RED PD_TAIL
                     : "=r"(any)
                     : PD_IN, "r"(ia), "r"(IB[0]), "r"(IB[1]), "r"(IB[2]), "r"(IB[3]), "r"(dump)
                     : "memory");
    } else {
        asm volatile(PD_HEAD PD_DIFF("%1", "%2", "%3") PD_RED PD_DIFF("%4", "%5", "%6") PD_RED PD_TAIL
                     : "=r"(any)
                     : PD_IN
                     : "memory");
    }
#undef PD_IN
    return any != 0;
}
#undef PD_D2
#undef PD_RSQ
#undef PD_LG2
#undef PD_LIN
#undef PD_S
#undef PD_DIFF
#undef PD_GEO
#undef PD_ROW
#undef PD_ABS
#undef PD_COL
#undef PD_MU
#undef PD_CHK
#undef PD_RED
#undef PD_HEAD
#undef PD_TAIL
#undef PM_PAIR
#undef PM_CHK
#undef PM_RED
#undef PM_HEAD

// Kl of the warp's table (see Sh), the histogram base (shared address) + 4
// (lane mod R) and this lane's word in the spare last row.
template <bool MU, int R, int LOGC>
struct Addr {
    static constexpr int LS = Sh<R, LOGC>::LS, LT = Sh<R, LOGC>::LT;
    uint32_t Kl;
    __device__ __forceinline__ static uint32_t shift(const DirectParams &dp)
    {
        if (R == 1) return 4u * (uint32_t)dp.CO - MAG_S_BITS * (4u * (uint32_t)dp.C) - (MAG_T_BITS << LT);
        return MU ? ((uint32_t)dp.CO << LT) - (MAG_S_BITS << LS) - (MAG_T_BITS << LT) : 0u - (MAG_S_BITS << LS);
    }
    // row k, column c from the base hb
    __device__ __forceinline__ static uint32_t cell(const DirectParams &dp, uint32_t hb, uint32_t k, uint32_t c)
    {
        return hb + (R == 1 ? 4u * (k * (uint32_t)dp.C + c) : (k << LS) + (c << LT));
    }
    __device__ __forceinline__ uint32_t hb(const DirectParams &dp) const { return Kl - shift(dp); }
    __device__ __forceinline__ uint32_t dump(const DirectParams &dp) const
    {
        return cell(dp, hb(dp), (uint32_t)(dp.rows - 1), R == 1 ? (uint32_t)dp.CO : 0u);
    }
};

// What a warp keeps from unit to unit, in shared memory (the registers belong
// to the tiles): counters for the launch's statistics, its table, the table's
// term and that term's units [t_lo, t_hi).
struct WarpState {
    unsigned long long n_cand, n_exact, binned, t_start;
    int tab, term;
    uint32_t t_lo, t_hi;
};

// A warp's shared-memory region and its pending exact rechecks.
struct WarpMem {
    float4 *arec;     // a-records of the unit's a-chunk
    float4 *buf;      // b buffer: x, y, z in bins and the b index
    uint2 *runs;      // the unit's runs: (first b index, offset in their concatenation)
    uint2 *xl;        // pairs (a index, b index) awaiting the exact recheck
    WarpState *st;
};

template <bool MID>
__device__ __forceinline__ ARec load_a(const float4 *arec, uint32_t ai)
{
    const float4 r0 = arec[3 * ai], r1 = arec[3 * ai + 1];
    if (MID) {
        const float4 r2 = arec[3 * ai + 2];
        return ARec{make_float2(r0.x, r0.y), make_float2(r0.z, r0.w), make_float2(r1.x, r1.y),
                    make_float2(r1.z, r1.w), make_float2(r2.x, r2.y), make_float2(r2.z, r2.w)};
    }
    const float2 r2 = *(const float2 *)&arec[3 * ai + 2];
    return ARec{make_float2(r0.x, r0.y), make_float2(r0.z, r0.w), make_float2(r1.x, r1.y), make_float2(r1.z, r1.w),
                r2, make_float2(0.f, 0.f)};
}

__device__ __forceinline__ void xl_put(uint2 *xl, uint32_t i, uint32_t ia, uint32_t ib) { xl[i] = make_uint2(ia, ib); }

// exact recheck of the n listed pairs, one per lane
template <bool MU, int R, int LOGC>
__device__ __forceinline__ void recheck(const CountParams &prm, const DirectParams &dp, const Mesh &m,
                                        const unsigned long long *T, const WarpMem &wm, uint32_t n, uint32_t hb,
                                        int lane)
{
    __syncwarp();
    const uint2 *xl = wm.xl;
    if (lane == 0) wm.st->n_exact += n;
#pragma unroll 1
    for (uint32_t e = (uint32_t)lane; e < n; e += 32) {
        const uint2 pr = xl[e];
        const int bin = exact_bin(prm, T, m.us, m.n_total, pr.x, pr.y);
        if (bin >= 0) {
            const uint32_t k = (uint32_t)bin / (uint32_t)prm.n_mu + (uint32_t)dp.row0, j = (uint32_t)bin % (uint32_t)prm.n_mu;
            const uint32_t col = MU ? j + (uint32_t)dp.CO : 0u;
            red_add(Addr<MU, R, LOGC>::cell(dp, hb, k, col), 1u);
        }
    }
    __syncwarp();
}

// The same as a call of its own.  The midpoint kernel needs all of its 128
// registers for the pair loop: with the rare code (rechecks, table switches)
// inlined it spills, 34.3 against 33.6 ms on the cut-sky mocks; the others do
// not, and run 1 to 2 % faster inlined.
template <bool MU, int R, int LOGC>
__device__ __noinline__ void recheck_apart(const CountParams &prm, const DirectParams &dp, const Mesh &m,
                                           const unsigned long long *T, const WarpMem &wm, uint32_t n, uint32_t hb,
                                           int lane)
{
    recheck<MU, R, LOGC>(prm, dp, m, T, wm, n, hb, lane);
}

// this lane's b-points of the tile (buffer slots 32 p + lane, packed in
// pairs p = 2q, 2q + 1); slots at or past nb are padding
__device__ __forceinline__ void load_tile(const float4 *buf, uint32_t nb, int lane, float2 (&BX)[NQ], float2 (&BY)[NQ],
                                          float2 (&BZ)[NQ])
{
#pragma unroll
    for (int q = 0; q < NQ; q++) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const uint32_t s = 32u * (uint32_t)(2 * q + h) + (uint32_t)lane;
            const float4 v = s < nb ? buf[s] : make_float4(FAR, FAR, FAR, 0.0f);
            if (h) {
                BX[q].y = v.x;
                BY[q].y = v.y;
                BZ[q].y = v.z;
            } else {
                BX[q].x = v.x;
                BY[q].x = v.y;
                BZ[q].x = v.z;
            }
        }
    }
}

// Every pair of the a-chunk (na points from sorted index a0) with the first nb
// entries of the warp's buffer; CHK: the first nself entries are points of
// the a-chunk's own cell (an auto count), of whose pairs only a < b count.
// Padding slots hold far-away points whose adds land in the spare last row.
// The a-points run two at a time, the last of an odd chunk alone.  The
// uncertainties of one a-point's pairs are or-ed into one predicate per lane;
// when any lane's is set, the a-points' pairs are recomputed with a flag each,
// and each uncertain pair's add is taken back and the pair joins the recheck
// list.
template <int V, int R, int LOGC, bool CHK>
__device__ __forceinline__ void tile(const CountParams &prm, const DirectParams &dp, const Mesh &m,
                                     const unsigned long long *T, const WarpMem &wm,
                                     const Addr<has_mu(V), R, LOGC> &ad, uint32_t nb, uint32_t nself, uint32_t na,
                                     uint32_t a0, int lane, uint32_t &n_list)
{
    constexpr bool MU = has_mu(V), MID = V == 2;
    float2 BX[NQ], BY[NQ], BZ[NQ];
    load_tile(wm.buf, nb, lane, BX, BY, BZ);
    // CHK: a self-cell slot counts a pair when a < b, any other real slot
    // always, a padding slot never
    uint32_t IB[NP] = {0u, 0u, 0u, 0u};
    if (CHK) {
#pragma unroll
        for (int p = 0; p < NP; p++) {
            const uint32_t s = 32u * (uint32_t)p + (uint32_t)lane;
            IB[p] = s < nself ? __float_as_uint(wm.buf[s].w) : (s < nb ? 0xFFFFFFFFu : 0u);
        }
    }
    // slot p of this lane holds a b-point (not padding): bit p
    uint32_t live = 0;
#pragma unroll
    for (int p = 0; p < NP; p++) live |= (32u * (uint32_t)p + (uint32_t)lane < nb ? 1u : 0u) << p;
    if (lane == 0) wm.st->n_cand += (unsigned long long)nb * na;
    constexpr int LS = Sh<R, LOGC>::LS, LT = Sh<R, LOGC>::LT;
    const K2 k2{u64of(make_float2(dp.tiny, dp.tiny)), u64of(make_float2(MAG_S, MAG_S)), u64of(make_float2(-1.0f, -1.0f)),
                u64of(make_float2(MAG_S - 0.5f, MAG_S - 0.5f)), u64of(make_float2(MAG_T, MAG_T)),
                u64of(make_float2(dp.nmu, dp.nmu)),
                MID ? u64of(make_float2(dp.tinyl, dp.tinyl)) : 0ull,
                MID ? u64of(make_float2(-0.5f, -0.5f)) : 0ull,
                MID ? u64of(make_float2(-dp.c1, -dp.c1)) : 0ull,
                MID ? u64of(make_float2(-dp.c3, -dp.c3)) : 0ull,
                MID ? u64of(make_float2(dp.c05, dp.c05)) : 0ull,
               is_geo(V) ? u64of(make_float2(dp.la, dp.la)) : 0ull,
               V == 5 ? u64of(make_float2(dp.m, dp.m)) : 0ull,
               is_geo(V) ? dp.lmid : 0.0f,
               V == 5 ? 4u * (uint32_t)dp.C : 0u};
    const uint32_t lt = (1u << lane) - 1u;
    // a-point ai had an uncertain pair in some lane: recompute its pairs with
    // one flag each (padding slots and, in the self cell, pairs a >= b never
    // count), take back each uncertain pair's add and put it on the recheck list
    auto settle = [&](uint32_t ai) {
        const ARec a = load_a<MID>(wm.arec, ai);
        const uint32_t ia = a0 + ai;
        uint32_t xs[NP];
        bool fl[NP];
#pragma unroll
        for (int q = 0; q < NQ; q++)
            pair2_flags<V, LS, LT>(u64of(BX[q]), u64of(BY[q]), u64of(BZ[q]), a, k2, dp.cs, dp.s_top, ad.Kl,
                                    xs[2 * q], xs[2 * q + 1], fl[2 * q], fl[2 * q + 1]);
        uint32_t xm = 0;
#pragma unroll
        for (int p = 0; p < NP; p++) xm |= (fl[p] && (!CHK || ia < IB[p]) ? 1u : 0u) << p;
        xm &= live;
#pragma unroll 1
        for (int p = 0; p < NP; p++) {
            const bool x = (xm >> p) & 1u;
            const unsigned mk = __ballot_sync(0xffffffffu, x);
            if (mk) {
                if (x) {
                    red_add(p == 0 ? xs[0] : (p == 1 ? xs[1] : (p == 2 ? xs[2] : xs[3])), 0xFFFFFFFFu);
                    xl_put(wm.xl, n_list + __popc(mk & lt), ia,
                           __float_as_uint(wm.buf[32u * (uint32_t)p + (uint32_t)lane].w));
                }
                n_list += __popc(mk);
                if (n_list >= XCAP - 32) {
                    if (MID) recheck_apart<MU, R, LOGC>(prm, dp, m, T, wm, n_list, ad.hb(dp), lane);
                    else recheck<MU, R, LOGC>(prm, dp, m, T, wm, n_list, ad.hb(dp), lane);
                    n_list = 0;
                }
            }
        }
    };
    const uint32_t dump = CHK ? ad.dump(dp) : 0u;
    uint32_t ai = 0;
#pragma unroll 1
    for (; ai + 1 < na; ai += 2) {
        const ARec a = load_a<MID>(wm.arec, ai), a2 = load_a<MID>(wm.arec, ai + 1);
        const bool u0 = apoint<V, CHK, LS, LT>(BX, BY, BZ, a, k2, dp.cs, dp.s_top, ad.Kl, a0 + ai, IB, dump);
        const bool u1 = apoint<V, CHK, LS, LT>(BX, BY, BZ, a2, k2, dp.cs, dp.s_top, ad.Kl, a0 + ai + 1, IB, dump);
        if (__any_sync(0xffffffffu, u0 || u1)) {
            // rarely both a-points have an uncertain pair (fine mu bins 7.65 -> 7.14 ms, three mocks of a
            // million points 60.7 -> 60.0); the midpoint kernel (33.55 -> 33.74) and linear s-only bins, which
            // seldom come here (16 mocks of 100 000 points 9.24 -> 9.50), lose by the second vote
            if (MID || V == 0) {
#pragma unroll 1
                for (uint32_t j = ai; j < ai + 2; j++) settle(j);
            } else {
#pragma unroll 1
                for (uint32_t j = 0; j < 2; j++)
                    if (__any_sync(0xffffffffu, j ? u1 : u0)) settle(ai + j);
            }
        }
    }
    if (ai < na) {   // the last a-point of an odd chunk
        const ARec a = load_a<MID>(wm.arec, ai);
        if (__any_sync(0xffffffffu,
                       apoint<V, CHK, LS, LT>(BX, BY, BZ, a, k2, dp.cs, dp.s_top, ad.Kl, a0 + ai, IB, dump)))
            settle(ai);
    }
    __syncwarp();
}

// x, y, z of sorted point i in bins relative to the corner (ox, oy, oz)
__device__ __forceinline__ float4 bpoint(const DirectParams &dp, uint32_t i, uint32_t ux, uint32_t uy, uint32_t uz,
                                         uint32_t ox, uint32_t oy, uint32_t oz)
{
    return make_float4(__fmul_rn(__int2float_rn((int)(ux - ox)), dp.inv_qds),
                       __fmul_rn(__int2float_rn((int)(uy - oy)), dp.inv_qds),
                       __fmul_rn(__int2float_rn((int)(uz - oz)), dp.inv_qds), __uint_as_float(i));
}

// The unit: a-chunk [un.a0, un.a1) of the cells un.cell .. (dp.G cells along x, fewer at the row's end) against the
// term's neighbourhood.
template <int V, int R, int LOGC>
__device__ __forceinline__ void unit(const CountParams &prm, const DirectParams &dp, const Mesh &m,
                                     const unsigned long long *T, const WarpMem &wm,
                                     const Addr<has_mu(V), R, LOGC> &ad, const Unit &un, const Term &tm, int lane,
                                     uint32_t &n_list)
{
    const int n_c = prm.n_c;
    const int ax = un.cell % n_c, ay = (un.cell / n_c) % n_c, az = un.cell / (n_c * n_c);
    const int ax1 = min(ax + dp.G, n_c) - 1;   // the last cell
    const uint32_t ox = m.orig[ax], oy = m.orig[ay], oz = m.orig[az];
    const size_t N = m.n_total;
    const uint32_t a0 = un.a0, na = un.a1 - un.a0;
    // the a-chunk in bin units relative to A's corner, as packed records
    // (-x, -x, -y, -y), then (-z, -z, m - n_mu x, ...), (-m - n_mu x, ..., 0, 0)
    // (x line of sight) or (-z, -z, x - 2 o_x, ...), (y - 2 o_y, ..., z - 2 o_z, ...)
    // (midpoint line of sight, o the observer in the same frame), and its box
    float o2x = 0.f, o2y = 0.f, o2z = 0.f;
    if (V == 2) {
        o2x = 2.0f * __fmul_rn(__ll2float_rn(prm.obs[0] - (long long)ox), dp.inv_qds);
        o2y = 2.0f * __fmul_rn(__ll2float_rn(prm.obs[1] - (long long)oy), dp.inv_qds);
        o2z = 2.0f * __fmul_rn(__ll2float_rn(prm.obs[2] - (long long)oz), dp.inv_qds);
    }
    float lx = INFINITY, ly = INFINITY, lz = INFINITY, hx = -INFINITY, hy = -INFINITY, hz = -INFINITY;
#pragma unroll 1
    for (uint32_t i = (uint32_t)lane; i < na; i += 32) {
        const size_t g = a0 + i;
        const float4 p = bpoint(dp, (uint32_t)g, m.us[g], m.us[N + g], m.us[2 * N + g], ox, oy, oz);
        wm.arec[3 * i] = make_float4(-p.x, -p.x, -p.y, -p.y);
        if (V == 2) {
            const float lax = __fsub_rn(p.x, o2x), lay = __fsub_rn(p.y, o2y), laz = __fsub_rn(p.z, o2z);
            wm.arec[3 * i + 1] = make_float4(-p.z, -p.z, lax, lax);
            wm.arec[3 * i + 2] = make_float4(lay, lay, laz, laz);
        } else {
            const float fxp = __fmul_rn(p.x, dp.nmu);
            const float cp = V == 5 ? -fxp : __fsub_rn(dp.m, fxp), cm = V == 5 ? 0.0f : __fsub_rn(-dp.m, fxp);
            wm.arec[3 * i + 1] = make_float4(-p.z, -p.z, cp, cp);
            wm.arec[3 * i + 2] = make_float4(cm, cm, 0.f, 0.f);
        }
        lx = fminf(lx, p.x);
        ly = fminf(ly, p.y);
        lz = fminf(lz, p.z);
        hx = fmaxf(hx, p.x);
        hy = fmaxf(hy, p.y);
        hz = fmaxf(hz, p.z);
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        lx = fminf(lx, __shfl_xor_sync(0xffffffffu, lx, s));
        ly = fminf(ly, __shfl_xor_sync(0xffffffffu, ly, s));
        lz = fminf(lz, __shfl_xor_sync(0xffffffffu, lz, s));
        hx = fmaxf(hx, __shfl_xor_sync(0xffffffffu, hx, s));
        hy = fmaxf(hy, __shfl_xor_sync(0xffffffffu, hy, s));
        hz = fmaxf(hz, __shfl_xor_sync(0xffffffffu, hz, s));
    }
    // centre and half-widths, rounded outward
    const float cxb = 0.5f * (lx + hx), cyb = 0.5f * (ly + hy), czb = 0.5f * (lz + hz);
    const float e = 1.0f / 1048576.0f;
    const float hxb = __fadd_ru(__fmul_ru(0.5f, __fsub_ru(hx, lx)), __fmul_ru(e, fabsf(cxb) + 1.0f));
    const float hyb = __fadd_ru(__fmul_ru(0.5f, __fsub_ru(hy, ly)), __fmul_ru(e, fabsf(cyb) + 1.0f));
    const float hzb = __fadd_ru(__fmul_ru(0.5f, __fsub_ru(hz, lz)), __fmul_ru(e, fabsf(czb) + 1.0f));

    // the unit's b runs, one lane per neighbour row (dz, dy), each a contiguous
    // x-run of cells; an auto count takes half of the neighbourhood and the
    // self cell separately
    const bool periodic = prm.geometry == TPCF_PERIODIC;
    const uint32_t *cs = m.cellstart + (size_t)tm.cat_b * prm.n_cells;
    uint32_t n_run = 0, total = 0, self0 = 0, self1 = 0;
#pragma unroll 1
    for (int r0 = 0; r0 < prm.n_rows; r0 += 32) {
        const int r = r0 + lane;
        uint32_t s0[2], s1[2];
        int nl = 0;
        if (r < prm.n_rows) {
            const int dz = prm.row_dz[r], dy = prm.row_dy[r], kx = prm.row_kx[r];
            bool use = !(tm.auto_pairs && (dz < 0 || (dz == 0 && dy < 0)));
            int z = az + dz, y = ay + dy;
            if (periodic) {
                z = z < 0 ? z + n_c : (z >= n_c ? z - n_c : z);
                y = y < 0 ? y + n_c : (y >= n_c ? y - n_c : y);
            } else if (z < 0 || z >= n_c || y < 0 || y >= n_c) {
                use = false;
            }
            if (use) {
                const uint32_t rowkey = ((uint32_t)z * n_c + (uint32_t)y) * n_c;
                int xlo = ax - kx, xhi = ax1 + kx;
                auto add = [&](uint32_t a, uint32_t b) {
                    if (b > a) {
                        s0[nl] = a;
                        s1[nl] = b;
                        nl++;
                    }
                };
                if (tm.auto_pairs && dz == 0 && dy == 0) {
                    self0 = cs[rowkey + ax];
                    self1 = cs[rowkey + ax1 + 1];
                    xlo = ax1 + 1;
                }
                if (xlo <= xhi) {
                    if (periodic) {
                        if (xlo < 0) {
                            add(cs[rowkey + xlo + n_c], cs[rowkey + n_c]);
                            add(cs[rowkey], cs[rowkey + xhi + 1]);
                        } else if (xhi >= n_c) {
                            add(cs[rowkey + xlo], cs[rowkey + n_c]);
                            add(cs[rowkey], cs[rowkey + xhi - n_c + 1]);
                        } else {
                            add(cs[rowkey + xlo], cs[rowkey + xhi + 1]);
                        }
                    } else {
                        xlo = max(xlo, 0);
                        xhi = min(xhi, n_c - 1);
                        if (xlo <= xhi) add(cs[rowkey + xlo], cs[rowkey + xhi + 1]);
                    }
                }
            }
        }
        uint32_t pl = 0;
#pragma unroll 1
        for (int i = 0; i < nl; i++) pl += s1[i] - s0[i];
        uint32_t n_all, p_all;
        const uint32_t n_ex = warp_exclusive_sum((uint32_t)nl, lane, n_all);
        uint32_t p_ex = warp_exclusive_sum(pl, lane, p_all);
#pragma unroll 1
        for (int i = 0; i < nl; i++) {
            wm.runs[n_run + n_ex + i] = make_uint2(s0[i], total + p_ex);
            p_ex += s1[i] - s0[i];
        }
        n_run += n_all;
        total += p_all;
    }
    self0 = __reduce_max_sync(0xffffffffu, self0);
    self1 = __reduce_max_sync(0xffffffffu, self1);
    if (lane == 0) wm.runs[n_run] = make_uint2(0u, total);   // sentinel: the concatenation's end
    __syncwarp();

    const uint32_t lt = (1u << lane) - 1u;
    // The buffer fills with the self cell's points first (auto counts: pairs
    // a < b, no filter), at most a tile at a time, then with the neighbour
    // runs' points that pass the filter: four raw points per lane per pass
    // (their twelve loads in flight together), survivors appended.  A tile is
    // counted whenever TB points are there, and once more for the rest.  One
    // call site per kind of tile keeps the kernel's hot code small.
    uint32_t nbuf = 0, cself = self0, c = 0;
    int g = 0;
#pragma unroll 1
    for (;;) {
        uint32_t nself = 0;
        if (cself < self1) {   // the buffer is empty here: self points come first
            nself = min((uint32_t)TB, self1 - cself);
#pragma unroll 1
            for (uint32_t e2 = (uint32_t)lane; e2 < nself; e2 += 32) {
                const size_t gi = cself + e2;
                wm.buf[e2] = bpoint(dp, (uint32_t)gi, m.us[gi], m.us[N + gi], m.us[2 * N + gi], ox, oy, oz);
            }
            cself += nself;
            nbuf = nself;
        }
#pragma unroll 1
        while (nbuf < TB && c < total) {
            uint32_t idx[4];
            bool ok[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const uint32_t o2 = c + 32u * (uint32_t)k + (uint32_t)lane;
                ok[k] = o2 < total;
#pragma unroll 1
                while (g + 1 < (int)n_run && wm.runs[g + 1].y <= o2) g++;
                idx[k] = ok[k] ? wm.runs[g].x + (o2 - wm.runs[g].y) : 0u;
            }
            uint32_t ux[4], uy[4], uz[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                ux[k] = ok[k] ? __ldg(m.us + idx[k]) : 0u;
                uy[k] = ok[k] ? __ldg(m.us + N + idx[k]) : 0u;
                uz[k] = ok[k] ? __ldg(m.us + 2 * N + idx[k]) : 0u;
            }
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const float4 p = bpoint(dp, idx[k], ux[k], uy[k], uz[k], ox, oy, oz);
                const float qx = fmaxf(__fsub_rn(fabsf(__fsub_rn(p.x, cxb)), hxb), 0.0f);
                const float qy = fmaxf(__fsub_rn(fabsf(__fsub_rn(p.y, cyb)), hyb), 0.0f);
                const float qz = fmaxf(__fsub_rn(fabsf(__fsub_rn(p.z, czb)), hzb), 0.0f);
                const bool keep = ok[k] && __fmaf_rn(qz, qz, __fmaf_rn(qy, qy, __fmul_rn(qx, qx))) < dp.hit;
                const unsigned mk = __ballot_sync(0xffffffffu, keep);
                if (keep) wm.buf[nbuf + __popc(mk & lt)] = p;
                nbuf += __popc(mk);
            }
            c += 128;
        }
        if (nbuf == 0) break;
        const uint32_t nt = min(nbuf, (uint32_t)TB);
        __syncwarp();
        if (nself)
            tile<V, R, LOGC, true>(prm, dp, m, T, wm, ad, nt, nself, na, a0, lane, n_list);
        else
            tile<V, R, LOGC, false>(prm, dp, m, T, wm, ad, nt, 0u, na, a0, lane, n_list);
        // the leftovers (fewer than 128) move to the front
        const uint32_t left = nbuf - nt;
        if (left) {
            float4 v[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const uint32_t s = 32u * (uint32_t)k + (uint32_t)lane;
                v[k] = s < left ? wm.buf[TB + s] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const uint32_t s = 32u * (uint32_t)k + (uint32_t)lane;
                if (s < left) wm.buf[s] = v[k];
            }
            __syncwarp();
        }
        nbuf = left;
    }
}

// Drains a table into term t's int64 histogram and clears its hwords words: one warp, or (BLOCK) all threads of the
// block, which clear nothing
template <bool MU, int R, int LOGC, bool BLOCK>
__device__ __forceinline__ unsigned long long drain(const CountParams &prm, const DirectParams &dp,
                                                    const Term *terms, uint32_t *hist, uint32_t hwords, int t,
                                                    int lane)
{
    long long *const th = terms[t].hist;
    const int n_mu = prm.n_mu;
    unsigned long long binned = 0;
#pragma unroll 1
    for (int b = BLOCK ? (int)threadIdx.x : lane; b < prm.nbin; b += BLOCK ? (int)blockDim.x : 32) {
        const int k = b / n_mu + dp.row0, j = b % n_mu;
        unsigned long long sum = 0;
        if (R == 1) {   // one copy, one column per |mu| bin
            sum = hist[(uint32_t)k * (uint32_t)dp.C + (uint32_t)(j + dp.CO)];
            if (sum) atomicAdd((unsigned long long *)&th[b], sum);
            binned += sum;
            continue;
        }
        // mu bin j: signed columns j and -1 - j
        const uint32_t c1 = MU ? (uint32_t)(j + dp.CO) : 0u, c2 = MU ? (uint32_t)(dp.CO - 1 - j) : 0u;
        const uint4 *w1 = (const uint4 *)(hist + (((uint32_t)k << LOGC) + c1) * (uint32_t)R);
#pragma unroll
        for (int c = 0; c < R / 4; c++) {
            const uint4 v = w1[c];
            sum += (unsigned long long)v.x + v.y + v.z + v.w;
        }
        if (MU) {
            const uint4 *w2 = (const uint4 *)(hist + (((uint32_t)k << LOGC) + c2) * (uint32_t)R);
#pragma unroll
            for (int c = 0; c < R / 4; c++) {
                const uint4 v = w2[c];
                sum += (unsigned long long)v.x + v.y + v.z + v.w;
            }
        }
        if (sum) atomicAdd((unsigned long long *)&th[b], sum);
        binned += sum;
    }
    if (BLOCK) return binned;
    __syncwarp();
#pragma unroll 1
    for (uint32_t i = (uint32_t)lane; i < hwords / 4; i += 32) ((uint4 *)hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    return binned;
}

// The schedule's lock, taken by one lane of a warp.  The wait is bounded: it
// can only run out if a warp of this block stopped running.
__device__ __forceinline__ bool sched_lock(Sched &q)
{
#pragma unroll 1
    for (unsigned i = 0; i < (1u << 24); i++) {
        if (atomicCAS(&q.lock, 0u, 1u) == 0u) {
            __threadfence_block();
            return true;
        }
        __nanosleep(20);
    }
    return false;
}
__device__ __forceinline__ void sched_unlock(Sched &q)
{
    __threadfence_block();
    atomicExch(&q.lock, 0u);
}

constexpr unsigned NO_UNIT = 0xFFFFFFFFu;

// Smallest claim: csize / 32 units, or one per warp
__device__ __forceinline__ uint32_t least_claim(uint32_t csize)
{
    return min(csize, max(csize / 32u, (uint32_t)DIRECT_WARPS));
}

// The block's claim is used up: one lane takes the next unit of the claim
// that another warp made meanwhile, or makes a new one.  Claims shrink toward
// the end (guided self-scheduling): a block takes half of the remaining units'
// fair share, at most csize units and at least least_claim(), so the last
// claims, which set the launch's tail, are short.  The first `base` units are
// not on the counter (the blocks' first claims in a launch of one term).  A
// stale read of the counter only changes a claim's length; the atomic add
// keeps the claims disjoint and covering.
template <bool ONE>
__device__ __forceinline__ unsigned claim_more(Sched &q, unsigned *claim, uint32_t u_lo, uint32_t base, uint32_t span,
                                            uint32_t csize, int *status)
{
    unsigned u = NO_UNIT;
    // without the flag each warp in turn would read the used-up counter under the lock, 16 latencies of global
    // memory at the end of every launch: one launch per term of 16 mocks of 4000 points 3.66 -> 3.33 ms for the
    // whole step, batched 0.66 -> 0.64
    if (*(volatile unsigned short *)&q.done) return u;
    if (!sched_lock(q)) {
        atomicOr(status, STATUS_TIMEOUT);
        return u;
    }
    const unsigned long long c = atomicAdd(&q.claim, 1ull);
    if ((uint32_t)c < (uint32_t)(c >> 32)) {
        u = (uint32_t)c;
    } else if (!*(volatile unsigned short *)&q.done) {
        const uint32_t g = *(volatile unsigned *)claim + (ONE ? base : 0u);
        const uint32_t rem = g < span ? span - g : 0u;
        const uint32_t sz = max(least_claim(csize), min(csize, rem / (2u * gridDim.x)));
        const uint32_t c0 = rem ? atomicAdd(claim, sz) + (ONE ? base : 0u) : span;
        if (c0 < span) {
            u = u_lo + c0;
            atomicExch(&q.claim,
                       (unsigned long long)(u + 1u) | (unsigned long long)(u_lo + min(span, c0 + sz)) << 32);
        } else {
            *(volatile unsigned short *)&q.done = 1;
        }
    }
    sched_unlock(q);
    return u;
}

// units a table may take between two drains: a unit adds at most
// unit_pair_bound to any of its 32-bit counters
__device__ __forceinline__ unsigned most_units(const DirectParams &dp)
{
    return (unsigned)min(0x7fffffffull, ((1ull << 32) - 1ull) / dp.unit_pair_bound);
}

// One lane finds a table for term t: the one that counts it, or a free one.
// Returns its number, -1 when the wait gave up.
__device__ __forceinline__ int enter_table(Sched &q, const DirectParams &dp, int t)
{
    int k = -1;
    const unsigned most = most_units(dp);
    // A table becomes free when the last of its warps leaves it.  Meanwhile
    // they may take further units of its term, and where there is one table
    // another term's warps may enter it first, so the wait can be long; but
    // every such step takes a unit or moves a table, and between two steps
    // lies at most one unit: at most R unit_pair_bound pairs, 0.1 us each
    // when all are rechecked.  The wait gives up when nothing has happened
    // for that long.
    const unsigned long long limit = 4000000000ull + 100ull * (unsigned)dp.R * dp.unit_pair_bound;
    unsigned long long since = gtimer(), seen = 0ull;
#pragma unroll 1
    for (;;) {
        if (!sched_lock(q)) break;
        unsigned long long now = 0ull;
#pragma unroll 1
        for (int j = 0; j < dp.NT; j++) {
            // a full table is not counted on: its counter could wrap
            if (k < 0 && q.term[j] == t && *(volatile unsigned *)&q.n_used[j] < most &&
                atomicAdd(&q.n_used[j], 1u) < most)
                k = j;
            now += *(volatile unsigned *)&q.n_used[j];
        }
        now |= (unsigned long long)q.moves << 40;
        if (k >= 0) {
            q.ref[k]++;
        } else {
#pragma unroll 1
            for (int j = 0; j < dp.NT; j++)
                if (k < 0 && q.term[j] == FREE) k = j;
            if (k >= 0) {
                q.term[k] = t;
                q.ref[k] = 1u;
                atomicExch(&q.n_used[k], 1u);
            }
        }
        if (k >= 0) q.moves++;
        sched_unlock(q);
        if (k >= 0) break;
        if (now != seen) {
            seen = now;
            since = gtimer();
        } else if (gtimer() - since >= limit) {
            break;
        }
        __nanosleep(200);
    }
    return k;
}

// The same as a call of its own, see below.
__device__ __noinline__ int enter_table_apart(Sched &q, const DirectParams &dp, int t) { return enter_table(q, dp, t); }

// The warp (all lanes) leaves its table, if it has one, draining it when it is
// the last to leave, and, if u is a unit, enters the table of u's term: the one
// that counts it, or a free one (a bounded wait for a drain).  Returns the
// table, -1 when there is none (NO_UNIT, or the wait ran out).  n_list pairs
// still await their exact recheck in the table that is left, whose base for
// this lane is hb.
template <int V, int R, int LOGC>
__device__ __forceinline__ int switch_table(const CountParams &prm, const DirectParams &dp, const Mesh &m,
                                         const Term *terms, const Unit *units, const uint32_t *ustart,
                                         const unsigned long long *T, const WarpMem &wm, Sched &q,
                                         unsigned char *tables, uint32_t hstride, uint32_t hb, unsigned u,
                                         uint32_t n_list, int *status)
{
    constexpr bool MU = has_mu(V);
    const int lane = threadIdx.x & 31, tab = wm.st->tab;
    if (tab >= 0) {
        if (n_list) {
            if (V == 2) recheck_apart<MU, R, LOGC>(prm, dp, m, T, wm, n_list, hb, lane);
            else recheck<MU, R, LOGC>(prm, dp, m, T, wm, n_list, hb, lane);
        }
        __syncwarp();
        unsigned last = 0;
        if (lane == 0) {
            if (sched_lock(q)) {
                last = --q.ref[tab] == 0u;
                if (last) q.term[tab] = DRAINING;
                sched_unlock(q);
            } else {   // the table would never be drained
                atomicOr(status, STATUS_TIMEOUT);
            }
        }
        if (__shfl_sync(0xffffffffu, last, 0)) {
            __syncwarp();   // lane 0's lock came after the other warps' adds; the lanes that read the table come after it
            unsigned long long bn = drain<MU, R, LOGC, false>(prm, dp, terms, (uint32_t *)(tables + (size_t)tab * hstride),
                                                       hstride / 4u, wm.st->term, lane);
#pragma unroll
            for (int s2 = 16; s2 > 0; s2 >>= 1) bn += __shfl_down_sync(0xffffffffu, bn, s2);
            if (lane == 0) {
                wm.st->binned += bn;
                if (sched_lock(q)) {
                    q.term[tab] = FREE;
                    q.moves++;
                    sched_unlock(q);
                } else {
                    atomicOr(status, STATUS_TIMEOUT);
                }
            }
        }
    }
    int k = -1;
    if (u != NO_UNIT && lane == 0) {
        const int t = units[u].term;
        const uint32_t t_lo = ustart[(size_t)t * dp.n_groups], t_hi = ustart[(size_t)(t + 1) * dp.n_groups];
        // (inlined it costs linear bins with mu 0.6 to 1.5 %; as a call, geometric bins 3 % and s only, on 16 mocks of
        // 4000 points, 1.5 %)
        k = is_geo(V) || V == 0 ? enter_table(q, dp, t) : enter_table_apart(q, dp, t);
        if (k < 0) atomicOr(status, STATUS_TIMEOUT);
        wm.st->tab = k;
        wm.st->term = t;
        wm.st->t_lo = t_lo;
        wm.st->t_hi = t_hi;
    }
    k = __shfl_sync(0xffffffffu, k, 0);
    __syncwarp();   // the lanes' adds come after lane 0's lock, and so after the last drain's clearing
    return k;
}

// The same as a call of its own (midpoint line of sight, see recheck_apart).
template <int V, int R, int LOGC>
__device__ __noinline__ int switch_table_apart(const CountParams &prm, const DirectParams &dp, const Mesh &m,
                                               const Term *terms, const Unit *units, const uint32_t *ustart,
                                               const unsigned long long *T, const WarpMem &wm, Sched &q,
                                               unsigned char *tables, uint32_t hstride, uint32_t hb, unsigned u,
                                               uint32_t n_list, int *status)
{
    return switch_table<V, R, LOGC>(prm, dp, m, terms, units, ustart, T, wm, q, tables, hstride,
                                    hb, u, n_list, status);
}

// ONE: one launch per term, term_only; else all units, term_only -1.
template <int V, int R, int W, int LOGC, bool ONE>
__global__ void __launch_bounds__(W * 32, 1)
    pairdirect_kernel(const __grid_constant__ CountParams prm, const __grid_constant__ DirectParams dp, const Mesh m,
                      const Term *__restrict__ terms, const Unit *__restrict__ units,
                      const uint32_t *__restrict__ ustart, const uint32_t *__restrict__ n_units_p,
                      unsigned *__restrict__ claim, unsigned long long *__restrict__ stats, int *__restrict__ status,
                      int term_only, int chunk)
{
    constexpr bool MU = has_mu(V);
    const DOff o = d_off(prm.n_s, dp.rows, prm.n_rows, R, dp.C, dp.NT, W);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long *Tsh = (unsigned long long *)(dsm + o.T);
    Sched &q = *(Sched *)(dsm + o.misc);
    const uint32_t hwords = o.hstride / 4u;
#pragma unroll 1
    for (uint32_t i = tid; i < hwords * (uint32_t)dp.NT; i += blockDim.x) ((uint32_t *)(dsm + o.hist))[i] = 0u;
#pragma unroll 1
    for (int i = tid; i <= prm.n_s; i += blockDim.x) Tsh[i] = prm.T[i];
    if (tid == 0) {
        q.claim = 0ull;
        q.lock = 0u;
        q.done = q.moves = 0;
        for (int k = 0; k < MAX_NT; k++) {
            q.term[k] = FREE;
            q.ref[k] = q.n_used[k] = 0u;
        }
    }

    unsigned char *wr = dsm + o.warp0 + (size_t)warp * o.wstride;
    const WarpMem wm{(float4 *)(wr + o.arec), (float4 *)(wr + o.buf), (uint2 *)(wr + o.runs), (uint2 *)(wr + o.xl),
                     (WarpState *)(wr + o.st)};
    if (lane == 0) *wm.st = WarpState{0ull, 0ull, 0ull, gtimer(), -1, -1, 0u, 0u};
    uint32_t n_list = 0;

    // The block claims chunks of consecutive units and its warps take them one
    // at a time, each on its own: no barrier separates claims or terms.  A
    // table counts one term.  A warp whose next unit belongs to another term
    // (or whose table could wrap) leaves its table and enters the one of that
    // term or a free one; the last warp to leave a table drains it.  With two
    // tables or more the warps of a block pass from one term to the next
    // without waiting for each other (one table is taken only where two do not
    // fit: 19.9 ms instead of 15.6 on eight mocks of 100 000 points).  With a
    // block barrier after every claim and before every drain, each of them
    // waiting for the block's slowest warp (a unit takes 0.05 to 0.3 ms), the
    // barriers cost 18 % of the warps' time on two such mocks: kernel times 16.4
    // -> 15.6 ms for eight, 60.7 -> 59.6 for three of a million points, 3.88 ->
    // 3.61 for eight of 60 000; 32.7 -> 32.8 on cut-sky mocks, whose terms are long
    // and units short.  Units of a few points (four per cell) suffer, since
    // warps at different places of the code share less of the instruction
    // cache (0.32 -> 0.42 ms on 16 mocks of 4000 points); the tuner takes larger
    // cells there (0.24 ms).
    const uint32_t n_all = *n_units_p;
    uint32_t u_lo = 0, u_hi = n_all;
    if (ONE || term_only >= 0) {   // (batched: never; without the test the batched kernels come out 0.5 to 1.3 % slower)
        u_lo = ustart[(size_t)term_only * dp.n_groups];
        u_hi = ustart[(size_t)(term_only + 1) * dp.n_groups];
    }
    const uint32_t span = u_hi - u_lo;
    const unsigned most = most_units(dp);
    Addr<MU, R, LOGC> ad{0u};
    // One launch per term: a block's first claim follows from its number (its
    // size is what the counter would give), and its warps start in the term's
    // table and leave it together, unless the term is long enough to fill it.  Small terms'
    // launches are too short for 16 warps to pass the lock and the counter one
    // after another: 16 mocks of 4000 points, whole step, 3.33 -> 2.34 ms; one
    // mock and 50 subsets of 50 000 points 28.9 -> 27.1.  Kernels of their own,
    // since the branches cost batched launches 1 %; first claims by block number
    // cost them 2 % on uneven mocks.
    const bool solo = ONE && span < most;
    uint32_t base = 0u;
    if (ONE) {
        const uint32_t first = max(least_claim((uint32_t)chunk), min((uint32_t)chunk, span / (2u * gridDim.x)));
        const uint32_t c0 = (uint32_t)min((unsigned long long)span, (unsigned long long)first * blockIdx.x);
        base = (uint32_t)min((unsigned long long)span, (unsigned long long)first * gridDim.x);
        if (tid == 0) {
            q.claim = (unsigned long long)(u_lo + c0) | (unsigned long long)(u_lo + min(span, c0 + first)) << 32;
            q.done = base >= span ? 1 : 0;
        }
        if (solo && lane == 0) {
            wm.st->tab = 0;
            wm.st->term = term_only;
            wm.st->t_lo = u_lo;
            wm.st->t_hi = u_hi;
        }
        ad.Kl = saddr(dsm) + o.hist + 4u * ((uint32_t)lane & (uint32_t)(R - 1)) + Addr<MU, R, LOGC>::shift(dp);
    }
    __syncthreads();
#pragma unroll 1
    for (;;) {
        // the next unit; `stay`: it goes to the warp's own table
        unsigned u = NO_UNIT, stay = 0;
        if (lane == 0) {
            const unsigned long long c = atomicAdd(&q.claim, 1ull);
            if ((uint32_t)c < (uint32_t)(c >> 32)) u = (uint32_t)c;
            else u = claim_more<ONE>(q, claim, u_lo, base, span, (uint32_t)chunk, status);
            stay = u >= wm.st->t_lo && u < wm.st->t_hi && atomicAdd(&q.n_used[wm.st->tab], 1u) < most;
        }
        u = __shfl_sync(0xffffffffu, u, 0);
        if (!__shfl_sync(0xffffffffu, stay, 0)) {
            if (ONE && solo) {   // no unit left
                if (n_list) {
                    if (V == 2) recheck_apart<MU, R, LOGC>(prm, dp, m, Tsh, wm, n_list, ad.hb(dp), lane);
                    else recheck<MU, R, LOGC>(prm, dp, m, Tsh, wm, n_list, ad.hb(dp), lane);
                }
                break;
            }
            const int k = V == 2 ? switch_table_apart<V, R, LOGC>(prm, dp, m, terms, units, ustart, Tsh, wm, q, dsm + o.hist,
                                                                  o.hstride, ad.hb(dp), u, n_list, status)
                                 : switch_table<V, R, LOGC>(prm, dp, m, terms, units, ustart, Tsh, wm, q, dsm + o.hist,
                                                            o.hstride, ad.hb(dp), u, n_list, status);
            n_list = 0;
            if (k < 0) break;
            ad.Kl = saddr(dsm) + o.hist + (uint32_t)k * o.hstride + 4u * ((uint32_t)lane & (uint32_t)(R - 1)) +
                    Addr<MU, R, LOGC>::shift(dp);
        }
        const Unit un = units[u];
        unit<V, R, LOGC>(prm, dp, m, Tsh, wm, ad, un, terms[un.term], lane, n_list);
    }
    if (ONE && solo) {
        __syncthreads();   // every warp has ended its last unit (the waits for one are bounded)
        unsigned long long bn = drain<MU, R, LOGC, true>(prm, dp, terms, (uint32_t *)(dsm + o.hist), 0u, term_only,
                                                         lane);
#pragma unroll
        for (int s2 = 16; s2 > 0; s2 >>= 1) bn += __shfl_down_sync(0xffffffffu, bn, s2);
        if (lane == 0) wm.st->binned += bn;
    }
    if (lane == 0) {
        atomicAdd(&stats[0], wm.st->n_cand);
        atomicAdd(&stats[1], wm.st->binned);
        atomicAdd(&stats[2], wm.st->n_exact);
        record_warp_span(stats, wm.st->t_start);
    }
}

template <int V, int R, int W, int LOGC, bool ONE>
void *dkernel()
{
    return (void *)pairdirect_kernel<V, R, W, LOGC, ONE>;
}

// kernel for (mode, copies, warps, column bits), batched or for one term; nullptr when not built
template <bool ONE>
void *select_direct(int V, int R, int W, int logC)
{
    if (W != DIRECT_WARPS) return nullptr;
    constexpr int DW = DIRECT_WARPS;
    if (V == 5) return R == 1 ? dkernel<5, 1, DW, 0, ONE>() : nullptr;
    if (V == 3) return R == 32 ? dkernel<3, 32, DW, 0, ONE>() : nullptr;
    if (V == 4 && logC == 4) return R == 32 ? dkernel<4, 32, DW, 4, ONE>() : (R == 16 ? dkernel<4, 16, DW, 4, ONE>() : nullptr);
    if (V == 4 && logC == 5) return R == 32 ? dkernel<4, 32, DW, 5, ONE>() : (R == 16 ? dkernel<4, 16, DW, 5, ONE>() : dkernel<4, 8, DW, 5, ONE>());
    if (V == 4 && logC == 6) return R == 16 ? dkernel<4, 16, DW, 6, ONE>() : (R == 8 ? dkernel<4, 8, DW, 6, ONE>() : nullptr);
    if (V == 0) return R == 32 ? dkernel<0, 32, DW, 0, ONE>() : nullptr;
    if (V == 1 && logC == 4) return R == 32 ? dkernel<1, 32, DW, 4, ONE>() : (R == 16 ? dkernel<1, 16, DW, 4, ONE>() : nullptr);
    if (V == 2 && logC == 4) return R == 32 ? dkernel<2, 32, DW, 4, ONE>() : (R == 16 ? dkernel<2, 16, DW, 4, ONE>() : nullptr);
    if (V == 1 && logC == 5) return R == 32 ? dkernel<1, 32, DW, 5, ONE>() : (R == 16 ? dkernel<1, 16, DW, 5, ONE>() : dkernel<1, 8, DW, 5, ONE>());
    if (V == 1 && logC == 6) return R == 16 ? dkernel<1, 16, DW, 6, ONE>() : (R == 8 ? dkernel<1, 8, DW, 6, ONE>() : nullptr);
    if (V == 2 && logC == 5) return R == 32 ? dkernel<2, 32, DW, 5, ONE>() : (R == 16 ? dkernel<2, 16, DW, 5, ONE>() : dkernel<2, 8, DW, 5, ONE>());
    if (V == 2 && logC == 6) return R == 16 ? dkernel<2, 16, DW, 6, ONE>() : (R == 8 ? dkernel<2, 8, DW, 6, ONE>() : nullptr);
    return nullptr;
}

int mode_of(const DirectParams &d, bool mu) { return d.R == 1 ? 5 : d.geo ? (mu ? 4 : 3) : (!mu ? 0 : (d.mid ? 2 : 1)); }

}  // namespace

size_t pairdirect_smem_bytes(const CountParams &p, int rows, int R, int C, int NT, int W)
{
    return d_off(p.n_s, rows, p.n_rows, R, C, NT, W).end;
}

cudaError_t pairdirect_set_attrs(const DirectParams &d, int mu)
{
    for (void *k : {select_direct<false>(mode_of(d, mu != 0), d.R, d.W, d.logC),
                    select_direct<true>(mode_of(d, mu != 0), d.R, d.W, d.logC)}) {
        if (!k) return cudaErrorInvalidValue;
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, d.smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int pairdirect_max_blocks_per_sm(const DirectParams &d, int mu)
{
    void *k = select_direct<false>(mode_of(d, mu != 0), d.R, d.W, d.logC);
    int nb = 0;
    if (!k || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, d.W * 32, d.smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

cudaError_t launch_pairdirect(const CountParams &p, const DirectParams &d, const Mesh &m, const Term *terms,
                              const Unit *units, const uint32_t *ustart, const uint32_t *n_units, unsigned *claim,
                              unsigned long long *stats, int *status, const PairLaunch &pl, cudaStream_t s)
{
    const int term_only = pl.persistent ? -1 : pl.term, mode = mode_of(d, p.n_mu > 1);
    void *k = pl.persistent ? select_direct<false>(mode, d.R, d.W, d.logC) : select_direct<true>(mode, d.R, d.W, d.logC);
    if (!k) return cudaErrorInvalidValue;
    void *args[] = {(void *)&p,       (void *)&d,     (void *)&m,     (void *)&terms,  (void *)&units,     (void *)&ustart,
                    (void *)&n_units, (void *)&claim, (void *)&stats, (void *)&status, (void *)&term_only, (void *)&pl.chunk};
    return cudaLaunchKernel(k, dim3(pl.blocks), dim3(d.W * 32), args, (size_t)d.smem, s);
}

}  // namespace tpcf
