// fixed.cuh -- the fixed-point form of an FP64 sweep.
//
// One SM issues an FP64 instruction for a warp every 19 cycles, and one warp
// every 64 whatever its parallelism (measured on GB300; a 32-bit integer
// multiply-add with a 64-bit result issues every 2 to 4).  B_g / g = I - L / g
// has non-negative entries and row sums 1, so a sweep is an average: no entry
// of the result exceeds the largest of the iterate, and a common power-of-two
// scale serves the whole vector.  The FP64 form's sweeps of levels of up to
// kFixRowsMax rows are therefore run on the integer pipe:
//   iterate   X = q 2^32 + r   (q, r: signed 32-bit, |X| < 2^63), y = X 2^-65,
//             rescaled by powers of two so that max |X| stays in [2^62, 2^63)
//             (the sweep's own maximum is reduced with its sums);
//   entries   C_ij = round(w_ij / g 2^60) = c1 2^29 + c0, D_i = sum_j C_ij exactly;
//   row       X_i + round((sum_j C_ij X_j - D_i X_i) 2^-60), all four products
//             exact in 64-bit sums, one rounding to nearest per row (the lanes of a
//             row each cut a few 2^-24 units before it).  Rows of a constant vector
//             give 0, so constant vectors are fixed points, and a mean that is
//             rounded to a whole unit only moves the vector along 1, which the
//             result's projection takes out.
// What it costs in accuracy.  The only rounding of a sweep is half a unit per entry.
// With max |x| = m 2^e, 1 <= m < 2, the unit is 2^-62 2^e, and FP64's last place at the
// largest entry is 2^-52 2^e: the noise of the whole vector, 0.29 sqrt(n) units as a
// standard deviation, is no more than that of one FP64 rounding of its largest
// entry, 0.29 last places, while sqrt(n) <= 2^10, however localised the vector is.
// That is where kFixRowsMax lies; larger levels keep the FP64 kernels.  (FP64 rounds
// several times a sweep, each entry by its own last place, and g - d_i by as much,
// the same way in every sweep.)  A coefficient is off by 2^-61 g, FP64's diagonal by
// 2^-54 g.
// A CPU model of both forms against 64-bit mantissas, 300 / 2,000 sweeps from one
// start, error of the vector: Barabasi-Albert graph of 20K vertices from a random
// start 1.5e-14 / 6.4e-14 (FP64) and 1.6e-16 / 4.2e-16 (here); on a pendant path of ten
// vertices 1.2e-14 / 3.8e-14 and 2.7e-17 / 4.3e-17, 65K vertices 1.8e-14 / 6.6e-14 and
// 5.8e-17 / 8.3e-17; on one vertex behind an edge of weight 0.01, the one kind where
// FP64 can be closer (its roundings there lie along the vector), 20K 6.3e-17 / 1.1e-16
// and 4.7e-17 / 5.1e-17, 300 sweeps on 250K 3.1e-17 and 2.2e-16, on 1M 2.4e-17 and
// 5.1e-16: no more than the roundings of the result itself.  (With 57 bits and
// the products r c0 dropped: 3.4e-15 / 3.8e-15 on the path, 6.1e-15 / 6.5e-15 on the
// vertex.)
// The stop sums (sum y, sum y^2, sum y y_prev) are integers as well, taken from X
// rounded to 60 bits, and the same in every order of addition.
#pragma once

#include "pi_kernels.cuh"

namespace cmg {

// ------------------------------------------------------------------ plan
constexpr int kFixMaxN = 4096;        // rows of a level k_power_fix takes
constexpr int kFixRowsMax = 1 << 20;  // rows of a level any fixed-point kernel takes (see above)

// What a plan kernel reports to the host.
struct PlanOut {
    int P;                     // CTAs (at most the number asked for)
    int ni;
    int max_e, max_i, max_r;   // most entries, items and rows of one CTA
    long long entries;
    int maxdeg;
    int by_warp;               // k_plan_small: one item of at most this many steps per warp (0: no)
};

// A level for k_plan_small: its CSR, g's reciprocal (fix_weight), steps per lane,
// CTAs, and the arrays to fill with their capacities.
struct SmallJob {
    int n, S, C, cap_items, ni;
    int one_cta, cap_warps;   // most items the one-per-warp form takes in one CTA, and in all
    const int *rp, *col;
    const double *w;
    unsigned long long ginv;
    int ge;
    int4 *item;
    int *range, *perm;
    uint16_t *inv;             // scratch
    uint16_t *ucol;
    int2 *uc, *ud;             // k_fill_small: ni items
    PlanOut *out;
};
// The levels of a hierarchy, by value: a launch holds its own copy, so the host's may
// change or go.  (Coarsening at least halves the vertices that have an edge, so a
// hierarchy has at most 13 such levels of up to kFixMaxN rows.)
constexpr int kSmallJobs = 16;
struct SmallJobs {
    SmallJob j[kSmallJobs];
};
static_assert(sizeof(SmallJobs) <= 4000, "kernel parameters");
cmg_status_t launch_plan_small(const SmallJobs &jobs, int count, cudaStream_t s);
cmg_status_t launch_fill_small(const SmallJobs &jobs, int count, cudaStream_t s);

// ------------------------------------------------------------------ arithmetic
constexpr int kFixTop = 63;   // |X| < 2^63; y = X 2^-65

__device__ __forceinline__ long long mad_s(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// X = q 2^32 + r
__device__ __forceinline__ int2 fix_split(long long X) {
    return make_int2((int)((X + (1ll << 31)) >> 32), (int)(unsigned)X);
}
__device__ __forceinline__ long long fix_join(int2 x) { return (long long)((unsigned long long)x.x << 32) + x.y; }

// C = c1 2^29 + c0 (|c0| <= 2^28, |c1| <= 2^30)
__device__ __forceinline__ int2 fix_split_c(long long C) {
    const int q = (int)((C + (1ll << 28)) >> 29);
    return make_int2(q, (int)(C - ((long long)q << 29)));
}

// round(w / g 2^60) for 0 < w <= g / 2: w as a normalised 64-bit mantissa times
// the 64-bit reciprocal of g's (G = ginv: 2^127 / mantissa, ge: exponent).
__device__ __forceinline__ long long fix_weight(double w, unsigned long long ginv, int ge) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(w);
    const int ef = (int)((b >> 52) & 0x7ffull);
    unsigned long long m = b & 0xfffffffffffffull;
    if (ef) m |= 1ull << 52;
    if (m == 0) return 0;
    const int lz = __clzll((long long)m);
    m <<= lz;
    const int we = (ef ? ef : 1) - 1075 - lz;        // w = m 2^we
    const unsigned long long h = __umul64hi(m, ginv);  // w / g = h 2^(we - ge - 63)
    const int sh = 3 - (we - ge);                     // times 2^60: h >> sh
    if (sh >= 64) return 0;
    if (sh < 1) return 1ll << 59;   // w > g / 2: not a weight of this level
    return (long long)((h >> sh) + ((h >> (sh - 1)) & 1ull));
}

// Accumulators of one lane's part of a row: hi in units of 2^61, m1 of 2^32, m2 of
// 2^29 and m0 of 1 (of the product X C).  The coefficients of a row and its diagonal
// add up to at most 2^60, so |hi| <= 2^62 and |m2| <= 2^62 over any row; m1 and m0 take
// 15 products (at most 2^59 each) between carries.
struct FixAcc {
    long long hi, m1, m2, m0;
    __device__ __forceinline__ void reset() { hi = m1 = m2 = m0 = 0; }
    __device__ __forceinline__ void add(int2 x, int2 c) {
        hi = mad_s(x.x, c.x, hi);
        m1 = mad_s(x.x, c.y, m1);
        m2 = mad_s(x.y, c.x, m2);
        m0 = mad_s(x.y, c.y, m0);
    }
    // after at most 15 entries
    __device__ __forceinline__ void carry() {
        m1 += m0 >> 32;
        m0 &= 0xffffffffll;
        hi += m1 >> 29;
        m1 &= (1ll << 29) - 1;
    }
    // round(product 2^-60) of the sum over aligned groups of 2^lg lanes (after carry):
    // the lanes' parts below 2^61 travel in units of 2^36, so that a row of 32
    // lanes is rounded once, like a row of one (cutting them at the result's unit
    // would shift every row the same way, sweep after sweep).
    __device__ __forceinline__ long long lanes(int lg) const {
        unsigned long long h = (unsigned long long)(hi + (m2 >> 32));
        unsigned l = ((unsigned)m1 >> 4) + ((unsigned)m2 >> 7);   // < 2^26 (m0 is below its unit)
        for (int o = (1 << lg) >> 1; o > 0; o >>= 1) {
            h += __shfl_xor_sync(0xffffffffu, h, o);
            l += __shfl_xor_sync(0xffffffffu, l, o);
        }
        return (long long)(2 * h) + (long long)((l + (1u << 23)) >> 24);
    }
};

// One lane's entries of an item in shared memory: `steps` (a multiple of 4) entries
// 32 apart from col / cf on, four at a time (columns, then values, then products).
template <typename IDX, typename LD>
__device__ __forceinline__ void fix_quads(FixAcc &t, int steps, const IDX *col, const int2 *cf, LD ldx) {
    int u = 0;
    for (; u + 8 <= steps; u += 8, col += 256, cf += 256) {
        int cc[8];
        int2 xx[8];
#pragma unroll
        for (int j = 0; j < 8; j++) cc[j] = (int)col[32 * j];
#pragma unroll
        for (int j = 0; j < 8; j++) xx[j] = ldx(cc[j]);
#pragma unroll
        for (int j = 0; j < 8; j++) t.add(xx[j], cf[32 * j]);
        t.carry();
    }
    if (u < steps) {
        int cc[4];
        int2 xx[4];
#pragma unroll
        for (int j = 0; j < 4; j++) cc[j] = (int)col[32 * j];
#pragma unroll
        for (int j = 0; j < 4; j++) xx[j] = ldx(cc[j]);
#pragma unroll
        for (int j = 0; j < 4; j++) t.add(xx[j], cf[32 * j]);
    }
    t.carry();
}

// The row's new value: p is the rounded product of its entries and of its diagonal
// (-D_i).
__device__ __forceinline__ long long fix_row(long long X, long long p, long long M, int e) {
    return (long long)((unsigned long long)(X + p - M) << e);
}

// Stop sums of the rows a lane computed in one sweep: A in units of X (modulo 2^64:
// the total is a few units a row), the others of X' = X / 8 rounded, |X'| <= 2^60 =
// q 2^32 + r: B = Bh 2^64 + Bm 2^37, C = Ch 2^64 + Cm 2^36.  Up to 64 rows fit
// (q^2 <= 2^56).
struct FixSum {
    long long A, Bh, Bm, Ch, Cm;
    unsigned mx;   // max |q| of X
    __device__ __forceinline__ void reset() {
        A = Bh = Bm = Ch = Cm = 0;
        mx = 0;
    }
    static __device__ __forceinline__ int2 narrow(long long X) { return fix_split((X + 4) >> 3); }   // X'
    __device__ __forceinline__ void square(int2 y, int2 q) {
        Bh = mad_s(y.x, y.x, Bh);
        // X'^2 = q^2 2^64 + (q r + r^2 / 2^33) 2^33
        Bm += mad_s(y.x, y.y, mad_s(y.y, y.y, 0) >> 33) >> 4;
        mx = max(mx, (unsigned)abs(q.x));
    }
    // a row whose value became Y = q; y, x: X' of the new and the old value
    __device__ __forceinline__ void add(long long Y, int2 q, int2 y, int2 x) {
        A += Y;
        square(y, q);
        Ch = mad_s(y.x, x.x, Ch);
        Cm += mad_s(y.x, x.y, mad_s(y.y, x.x, mad_s(y.y, x.y, 0) >> 32)) >> 4;
    }
    // an entry of the start vector, whose sum is far from 0: its low 20 bits to A,
    // the others to Ch
    __device__ __forceinline__ void add_start(long long X, int2 q) {
        A += X & 0xfffff;
        Ch += X >> 20;
        square(narrow(X), q);
    }
};

constexpr int kFixSums = 6;   // 64-bit words of a record of sums: five values and max |q|

// A lane's sums in five 64-bit values whose totals fit: A, then B as U 2^80 + V 2^37 and
// C as U 2^80 + V 2^36 (units of X'^2).  A row adds at most 2^40 to a U and a lane
// 2^44 to a V: 2^22 rows and 2^18.9 lanes fit (the kernels have at most 2^17.3).
// start: A's two parts and B.
struct FixVals {
    long long v[5];
};
__device__ __forceinline__ FixVals fix_vals(const FixSum &f, bool start) {
    FixVals r;
    const long long bh = f.Bh + (f.Bm >> 27), ch = f.Ch + (f.Cm >> 28);
    r.v[0] = f.A;
    r.v[1] = bh >> 16;
    r.v[2] = ((bh & 0xffff) << 27) + (f.Bm & ((1ll << 27) - 1));
    r.v[3] = start ? f.Ch : ch >> 16;
    r.v[4] = start ? 0 : ((ch & 0xffff) << 28) + (f.Cm & ((1ll << 28) - 1));
    return r;
}

// The same values of a single row that went from x to Y = y, in fewer steps (one row
// fits without the narrower X').
__device__ __forceinline__ FixVals fix_vals_row(long long Y, int2 y, int2 x) {
    FixVals r;
    // X^2 = bh 2^64 + (bm mod 2^31) 2^33, X P = ch 2^64 + (cm mod 2^32) 2^32
    const long long bm = mad_s(y.x, y.y, mad_s(y.y, y.y, 0) >> 33), bh = mad_s(y.x, y.x, bm >> 31);
    const long long cm = mad_s(y.x, x.y, mad_s(y.y, x.x, mad_s(y.y, x.y, 0) >> 32)), ch = mad_s(y.x, x.x, cm >> 32);
    r.v[0] = Y;
    r.v[1] = bh >> 22;   // X^2 = 64 X'^2
    r.v[2] = ((bh & 0x3fffff) << 21) + (((unsigned)bm & 0x7fffffffu) >> 10);
    r.v[3] = ch >> 22;
    r.v[4] = ((ch & 0x3fffff) << 22) + ((unsigned)cm >> 10);
    return r;
}

// Warp sums of the five values: value 0 in lanes 0..3, 1 in 4..7, 2 in 8..11, 3 in
// 16..19, 4 in 20..23 (the lanes halve what they carry at each of the first
// three exchanges: 16 shuffles instead of 50).
__device__ __forceinline__ long long fix_warp_vals(const FixVals &f, int lane) {
    auto ex = [](long long v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); };
    bool b = lane & 16;
    long long a0 = (b ? f.v[3] : f.v[0]) + ex(b ? f.v[0] : f.v[3], 16);
    long long a1 = (b ? f.v[4] : f.v[1]) + ex(b ? f.v[1] : f.v[4], 16);
    long long a2 = (b ? 0ll : f.v[2]) + ex(b ? f.v[2] : 0ll, 16);
    b = lane & 8;
    const long long c0 = (b ? a2 : a0) + ex(b ? a0 : a2, 8);
    const long long c1 = (b ? 0ll : a1) + ex(b ? a1 : 0ll, 8);
    b = lane & 4;
    long long e = (b ? c1 : c0) + ex(b ? c0 : c1, 4);
    e += ex(e, 2);
    e += ex(e, 1);
    return e;
}

// A warp's sums as a record of kFixSums words.
__device__ __forceinline__ void fix_warp_record(const FixSum &f, bool start, int lane, long long *rec) {
    const unsigned m = __reduce_max_sync(0xffffffffu, f.mx);
    long long v = fix_warp_vals(fix_vals(f, start), lane);
    const int grp = lane >> 2;
    if (grp == 6) v = (long long)m;
    if ((lane & 3) == 0 && grp != 3 && grp != 7) rec[grp < 3 ? grp : grp - 1] = v;
    __syncwarp();
}

// Sum of `count` records (16-byte aligned) by one warp: value by lane group as
// fix_warp_vals leaves it, and max |q| of all.
__device__ __forceinline__ long long fix_sum_records(const long long *rec, int count, int lane, unsigned *mx) {
    FixVals f;
    unsigned m = 0;
#pragma unroll
    for (int j = 0; j < 5; j++) f.v[j] = 0;
    for (int r = lane; r < count; r += 32) {
        const longlong2 *src = reinterpret_cast<const longlong2 *>(rec + (size_t)r * kFixSums);
        const longlong2 u0 = src[0], u1 = src[1], u2 = src[2];
        f.v[0] += u0.x;
        f.v[1] += u0.y;
        f.v[2] += u1.x;
        f.v[3] += u1.y;
        f.v[4] += u2.x;
        m = max(m, (unsigned)u2.y);
    }
    *mx = __reduce_max_sync(0xffffffffu, m);
    return fix_warp_vals(f, lane);
}

// Slot of a fixed-point sweep: mean to subtract, rescale, decisions.
struct FixSlot {
    long long M;
    int e, stop;
};

// State of the control warp, by lane where noted (the warp runs one chain per sweep
// whose length is instructions, fetched anew every sweep behind the row warps'
// code: the decisions are taken with a few FP64 instructions on the totals, whose
// pipe the sweeps leave idle, where ctrl_step's float-float form takes 300 FP32
// instructions).
struct FixCtl {
    double B, K, Z;    // lanes 4..7: ||y||^2 of the last sweep, times (1 - tol)^2,
                       // times the annihilation threshold of the next
    double C, Bp;      // lanes 16..19: the last y . y_prev; lanes 4..7: B before
    double muA;        // sum y of the last sweep (X units), every lane
    double mu_p;
    long long M;       // mean subtracted in the next sweep
    int e;             // rescale of the next sweep
};

// One control step for sweep s >= 1 (ctrl_step's decisions): v is the sweep's
// total of the lane's value (fix_warp_vals' placement), mx its max |q|.
// Returns 0, 1 (converged) or 2 (annihilated); *next: M, e of sweep s + 2.
__device__ __forceinline__ int fix_decide(const PiArgs &a, int lane, long long v, unsigned mx, double omt2, float inv_n,
                                          FixCtl &c, FixSlot *next) {
    const int grp = lane >> 2;
    // value to double, in units of y y (2^124 of X' X') or, for A, of X
    double d = __ll2double_rn(v);
    const int sh = grp == 0 ? 0 : (grp == 1 || grp == 4 ? -44 : (grp == 2 ? -87 : -88));
    if (v != 0) d = __hiloint2double(__double2hiint(d) + (sh << 20), __double2loint(d));
    const double up = __shfl_down_sync(0xffffffffu, d, 4);
    const double t = d + up;                 // lanes 4..7: B, 16..19: C
    const double f = grp == 1 ? c.K : t;     // lanes 4..7: B K, 16..19: C C
    const double p = t * f;
    // cos >= 1 - tol  <=>  C > 0 and C^2 >= (1 - tol)^2 B B_prev; the products are
    // non-negative doubles and order as integers
    const double cc = __shfl_sync(0xffffffffu, p, 16);
    const double cv = __shfl_sync(0xffffffffu, t, 16);
    const bool zero = __double_as_longlong(t) <= __double_as_longlong(c.Z);
    const bool conv = cv > 0.0 && __double_as_longlong(cc) >= __double_as_longlong(p);
    const int code = __shfl_sync(0xffffffffu, zero ? 2 : (conv ? 1 : 0), 4);
    const double A = __shfl_sync(0xffffffffu, d, 0);
    c.C = cv;
    c.Bp = c.B;
    c.mu_p = c.muA;
    c.muA = A;
    c.B = t;
    // mean of the next sweep, predicted: 2^e (mean - M); a few units
    const float m = (float)A * inv_n - (float)c.M;
    const long long Mn = (long long)__float2int_rn(c.e ? ldexpf(m, c.e) : m);
    // |X_s| < (mx + 1) 2^32, and an average, less a mean of a few units, stays below
    // (mx + 2) 2^32 2^e: lift that to 2^63 (q must stay below 2^31)
    const int en = min(24, max(0, __clz((int)(mx + 2)) - 1 - c.e));
    c.K = omt2 * t;
    c.Z = t * (double)(c.e ? ldexpf(a.zero_tol2, 2 * c.e) : a.zero_tol2);
    next->M = Mn;
    next->e = en;
    c.M = Mn;
    c.e = en;
    return code;
}

// State and first slots from the start vector's totals (value by lane group, as
// fix_warp_vals leaves a start's).
__device__ __forceinline__ void fix_ctl_start(const PiArgs &a, int lane, long long v, double omt2, int n, FixCtl &c,
                                              FixSlot *slots) {
    const int grp = lane >> 2;
    double d = __ll2double_rn(v);
    if (grp == 1) d *= 0x1p-44;
    if (grp == 2) d *= 0x1p-87;
    const double B = __shfl_sync(0xffffffffu, d, 4) + __shfl_sync(0xffffffffu, d, 8);
    const double A = fma(__shfl_sync(0xffffffffu, d, 16), 0x1p20, __shfl_sync(0xffffffffu, d, 0));
    const long long lo = __shfl_sync(0xffffffffu, v, 0), hi = __shfl_sync(0xffffffffu, v, 16);
    const double mu0 = A * 0x1p-65 / (double)n;
    double ss0 = B - (double)n * mu0 * mu0;
    if (ss0 < 0.0) ss0 = 0.0;
    c.B = c.Bp = ss0;
    c.K = omt2 * ss0;
    c.Z = ss0 * (double)a.zero_tol2;
    c.C = 0.0;
    c.muA = c.mu_p = A;
    c.M = 0;
    c.e = 0;
    if (lane == 0) {
        // sweep 1: the mean of y_0 to a unit, from the integer sums
        const long long m = hi / n;
        slots[1].M = m * (1ll << 20) + ((hi - m * n) * (1ll << 20) + lo + n / 2) / n;
        slots[1].e = 0;
        slots[1].stop = 0;
        slots[0].M = 0;   // sweep 2: m_1 = 0
        slots[0].e = 0;
        slots[0].stop = 0;
    }
}

// Result of a run whose last decided sweep is rs with `code` (fix_decide); buf:
// the ring slot of sweep rs.  res[0..1]: rs, annihilated.
__device__ __forceinline__ void fix_finish(const PiArgs &a, int lane, int n, int rs, int code, bool counted, bool bad,
                                           bool writes, int buf, const FixCtl &c, int *res) {
    const double to_mean = 0x1p-65 / (double)n;
    const double B = __shfl_sync(0xffffffffu, c.B, 4), Bp = __shfl_sync(0xffffffffu, c.Bp, 4);
    if (lane != 0) return;
    const bool zero = code == 2;
    res[0] = rs;
    res[1] = zero;
    if (!writes) return;
    PiResult r;
    const double ss = zero ? Bp : B;
    r.mu = (zero ? c.mu_p : c.muA) * to_mean;
    r.inv_s = ss > 0.0 ? 1.0 / sqrt(ss) : 0.0;
    const double den = sqrt(B * Bp);
    r.cos = rs == 0 ? 0.0 : (zero ? 1.0 : (den > 0.0 ? c.C / den : 1.0));
    r.mu_prev = c.mu_p * to_mean;
    r.inv_s_prev = Bp > 0.0 ? 1.0 / sqrt(Bp) : 0.0;
    r.buf = zero ? (buf + 2) % 3 : buf;
    r.buf_prev = (buf + 2) % 3;
    r.sweeps = rs;
    r.capped = counted && a.mode == 0 && code == 0 ? 1 : 0;
    r.zero = zero;
    r.pad = 0;
    if (bad) {
        // an infinity or NaN in the start vector: no sweep converges and every
        // one returns NaN, so none is run
        r.mu = r.cos = r.mu_prev = nan("");
        r.sweeps = a.mode == 1 ? max(a.k_fixed, 0) : a.max_sweeps;
        r.capped = a.mode == 0 ? 1 : 0;
    }
    *a.res = r;
}

__device__ __forceinline__ double fix_value(int2 x) {
    return fma((double)x.x, 0x1p32, (double)x.y) * 0x1p-65;
}

// The exponent k that scales a start vector of largest magnitude m (finite,
// > 0) to |x| 2^k in [2^61, 2^62): the first sweep subtracts a mean of that size.
__device__ __forceinline__ int fix_start_exponent(double m) {
    int ex;
    frexp(m, &ex);   // m = f 2^ex, f in [0.5, 1)
    return kFixTop - 1 - ex;
}

// The start vector of a level held by one CTA or cluster, the same in every CTA:
// values as doubles in ring slot 0, their largest magnitude, then fixed point; the
// warps' sums to s_rec (fix_warp_record).  *s_bad: an entry is not finite (the
// vector is then 0).  Every thread of the CTA calls it; ends with a CTA barrier.
__device__ __forceinline__ void fix_start(const PiArgs &a, int2 *ring, double *s_mx, long long (*s_rec)[kFixSums],
                                          int *s_bad) {
    const int n = a.n, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const void *cb = nullptr;
    double cmu = 0.0, cinv = 0.0;
    if (a.start == 1) {
        cb = a.cbuf[a.cres->buf];
        cmu = a.cres->mu;
        cinv = a.cres->inv_s;
    }
    if (tid == 0) *s_bad = 0;
    __syncthreads();
    double mx = 0.0;
    int bad = 0;
    for (int i = tid; i < n; i += blockDim.x) {
        const double v = start_value(a, a.perm[i], cb, cmu, cinv);
        reinterpret_cast<double *>(ring)[i] = v;
        if (isfinite(v)) mx = fmax(mx, fabs(v));
        else bad = 1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) s_mx[warp] = mx;
    if (bad) *s_bad = 1;
    __syncthreads();
    mx = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) mx = fmax(mx, s_mx[w]);
    const int k = mx > 0.0 ? fix_start_exponent(mx) : 0;
    FixSum f;
    f.reset();
    for (int i = tid; i < n; i += blockDim.x) {
        const double v = reinterpret_cast<double *>(ring)[i];
        const long long X = *s_bad ? 0 : __double2ll_rn(ldexp(v, k));
        const int2 x = fix_split(X);
        f.add_start(X, x);
        ring[i] = x;
    }
    fix_warp_record(f, true, lane, s_rec[warp]);
    __syncthreads();
}

// The reciprocal fix_weight takes: false when g is not a positive finite number.
bool fix_reciprocal(double g, unsigned long long *ginv, int *ge);

}  // namespace cmg
