// fixed.cuh -- the fixed-point form of an FP64 sweep.
//
// One SM issues an FP64 instruction for a warp every 19 cycles, and one warp
// every 64 whatever its parallelism (measured on GB300; a 32-bit integer
// multiply-add with a 64-bit result issues every 2 to 4).  B_g / g = I - L / g
// has non-negative entries and row sums 1, so a sweep is an average: no entry
// of the result exceeds the largest of the iterate, and a common power-of-two
// scale serves the whole vector.  The FP64 form's sweeps are therefore run on
// the integer pipe, in 60-bit fixed point:
//   iterate   X = q 2^29 + r   (q, r: signed 32-bit, |r| <= 2^28, |X| < 2^59),
//             y = X 2^-58, rescaled by powers of two so that max |X| stays near
//             2^56 (the sweep's own maximum is reduced with its sums);
//   entries   C_ij = round(w_ij / g 2^60) = c1 2^29 + c0, D_i = sum_j C_ij exactly
//             (constant vectors are fixed points, as in exact arithmetic);
//   row       X_i - D_i X_i + sum_j C_ij X_j with the products q c1 and
//             q c0 + r c1 accumulated in two 64-bit sums (r c0, below 2^-4 units
//             of the result's last bit, is dropped), rounded once.
// A sweep's rounding error is half a unit of 2^-55 to 2^-56 relative to max |x|, where
// FP64's three roundings of g u - L u are about 2^-53 of each entry and of g - d_i:
// over the families and sizes of the tests, and the timed cases, the vector's
// error against a 64-bit reference is no larger than the FP64 sweeps' was.
// The stop sums (sum y, sum y^2, sum y y_prev) are integers as well: exact to
// 2^-28 of the last bit's square, and the same in every order of addition.
#pragma once

#include "pi_kernels.cuh"

namespace cmg {

// ------------------------------------------------------------------ plan
constexpr int kFixMaxN = 4096;   // rows of a level k_power_fix takes

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
cmg_status_t launch_plan_small(const SmallJob *jobs_dev, int count, cudaStream_t s);
cmg_status_t launch_fill_small(const SmallJob *jobs_dev, int count, cudaStream_t s);

// ------------------------------------------------------------------ arithmetic
constexpr int kFixBits = 58;   // y = X 2^-58

__device__ __forceinline__ long long mad_s(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

__device__ __forceinline__ int2 fix_split(long long X) {
    const int q = (int)((X + (1ll << 28)) >> 29);
    return make_int2(q, (int)(X - ((long long)q << 29)));
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

// Accumulators of one lane's part of a row: hi in units of 2^58, m1 and m2 of 2^29
// (of the product X C).  m1 takes at most 32 products q c0 (below 2^55 each)
// between carries; three chains, since a multiply-add waits for its own.
struct FixAcc {
    long long hi, m1, m2;
    __device__ __forceinline__ void reset() { hi = m1 = m2 = 0; }
    __device__ __forceinline__ void add(int2 x, int2 c) {
        hi = mad_s(x.x, c.x, hi);
        m1 = mad_s(x.x, c.y, m1);
        m2 = mad_s(x.y, c.x, m2);
    }
    // after at most 32 entries
    __device__ __forceinline__ void carry() {
        m1 += m2;
        hi += m1 >> 29;
        m1 &= (1ll << 29) - 1;
        m2 = 0;
    }
    // the accumulated product / 2^60 in sixteenths, and its sum over aligned
    // groups of 2^lg lanes (after carry).  Each lane rounds to nearest: cutting here
    // shifts a row by up to half a unit per sweep in the same direction, and
    // thousands of sweeps add that up (1e-12 in lambda2 on a power-law graph).
    __device__ __forceinline__ long long lanes(int lg) const {
        long long v = (hi << 2) + ((m1 + (1ll << 26)) >> 27);
        for (int o = (1 << lg) >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
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
        if ((u & 24) == 24) t.carry();
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

// The row's new value: p is the lane-summed product of its entries and of its
// diagonal (-D_i) in sixteenths.
__device__ __forceinline__ long long fix_row(int2 xi, long long p, long long M, int e) {
    const long long X = ((long long)xi.x << 29) + xi.y;
    return (X + ((p + 8) >> 4) - M) << e;
}

// Stop sums of the rows a lane computed in one sweep.
struct FixSum {
    long long A, Bh, Bm, Ch, Cm;
    unsigned mx;
    __device__ __forceinline__ void reset() {
        A = Bh = Bm = Ch = Cm = 0;
        mx = 0;
    }
    __device__ __forceinline__ void add(long long Y, int2 y, int2 x) {
        A += Y;
        Bh = mad_s(y.x, y.x, Bh);
        // X^2 = q^2 2^58 + (q r + r^2 / 2^30) 2^30, and likewise X P
        Bm = mad_s(y.x, y.y, Bm) + (mad_s(y.y, y.y, 1ll << 29) >> 30);
        Ch = mad_s(y.x, x.x, Ch);
        Cm = mad_s(y.x, x.y, mad_s(y.y, x.x, Cm)) + (mad_s(y.y, x.y, 1ll << 28) >> 29);
        mx = max(mx, (unsigned)abs(y.x));
    }
};

// A sweep's sums as 16 words that add with 32-bit atomics in any order: three
// words of 22 bits (the third signed) per sum, then max |q|.  Totals of up to
// 2^14 rows fit.
constexpr int kFixWords = 16;

// The three words of a warp's 64-bit sum (carried, so that the words of up to
// 1,023 warps add without overflow); every lane receives them.
__device__ __forceinline__ void fix_warp_words(long long v, unsigned (&w)[3]) {
    unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)v & 0x3fffffu);
    unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 22) & 0x3fffffu);
    unsigned s2 = __reduce_add_sync(0xffffffffu, (unsigned)(int)(v >> 44));
    s1 += s0 >> 22;
    w[0] = s0 & 0x3fffffu;
    w[2] = s2 + (s1 >> 22);
    w[1] = s1 & 0x3fffffu;
}

// A lane's sums in five 64-bit values whose totals over up to 4,096 rows fit: A (its
// total is near 0: exact modulo 2^64), then B as U 2^74 + V 2^30 and C as
// U 2^74 + V 2^29 (units of X^2).
struct FixVals {
    long long v[5];
};
__device__ __forceinline__ FixVals fix_vals(const FixSum &f) {
    FixVals r;
    const long long bh = f.Bh + (f.Bm >> 28), ch = f.Ch + (f.Cm >> 29);
    r.v[0] = f.A;
    r.v[1] = bh >> 16;
    r.v[2] = ((bh & 0xffff) << 28) + (f.Bm & ((1ll << 28) - 1));
    r.v[3] = ch >> 16;
    r.v[4] = ((ch & 0xffff) << 29) + (f.Cm & ((1ll << 29) - 1));
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

// Float-float of v 2^e by integer operations (a 64-bit conversion takes about 160
// cycles): the leading 24 bits, then the next 24, truncated.  Exponents must stay
// in the floats' range.
__device__ __forceinline__ ff fix_ff(long long v, int e) {
    const unsigned sign = v < 0 ? 0x80000000u : 0u;
    unsigned long long m = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
    if (m == 0) return ff_zero();
    const int lz = __clzll((long long)m);
    m <<= lz;                                    // value = m 2^(e - lz)
    const int x = 63 - lz + e;                   // exponent of the leading bit
    const float h = __uint_as_float(sign | ((unsigned)(x + 127) << 23) | ((unsigned)(m >> 40) & 0x7fffffu));
    const unsigned r = (unsigned)(m >> 16) & 0xffffffu;
    const float l = __uint2float_rn(r) * __uint_as_float((unsigned)(x - 47 + 127) << 23);
    return fast_two_sum(h, sign ? -l : l);
}

// Stop sums in units of y from the total words (lane l holds word l, l < 16);
// every lane receives them, and max |q| through *mx.
__device__ __forceinline__ Part fix_part(unsigned word, int lane, unsigned *mx) {
    *mx = __shfl_sync(0xffffffffu, word, 15);
    // lane k < 5: sum k = w0 + 2^22 w1 + 2^44 w2
    const unsigned w0 = __shfl_sync(0xffffffffu, word, min(3 * lane, 31));
    const unsigned w1 = __shfl_sync(0xffffffffu, word, min(3 * lane + 1, 31));
    const int w2 = (int)__shfl_sync(0xffffffffu, word, min(3 * lane + 2, 31));
    const long long top = ((long long)w2 << 22) + (long long)w1 + (long long)(w0 >> 22);   // units of 2^22
    // the low 22 bits are below 2^-48 of any sum that matters beside them
    ff s = fix_ff(top, 22);
    s = ff_add_f(s, (float)(w0 & 0x3fffffu));
    auto get = [&](int k) {
        return ff_make(__shfl_sync(0xffffffffu, s.hi, k), __shfl_sync(0xffffffffu, s.lo, k));
    };
    auto scale = [](ff a, float p) { return ff_make(a.hi * p, a.lo * p); };
    const ff A = get(0), Bh = get(1), Bm = get(2), Ch = get(3), Cm = get(4);
    Part P;
    P.A = scale(A, 0x1p-58f);
    P.B = ff_add(scale(Bh, 0x1p-58f), scale(Bm, 0x1p-86f));
    P.C = ff_add(scale(Ch, 0x1p-58f), scale(Cm, 0x1p-87f));
    return P;
}

// round(m 2^58) for a float-float m in (-2, 2); beyond the first sweeps the mean is a
// few units, and the 32-bit conversion is the fast one
__device__ __forceinline__ long long fix_mean(ff m) {
    const float h = m.hi * 0x1p58f;
    if (fabsf(h) < 0x1p30f) return __float2int_rn(h) + __float2int_rn((h - rintf(h)) + m.lo * 0x1p58f);
    return __float2ll_rn(m.hi * 0x1p58f) + __float2ll_rn(m.lo * 0x1p58f);
}

// Slot of a fixed-point sweep: mean to subtract, rescale, decisions.
struct FixSlot {
    long long M;
    int e, stop;
};

// The control step of sweep s >= 1 (ctrl_step's decisions, from the integer
// sums): fills the slot of sweep s + 2.  mx: max |q| of sweep s.
__device__ __forceinline__ void fix_ctrl(const PiArgs &a, int s, const Part &P, unsigned mx, Ctl &c, FixSlot *next,
                                         bool count_exit) {
    const float nf = (float)a.n;
    const ff mu = ff_mul(P.A, c.inv_n);
    const ff ss = ff_add_f(P.B, -nf * mu.hi * mu.hi);
    const ff cs = ff_add_f(P.C, -nf * mu.hi * c.mu_prev.hi);
    const bool zero = ss.hi <= a.zero_tol2 * (c.e_prev ? ldexpf(c.ss_prev.hi, 2 * c.e_prev) : c.ss_prev.hi);
    const bool conv = cs.hi > 0.f && !ff_lt(ff_mul(cs, cs), ff_mul(ff_mul(ss, c.ss_prev), c.omt2));
    bool stop = zero;
    if (a.mode == 0) stop = stop || conv || count_exit;
    else stop = stop || count_exit;
    if (stop && !c.stopped) ctl_stop(a, s, mu, ss, cs, zero, conv, c);
    const ff dm = ff_sub(mu, c.m_cur);
    const ff m_next = c.e_cur ? ff_make(ldexpf(dm.hi, c.e_cur), ldexpf(dm.lo, c.e_cur)) : dm;
    // |X_s| < 2^b, so |X_{s+1}| < 2^(b + e_s) (an average, less a mean of a few
    // units): lift it to 2^56, so that 248 rows' q^2 add up below 2^63
    const int b = 61 - __clz((int)mx) + c.e_cur;
    const int e_next = min(24, max(0, 56 - b));
    if (next) {
        next->M = fix_mean(m_next);
        next->e = e_next;
        next->stop = stop ? 1 : 0;
    }
    c.mu_prev = mu;
    c.ss_prev = ss;
    c.m_cur = m_next;
    c.e_prev = c.e_cur;
    c.e_cur = e_next;
}

// State of the register form's control warp, by lane where noted (the warp runs
// one chain per sweep whose length is instructions, fetched anew every sweep
// behind the row warps' code: the decisions are taken with a few FP64
// instructions on the totals, whose pipe the sweeps leave idle, where the
// float-float form of fix_ctrl takes 300 FP32 instructions).
struct FixCtl {
    double B, K, Z;    // lanes 4..7: ||y||^2 of the last sweep, times (1 - tol)^2,
                       // times the annihilation threshold of the next
    double C, Bp;      // lanes 16..19: the last y . y_prev; lanes 4..7: B before
    double muA;        // sum y of the last sweep (X units), every lane
    double mu_p;
    long long M;       // mean subtracted in the next sweep
    int e;             // rescale of the next sweep
};

// One control step for sweep s >= 1 (fix_ctrl's decisions): v is the sweep's
// total of the lane's value (fix_warp_vals' placement), mx its max |q|.
// Returns 0, 1 (converged) or 2 (annihilated); *next: M, e of sweep s + 2.
__device__ __forceinline__ int fix_decide(const PiArgs &a, int lane, long long v, unsigned mx, double omt2, float inv_n,
                                          FixCtl &c, FixSlot *next) {
    const int grp = lane >> 2;
    // value to double, in units of y y (2^116) or, for A, of X
    double d = __ll2double_rn(v);
    const int sh = grp == 0 ? 0 : (grp == 1 || grp == 4 ? -42 : (grp == 2 ? -86 : -87));
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
    // |X_s| < 2^b, so |X_{s+1}| < 2^(b + e_s): lift it to 2^56
    const int en = min(24, max(0, 56 - (61 - __clz((int)mx) + c.e)));
    c.K = omt2 * t;
    c.Z = t * (double)(c.e ? ldexpf(a.zero_tol2, 2 * c.e) : a.zero_tol2);
    next->M = Mn;
    next->e = en;
    c.M = Mn;
    c.e = en;
    return code;
}

// State and first slots from the start vector's totals (read: value by lane group
// as fix_decide wants it, A 2^-20 in the place of C's first value, and the maximum).
template <typename READ>
__device__ __forceinline__ void fix_ctl_start(const PiArgs &a, int lane, READ read, double omt2, int n, FixCtl &c,
                                              FixSlot *slots) {
    unsigned m;
    const long long v = read(&m);
    const int grp = lane >> 2;
    double d = __ll2double_rn(v);
    if (grp == 1) d *= 0x1p-42;
    if (grp == 2) d *= 0x1p-86;
    const double A = fma(__shfl_sync(0xffffffffu, d, 16), 0x1p20, __shfl_sync(0xffffffffu, d, 0));
    const double B = __shfl_sync(0xffffffffu, d, 4) + __shfl_sync(0xffffffffu, d, 8);
    const double mu0 = A * 0x1p-58 / (double)n;
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
        slots[1].M = __double2ll_rn(A / (double)n);   // sweep 1: exact mean of y_0
        slots[1].e = 0;
        slots[1].stop = 0;
        slots[0].M = 0;                               // sweep 2: m_1 = 0
        slots[0].e = 0;
        slots[0].stop = 0;
    }
}

// Result of a run whose last decided sweep is rs with `code` (fix_decide); buf:
// the ring slot of sweep rs.  res[0..1]: rs, annihilated.
__device__ __forceinline__ void fix_finish(const PiArgs &a, int lane, int n, int rs, int code, bool counted, bool bad,
                                           bool writes, int buf, const FixCtl &c, int *res) {
    const double to_mean = 0x1p-58 / (double)n;
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
    return fma((double)x.x, 0x1p29, (double)x.y) * 0x1p-58;
}

// The reciprocal fix_weight takes: false when g is not a positive finite number.
bool fix_reciprocal(double g, unsigned long long *ginv, int *ge);

// The exponent k that scales a start vector of largest magnitude m (finite,
// > 0) to |x| 2^k in (2^55, 2^56].
__device__ __forceinline__ int fix_start_exponent(double m) {
    int ex;
    frexp(m, &ex);   // m = f 2^ex, f in [0.5, 1)
    return 56 - ex;
}

}  // namespace cmg
