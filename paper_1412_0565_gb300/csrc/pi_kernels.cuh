// pi_kernels.cuh -- what the power-iteration kernels of the single-graph form
// share (refine.cu, resident.cu): the launch arguments, the stop sums of a
// sweep as CTAs exchange them, the start vector, and the control step that
// turns a sweep's sums into the stop decision and the next scalars (see the
// head of refine.cu for the method).
#pragma once

#include <math.h>

#include "ffloat.cuh"
#include "internal.h"
#include "pi_common.cuh"

namespace cmg {

// Loads of data written by other CTAs of the same launch go through L2.
#define LDX(p) __ldcg(p)
// Gathers of the iterate: ordinary (L1-cached) loads.  The iterate read in a
// sweep was written before the preceding grid barrier, whose acquire by the
// CTA's thread 0 (followed by __syncthreads) orders these loads after the
// writes; the parity tests check this bit for bit against L2-only loads.
#ifdef CMG_X_LDCG
#define LDXG(p) __ldcg(p)
#else
#define LDXG(p) (*(p))
#endif

// Stop sums of one CTA as stored for the other CTAs' control warps: two
// 16-byte words, so that a lane fetches a record with two loads.
struct __align__(16) PartRec {
    float4 ab;   // A.hi, A.lo, B.hi, B.lo
    float4 c;    // C.hi, C.lo
};
constexpr int kPartDoubles = (int)(sizeof(PartRec) / sizeof(double));

struct PiArgs {
    int n;
    const int *rp;
    const int *col;
    const double *w;
    const float *w32;
    double g;
    const int *tile_row;
    int ntiles;
    int mode;
    int k_fixed;
    int max_sweeps;
    double tol;
    uint64_t seed;
    int start;              // 0 Gaussian, 1 prolongation, 2 explicit
    const void *cbuf[3];    // coarse ring (start = 1)
    int cfp64;              // the coarse ring holds doubles (else floats)
    const PiResult *cres;
    const int *agg;
    const double *x_init;   // start = 2
    void *buf[3];           // iterate ring
    double *gd;             // FP64 form: g - d_i
    PiResult *res;
    PartRec *partials;      // [2][gridDim.x]: the CTAs' stop sums, by sweep parity
    float zero_tol2;        // (64 eps)^2 of the sweep precision
    const int *cinvp;       // coarse level's layout order (start = 1), or nullptr
    // slice kernel: the level's sweep layout (rows in layout order)
    const int *perm;
    int lay_h, lay_nsl;
    const int *lay_meta;
    const void *lay_col;
    const void *lay_w;
    const int *hchunk;      // heavy rows: first chunk per row ([h+1]), or nullptr
    const int *crow;        // heavy row of each chunk
    int *hcount;            // chunks finished per heavy row
    void *cpart;            // chunk partial sums
    int nchunks;
    int stage_n;            // iterate entries 0..stage_n-1 copied to shared memory per sweep
    // two-phase kernel: the level's XLayout (see internal.h)
    int x_T, x_Q, x_SB, x_VMAX;
    const uint16_t *x_src, *x_dst;
    const void *x_w;
    const int *x_ps, *x_sal, *x_qoff, *x_ndb, *x_dbr, *x_dbl, *x_cdel, *x_choff;
    const uint2 *x_chk;
    double *x_pmax;
    void *x_buf[2];
    // row kernel: items, first item of each CTA, capacities of its shared memory
    // (res_entries: also the resident slice kernel's)
    const int4 *items;
    const int *item_range;
    int res_entries, res_items, res_rows;
    int nitems;             // fixed-point sweeps: items of the level
    void *fix_acc;          // row kernel: the CTAs' stop sums (see k_power_rows)
    const int2 *fix_d;      // fixed-point sweeps: diagonal D_i by row in layout order
};


__device__ __forceinline__ void store_part(PartRec *dst, const Part &q) {
    dst->ab = make_float4(q.A.hi, q.A.lo, q.B.hi, q.B.lo);
    dst->c = make_float4(q.C.hi, q.C.lo, 0.f, 0.f);
}

// Sum of the gridDim.x records at src by one warp: lane l takes records l,
// l + 32, ... in order, then the lanes' tree.  Five records per lane are
// fetched before the first is added: what bounds the control warp on levels
// whose rows take less than it is the number of dependent trips to L2 (two
// here for 304 CTAs; ten with a fetch per addition, 3.7 us).
__device__ __forceinline__ Part grid_part(const PartRec *src, int lane) {
    Part q = part_zero();
    const int nb = (int)gridDim.x;
    for (int b0 = lane; b0 < nb; b0 += 32 * 5) {
        float4 ab[5], c[5];
#pragma unroll
        for (int u = 0; u < 5; u++) {
            ab[u] = c[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (b0 + 32 * u < nb) {
                ab[u] = __ldcg(&src[b0 + 32 * u].ab);
                c[u] = __ldcg(&src[b0 + 32 * u].c);
            }
        }
#pragma unroll
        for (int u = 0; u < 5; u++) {
            if (b0 + 32 * u >= nb) continue;
            Part t;
            t.A = ff_make(ab[u].x, ab[u].y);
            t.B = ff_make(ab[u].z, ab[u].w);
            t.C = ff_make(c[u].x, c[u].y);
            q = part_add(q, t);
        }
    }
    return warp_sum_part(q);
}

// Start value of row i: Gaussian (Alg. 1 Step 2), prolongation (I^T y of
// Alg. 1 Step 3) of the coarse result, or an explicit vector.
// The coarse ring has the coarse level's own sweep precision (a level held in
// one CTA keeps FP64 sweeps in the FP32 form).
__device__ __forceinline__ double start_value(const PiArgs &a, int i, const void *cb, double cmu,
                                              double cinv) {
    if (a.start == 0) return gaussian_entry(a.seed, i);
    if (a.start == 1) {
        const int c = a.agg[i];
        const int k = a.cinvp ? a.cinvp[c] : c;
        const double v = a.cfp64 ? reinterpret_cast<const double *>(cb)[k]
                                 : (double)reinterpret_cast<const float *>(cb)[k];
        return (v - cmu) * cinv;
    }
    return a.x_init[i];
}


// ------------------------------------------------------------------ control
// Sweep parameters and decisions, double-buffered by sweep parity in shared
// memory.  Slot for sweep t holds what the rows of sweep t need (m_{t-1},
// e_{t-1}) and the stop decision taken for sweep t-2.
struct Slot {
    // FP64 rows: the same scalars as doubles, formed once per sweep by the
    // control warp (an FP64 operation issues at 2 per SM per clock: per-row-
    // thread copies of this arithmetic cost every row warp FP64 issue slots)
    double m_d;     // m as a double
    double sig_d;   // 2^e / g
    double gm_d;    // g m
    ff m;           // mean estimate to subtract
    int e;          // power-of-two rescale exponent
    int stop;       // decision for sweep t-2: 0 continue, 1 stop
    int zero;       // that sweep annihilated the iterate
    int pad;
};

// fp64: also form the doubles (the FP32 kernels leave them unused); inv_g is
// 1 / g, divided once per launch (an FP64 division is a chain of about ten
// dependent FP64 instructions, and the scaling exponent is 0 in nearly every
// sweep)
__device__ __forceinline__ Slot slot_make(ff m, int e, double g, double inv_g, bool fp64) {
    Slot sl;
    sl.m = m;
    sl.e = e;
    sl.stop = 0;
    sl.zero = 0;
    sl.pad = 0;
    sl.m_d = sl.sig_d = sl.gm_d = 0.0;
    if (fp64) {
        sl.m_d = ff_to_double(m);
        sl.sig_d = e ? ldexp(inv_g, e) : inv_g;
        sl.gm_d = g * sl.m_d;
    }
    return sl;
}

// Scalars of the reduced sweeps, kept by the control warp (all lanes hold
// the same values).
struct Ctl {
    ff mu_prev, ss_prev;   // mean and squared norm of y_{s-1}
    ff m_cur;              // m_s: used by sweep s+1
    ff inv_n, omt2;        // 1/n and (1 - tol)^2
    int e_cur, e_prev;     // e_s, e_{s-1}
    double inv_g;          // 1/g
    // result of the decision (valid once `stopped`)
    int stopped, zero, res_sweep, capped;
    double mu_res, ss_res, mu_res_prev, ss_res_prev, cos_res;
};


// Records the decision to stop after sweep s.
__device__ __forceinline__ void ctl_stop(const PiArgs &a, int s, ff mu, ff ss, ff cs, bool zero, bool conv, Ctl &c) {
    c.stopped = 1;
    c.zero = zero;
    c.res_sweep = s;
    if (zero) {
        c.mu_res = to_d(c.mu_prev);
        c.ss_res = to_d(c.ss_prev);
        c.cos_res = 1.0;
    } else {
        c.mu_res = to_d(mu);
        c.ss_res = to_d(ss);
        c.mu_res_prev = to_d(c.mu_prev);
        c.ss_res_prev = to_d(c.ss_prev);
        const double den = sqrt(c.ss_res * c.ss_res_prev);
        c.cos_res = den > 0.0 ? to_d(cs) / den : 1.0;
    }
    c.capped = (a.mode == 0 && !zero && !conv) ? 1 : 0;
}

// One control step for sweep s (s >= 1) with its reduced sums P.  Decides,
// and fills the slot for sweep s+2 (m_{s+1}, e_{s+1}).  `count_exit`: the
// loop ends after sweep s regardless (fixed count or sweep cap reached).
__device__ __forceinline__ void ctrl_step(const PiArgs &a, int s, const Part &P, Ctl &c,
                                          Slot *next, bool count_exit, bool fp64) {
    const float nf = (float)a.n;
    // the mean is at rounding level: n mu^2 and n mu mu_prev need no extra
    // precision, mu itself does (it is subtracted from the iterate)
    const ff mu = ff_mul(P.A, c.inv_n);
    const ff ss = ff_add_f(P.B, -nf * mu.hi * mu.hi);
    const ff cs = ff_add_f(P.C, -nf * mu.hi * c.mu_prev.hi);
    // annihilated: ||proj y_s|| <= 64 eps 2^{e_{s-1}} ||proj y_{s-1}||
    const bool zero = ss.hi <= a.zero_tol2 * (c.e_prev ? ldexpf(c.ss_prev.hi, 2 * c.e_prev) : c.ss_prev.hi);
    // cos_s >= 1 - tol  <=>  cs > 0 and cs^2 >= (1 - tol)^2 ss_s ss_{s-1}
    const bool conv = cs.hi > 0.f && !ff_lt(ff_mul(cs, cs), ff_mul(ff_mul(ss, c.ss_prev), c.omt2));
    bool stop = zero;
    if (a.mode == 0) stop = stop || conv || count_exit;
    else stop = stop || count_exit;
    if (stop && !c.stopped) ctl_stop(a, s, mu, ss, cs, zero, conv, c);
    // parameters of sweep s+2 (exact power-of-two scaling of mu_s - m_s)
    const ff dm = ff_sub(mu, c.m_cur);
    const ff m_next = c.e_cur ? ff_make(ldexpf(dm.hi, c.e_cur), ldexpf(dm.lo, c.e_cur)) : dm;
    int e_next = 0;
    // (1e-14 is above 2^-48: without a pending rescale no new one is due)
    if (c.e_cur != 0 || ss.hi <= 1e-14f) {
        // predicted log2 ||y_{s+1}|| <= log2 ||y_s|| + e_s; lift it back to ~1
        const float l2 = 0.5f * log2f(fmaxf(ss.hi, 1e-37f)) + (float)c.e_cur;
        if (l2 < -24.f) e_next = (int)(-l2);
    }
    if (next) {
        *next = slot_make(m_next, e_next, a.g, c.inv_g, fp64);
        next->stop = stop ? 1 : 0;
        next->zero = zero ? 1 : 0;
    }
    c.mu_prev = mu;
    c.ss_prev = ss;
    c.m_cur = m_next;
    c.e_prev = c.e_cur;
    c.e_cur = e_next;
}

__device__ __forceinline__ void ctl_init(Ctl &c, const PiArgs &a, double mu0, double ss0, int e0) {
    c.mu_prev = ff_from_double(mu0);
    c.ss_prev = ff_from_double(ss0);
    c.m_cur = ff_zero();   // m_1: the start was projected exactly
    c.inv_n = ff_from_double(1.0 / (double)a.n);
    c.inv_g = 1.0 / a.g;
    const double omt = 1.0 - a.tol;
    c.omt2 = ff_from_double(omt * omt);
    c.e_cur = 0;
    c.e_prev = e0;
    c.stopped = 0;
    c.zero = 0;
    c.res_sweep = 0;
    c.capped = 0;
    c.mu_res = mu0;
    c.ss_res = ss0;
    c.mu_res_prev = mu0;
    c.ss_res_prev = ss0;
    c.cos_res = 0.0;
}


__device__ __forceinline__ void write_result(const PiArgs &a, const Ctl &c, int buf, int buf_prev) {
    PiResult r;
    r.mu = c.mu_res;
    r.inv_s = c.ss_res > 0.0 ? 1.0 / sqrt(c.ss_res) : 0.0;
    r.cos = c.cos_res;
    r.mu_prev = c.mu_res_prev;
    r.inv_s_prev = c.ss_res_prev > 0.0 ? 1.0 / sqrt(c.ss_res_prev) : 0.0;
    r.buf = buf;
    r.buf_prev = buf_prev;
    r.sweeps = c.res_sweep;
    r.capped = c.capped;
    r.zero = c.zero;
    r.pad = 0;
    *a.res = r;
}

template <typename T>
__device__ __forceinline__ const T *wsel(const PiArgs &a);
template <>
__device__ __forceinline__ const double *wsel<double>(const PiArgs &a) { return a.w; }
template <>
__device__ __forceinline__ const float *wsel<float>(const PiArgs &a) { return a.w32; }


template <typename P>
__device__ __forceinline__ P pick3(P p0, P p1, P p2, int k) {
    return k == 0 ? p0 : (k == 1 ? p1 : p2);
}

__device__ __forceinline__ void bar_rows(int nthreads) {
    asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

}  // namespace cmg
