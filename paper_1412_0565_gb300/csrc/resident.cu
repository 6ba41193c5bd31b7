// resident.cu -- the row kernel: FP64 power-iteration sweeps of a level spread over
// all SMs, in fixed point (fixed.cuh), with the level's matrix held in the SMs'
// shared memory for the whole launch where it fits (see k_power_rows); and the
// plans that deal rows to warps and CTAs, k_power_fix's included.
#include <algorithm>

#include "fixed.cuh"

namespace cmg {

// ------------------------------------------------------------------ plan
// Lanes per row by row length: steps of at most S entries per lane while the row
// fits a warp, S = 8 on levels with at most kWideEntries entries per SM (a sweep
// there is a chain of latencies: a row of 16 entries on one lane is two rounds of
// gathers, on two lanes one) and 16 above, where the instructions are the bound and
// every split row costs extra sums.  us per sweep, S = 8 and 16: 15K rows and 93K
// entries 4.1 and 4.3, 10K and 153K 3.5 and 3.65; 114K and 1.5M 11.2 and 9.5.
constexpr int kWideEntries = 8192;
// Cost of an item beside its entries, in entries: the rows' finish and stop sums.
// (64: 4.4 us per sweep against 3.4 on 5,047 rows and 23K entries, the CTAs too few;
// 1,024: 10.7 against 9.5 on 114K rows and 1.5M entries.)
constexpr int kItemCost = 256;
// Work of one CTA at least, in entries (an item counts kItemCost): below it more
// CTAs make the barrier dearer and the rows no faster, and leave no SM to the
// other streams of a server.  (1,024: the same times; 4,096: 4.4 us per sweep against
// 3.4 on 5,047 rows and 23K entries; 8,192: 6.4 against 3.7 on 20K rows and 160K.)
constexpr int kCtaWork = 2048;
constexpr int kPlanThreads = 1024;
constexpr int kStreamThreads = 384;   // two CTAs per SM with 85 registers a thread
constexpr int kRowsMaxRow = 4096;  // longest row the items take (one warp each)

__device__ __forceinline__ int plan_deg(const int *rp, const uint32_t *perm, int p) {
    const int v = (int)perm[p];
    return rp[v + 1] - rp[v];
}

__device__ __forceinline__ int plan_scan(int v, int *sm, int *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sm[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int t = sm[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        sm[lane] = t;
    }
    __syncthreads();
    const int before = warp > 0 ? sm[warp - 1] : 0;
    *total = sm[31];
    __syncthreads();
    return before + x - v;
}

// P is cut to one CTA per kCtaWork; CTA p takes the items from the first whose entries before it, at kItemCost
// more per item, reach p / P of the total.
// (cut: false takes P as it is)
__device__ __forceinline__ void plan_ranges(int P, bool cut, int ni, const int4 *item, int *range, PlanOut *out) {
    const int tid = threadIdx.x;
    __shared__ int s_max[3];
    if (tid < 3) s_max[tid] = 0;
    const long long total = (long long)item[ni].y + (long long)kItemCost * ni;
    if (cut) P = (int)min((long long)P, total / kCtaWork + 1);
    for (int p = tid; p <= P; p += blockDim.x) {
        const long long target = total * p / P;
        int lo = 0, hi = ni;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((long long)item[mid].y + (long long)kItemCost * mid < target) lo = mid + 1;
            else hi = mid;
        }
        range[p] = p == P ? ni : lo;
    }
    __syncthreads();
    for (int p = tid; p < P; p += blockDim.x) {
        const int a = range[p], b = range[p + 1];
        atomicMax(&s_max[0], item[b].y - item[a].y);
        atomicMax(&s_max[1], b - a);
        atomicMax(&s_max[2], item[b].x - item[a].x);
    }
    __syncthreads();
    if (tid == 0) {
        out->P = P;
        out->ni = ni;
        out->max_e = s_max[0];
        out->max_i = s_max[1];
        out->max_r = s_max[2];
        out->entries = item[ni].y;
    }
}

// Items of n rows in degree order, one CTA: rows longer than 16 S entries take 32
// lanes each, rows longer than 8 S 16 lanes, ... rows of at most S one lane; an
// item is 32 lanes (32 / G rows) and as many steps as its first (longest) row
// needs.  deg(p): length of the row at position p.  At most cap items are
// written; returns their number.
// quad: steps are rounded up to a multiple of 4 (the kernels that sweep from shared
// memory take four entries at a time without a test per entry; a streamed level
// would read the padding from L2).
template <typename DEG>
__device__ __forceinline__ int plan_units(int n, int S, bool quad, DEG deg, int cap, int4 *item) {
    __shared__ int s_row[7], s_unit[7], s_sm[32];
    const int tid = threadIdx.x;
    if (tid < 7) {
        // first position whose row is no longer than 16 S, 8 S, 4 S, 2 S, S, -1
        const int thr = tid == 0 ? 0x7fffffff : (tid == 6 ? -1 : (S << (5 - tid)));
        int lo = 0, hi = n;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (deg(mid) > thr) lo = mid + 1;
            else hi = mid;
        }
        s_row[tid] = lo;
    }
    __syncthreads();
    if (tid == 0) {
        s_unit[0] = 0;
        for (int c = 0; c < 6; c++) {
            const int per = 1 << c;   // rows per item: 32 lanes / 2^(5-c)
            s_unit[c + 1] = s_unit[c] + (s_row[c + 1] - s_row[c] + per - 1) / per;
        }
    }
    __syncthreads();
    const int nu = s_unit[6];
    constexpr int K = 8;
    long long run = 0;
    for (int u0 = 0; u0 < nu; u0 += kPlanThreads * K) {
        int st[K], r0[K], lw[K], sum = 0;
#pragma unroll
        for (int k = 0; k < K; k++) {
            const int u = u0 + tid * K + k;
            st[k] = r0[k] = lw[k] = 0;
            if (u < nu) {
                int c = 0;
                while (u >= s_unit[c + 1]) c++;
                r0[k] = s_row[c] + ((u - s_unit[c]) << c);
                const int rows = min(1 << c, s_row[c + 1] - r0[k]);
                lw[k] = (5 - c) | (rows << 3);
                st[k] = (deg(r0[k]) + (32 >> c) - 1) >> (5 - c);
                if (quad) st[k] = (st[k] + 3) & ~3;
            }
            sum += st[k];
        }
        int tot;
        long long off = run + plan_scan(sum, s_sm, &tot);
#pragma unroll
        for (int k = 0; k < K; k++) {
            const int u = u0 + tid * K + k;
            if (u < nu && u < cap) item[u] = make_int4(r0[k], (int)(32 * off), st[k], lw[k]);
            off += st[k];
        }
        run += tot;
    }
    // beyond 32-bit offsets: the caller sees the entry count
    if (tid == 0) item[min(nu, cap)] = make_int4(n, run > 0x3ffffff ? 0x7fffffff : (int)(32 * run), 0, 0);
    __syncthreads();
    return nu;
}

__global__ void __launch_bounds__(kPlanThreads) k_plan_units(int n, const int *__restrict__ rp,
                                                             const uint32_t *__restrict__ perm, int S, int quad, int P, int cap,
                                                             int4 *__restrict__ item, int *__restrict__ range,
                                                             PlanOut *__restrict__ out) {
    const int nu = plan_units(n, S, quad != 0, [&](int p) { return plan_deg(rp, perm, p); }, cap, item);
    if (threadIdx.x == 0) out->maxdeg = plan_deg(rp, perm, 0);
    plan_ranges(P, true, min(nu, cap), item, range, out);
}

// Entries and diagonal of one item in fixed point (one warp); short rows and
// missing rows are padded with coefficient 0 and a valid column.
template <typename PERM, typename INV, typename IDX>
__device__ __forceinline__ void fill_item(int4 it, int lane, const int *rp, const int *col, const double *w,
                                          unsigned long long ginv, int ge, const PERM *perm, const INV *inv, IDX *ucol,
                                          int2 *uc, int2 *ud) {
    const int lg = it.w & 7, rows = it.w >> 3, r = lane >> lg, g = lane & ((1 << lg) - 1);
    const int p = it.x + (r < rows ? r : 0);
    int e0 = 0, deg = 0;
    if (r < rows) {
        const int v = (int)perm[p];
        e0 = rp[v];
        deg = rp[v + 1] - e0;
    }
    long long sum = 0;
    for (int t = 0; t < it.z; t++) {
        const int k = (t << lg) + g;
        const size_t d = (size_t)it.y + 32 * t + lane;
        long long Cij = 0;
        int cl = p;
        if (k < deg) {
            Cij = fix_weight(w[e0 + k], ginv, ge);
            cl = (int)inv[col[e0 + k]];
        }
        ucol[d] = (IDX)cl;
        uc[d] = fix_split_c(Cij);
        sum += Cij;
    }
    for (int o = (1 << lg) >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (r < rows && g == 0) ud[p] = fix_split_c(sum);
}

// The plan of levels of at most kFixMaxN rows, one CTA per level and one launch for
// all of them: degree order (a stable counting sort), items and ranges.  (The one-CTA and
// cluster kernels sorted and laid out their level in the sweep launch itself,
// and the cluster's plan read its row pointers back to the host.)
__global__ void __launch_bounds__(kPlanThreads) k_plan_small(const __grid_constant__ SmallJobs jobs) {
    __shared__ SmallJob J;
    __shared__ unsigned short s_perm[kFixMaxN], s_inv[kFixMaxN];
    __shared__ int s_hist[kFixMaxN + 1];
    __shared__ int s_md;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        J = jobs.j[blockIdx.x];
        s_md = 0;
    }
    __syncthreads();
    const int n = J.n;
    // the sort's bucket (degrees of valid rows are below n)
    auto len = [&](int i) { return J.rp[i + 1] - J.rp[i]; };
    for (int i = tid; i < n; i += kPlanThreads) atomicMax(&s_md, min(len(i), kFixMaxN - 1));
    __syncthreads();
    const int D = s_md;
    for (int b = tid; b <= D; b += kPlanThreads) s_hist[b] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += kPlanThreads) {
        const int b = D - min(len(i), kFixMaxN - 1);
        s_inv[i] = (unsigned short)b;
        atomicAdd(&s_hist[b], 1);
    }
    __syncthreads();
    if (warp == 0) {
        int carry = 0;
        for (int b0 = 0; b0 <= D; b0 += 32) {
            const int b = b0 + lane;
            const int c = b <= D ? s_hist[b] : 0;
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            if (b <= D) s_hist[b] = carry + incl - c;
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
        __syncwarp();
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            const unsigned act = __ballot_sync(0xffffffffu, i < n);
            if (i < n) {
                const int b = s_inv[i];
                const unsigned peers = __match_any_sync(act, b);
                const int r = __popc(peers & ((1u << lane) - 1u));
                const int base = s_hist[b];
                s_perm[base + r] = (unsigned short)i;
                __syncwarp(act);
                if (r == 0) s_hist[b] = base + __popc(peers);
            }
            __syncwarp();
        }
    }
    __syncthreads();
    for (int p = tid; p < n; p += kPlanThreads) {
        J.inv[s_perm[p]] = (uint16_t)p;
        J.perm[p] = s_perm[p];
    }
    __syncthreads();
    // one item per row warp: of at most 8 steps where one CTA holds them all, else
    // of 16; beyond the warps, items of up to J.S steps dealt by their entries
    auto deg = [&](int p) { return len(s_perm[p]); };
    int nu = plan_units(n, 8, false, deg, J.cap_items, J.item);
    int steps = D <= 256 && nu <= J.one_cta ? 8 : 0;
    if (!steps) {
        nu = plan_units(n, 16, false, deg, J.cap_items, J.item);
        if (D <= 512 && nu <= J.cap_warps) steps = 16;
        else nu = plan_units(n, J.S, true, deg, J.cap_items, J.item);
    }
    plan_ranges(J.C, false, min(nu, J.cap_items), J.item, J.range, J.out);
    const bool fits = nu <= J.cap_items;
    if (tid == 0) {
        J.out->by_warp = steps;
        J.out->maxdeg = fits ? 0 : -1;   // -1: more items than the capacity
        if (!fits) J.out->ni = 0;
    }
}

// Entries and diagonal of the planned levels, a warp per item (blockIdx.y: level).
__global__ void k_fill_small(const __grid_constant__ SmallJobs jobs) {
    const SmallJob &J = jobs.j[blockIdx.y];
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < J.ni; u += warps)
        fill_item(J.item[u], lane, J.rp, J.col, J.w, J.ginv, J.ge, J.perm, J.inv, J.ucol, J.uc, J.ud);
}

template <typename IDX>
__global__ void k_fill_units(int ni, const int4 *__restrict__ item, const int *__restrict__ rp,
                             const int *__restrict__ col, const double *__restrict__ w, unsigned long long ginv, int ge,
                             const uint32_t *__restrict__ perm, const int *__restrict__ inv, IDX *__restrict__ ucol,
                             int2 *__restrict__ uc, int2 *__restrict__ ud) {
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < ni; u += warps)
        fill_item(item[u], lane, rp, col, w, ginv, ge, perm, inv, ucol, uc, ud);
}

// ------------------------------------------------------------------ kernel
constexpr int kFixRec = 8;   // 64-bit words of one sweep's sums: 5 values, max |q|, 2 spare

// Words of the sums in device memory: three sweeps' records, then the start
// vector's largest magnitude.
constexpr int kFixAccWords = 3 * kFixRec + 8;

// Sweeps of a level of up to kFixRowsMax rows over all SMs (cooperative, warp 0 the control warp, one grid
// barrier per sweep, iterates in degree order, deferred decisions as in
// k_power_sell).  A row warp takes items: 32 lanes on 32 / G rows, entry t of
// lane l at offset 32 t + l.  The CTAs add their integer stop sums to one record
// in L2 (any order gives the same sums), which every control warp then reads
// with one load.
//
// RES: one CTA per SM copies its items' columns, coefficients and diagonal into
// shared memory once and sweeps from there.  On levels of a few million
// entries at most, what bounds a sweep is the chain of dependent trips to L2
// (columns and coefficients, then the iterate, per group of 8 entries) plus the
// barrier: from shared memory only the gathers remain, and with STAGE (the
// whole iterate copied to shared memory at the top of a sweep) one trip.
// Otherwise two CTAs per SM stream the items, each with its columns,
// coefficients and own row in flight together, the next item's descriptor too.
// us per sweep: slice kernel in FP64, this kernel in FP64, in fixed point: 1,542 rows
// and 103K entries 17.3, 6.3, 4.0; 5,688 rows and 129K entries 16.0, 6.6, 4.4; 20K
// rows and 160K entries 16.0, 5.0, 3.6; the 100^3 grid's levels of 1M, 348K, 114K, 35K
// and 10K rows 40.4 / 23.6 / 14.7 / 9.4 / 8.3, 38.0 / 22.5 / 11.3 / 6.9 / 4.8, and
// 24.8 / 19.9 / 9.5 / 5.1 / 3.5.
template <typename IDX, bool RES, bool STAGE, bool STREAM>
__global__ void __launch_bounds__(RES ? 1024 : kStreamThreads, RES ? 1 : 2) k_power_rows(PiArgs a, GridSync *gs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(16) long long s_pw[32][kFixSums];   // the warps' sums
    __shared__ FixSlot s_slot[2];
    __shared__ GridBar s_bar;
    __shared__ int s_res[2];       // sweeps of the result, annihilated
    const int n = a.n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nw = (int)(blockDim.x >> 5);
    if (tid == 0) grid_bar_init(&s_bar, gs);
    int2 *const ring0 = (int2 *)a.buf[0], *const ring1 = (int2 *)a.buf[1], *const ring2 = (int2 *)a.buf[2];
    const int ib = a.item_range[blockIdx.x], ie = a.item_range[blockIdx.x + 1];
    const int4 first = a.items[ib], last = a.items[ie];
    const int r0 = first.x, r1 = last.x, e_lo = first.y;
    // shared memory (RES): items, coefficients, diagonal, the staged iterate, columns
    int4 *s_item = reinterpret_cast<int4 *>(smem_raw);
    int2 *s_w = reinterpret_cast<int2 *>(s_item + a.res_items);
    int2 *s_x = s_w + a.res_entries;
    int2 *s_d = s_x + (STAGE ? ((n + 1) & ~1) : 0);
    IDX *s_c = reinterpret_cast<IDX *>(s_d + ((a.res_rows + 1) & ~1));
    if (RES) {
        const int2 *gw = reinterpret_cast<const int2 *>(a.lay_w) + e_lo;
        const IDX *gc = reinterpret_cast<const IDX *>(a.lay_col) + e_lo;
        const int ne = last.y - e_lo;   // a multiple of 32: 16-byte copies
        for (int k = tid; k < ne / 2; k += blockDim.x)
            reinterpret_cast<uint4 *>(s_w)[k] = __ldg(reinterpret_cast<const uint4 *>(gw) + k);
        for (int k = tid; k < ne * (int)sizeof(IDX) / 16; k += blockDim.x)
            reinterpret_cast<uint4 *>(s_c)[k] = __ldg(reinterpret_cast<const uint4 *>(gc) + k);
        for (int k = tid; k < r1 - r0; k += blockDim.x) s_d[k] = __ldg(a.fix_d + r0 + k);
        for (int k = tid; k < ie - ib; k += blockDim.x) {
            int4 it = a.items[ib + k];
            it.y -= e_lo;
            s_item[k] = it;
        }
    }
    const IDX *C = RES ? s_c : reinterpret_cast<const IDX *>(a.lay_col);
    const int2 *W = RES ? s_w : reinterpret_cast<const int2 *>(a.lay_w);
    unsigned long long *const acc = reinterpret_cast<unsigned long long *>(a.fix_acc);
    // the records of the warps from `first_warp` on, added to record k
    auto publish = [&](int first_warp, int k) {
        unsigned m;
        const long long v = fix_sum_records(s_pw[first_warp], nw - first_warp, lane, &m);
        const int grp = lane >> 2;
        if ((lane & 3) == 0 && grp != 3 && grp != 7) {
            unsigned long long *dst = acc + kFixRec * k + (grp < 3 ? grp : grp - 1);
            if (grp == 6) atomicMax(dst, (unsigned long long)m);
            else atomicAdd(dst, (unsigned long long)v);
        }
        __syncwarp();
    };
    // record k as fix_decide wants it: value by lane group, and max |q|
    auto read_acc = [&](int k, unsigned *m) -> long long {
        const int grp = lane >> 2;
        long long v = 0;
        if (grp != 3 && grp != 7) v = (long long)__ldcg(acc + kFixRec * k + (grp < 3 ? grp : grp - 1));
        *m = (unsigned)__shfl_sync(0xffffffffu, (int)v, 24);
        return grp == 6 ? 0 : v;
    };

    // ---- start vector: values as doubles in ring slot 0 and their largest
    // magnitude over the grid, then fixed point
    {
        const void *cb = nullptr;
        double cmu = 0.0, cinv = 0.0;
        if (a.start == 1) {
            cb = a.cbuf[a.cres->buf];
            cmu = a.cres->mu;
            cinv = a.cres->inv_s;
        }
        unsigned long long mb = 0;
        for (int p = r0 + tid; p < r1; p += blockDim.x) {
            const double v = start_value(a, a.perm[p], cb, cmu, cinv);
            reinterpret_cast<double *>(ring0)[p] = v;
            // magnitudes order as their bits; infinities and NaN are the largest
            mb = max(mb, (unsigned long long)__double_as_longlong(fabs(v)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
        if (lane == 0) atomicMax(acc + 3 * kFixRec, mb);
    }
    if (!grid_sync(&s_bar)) return;
    bool bad;
    {
        const double mx = __longlong_as_double((long long)__ldcg(acc + 3 * kFixRec));
        bad = !isfinite(mx);
        const int k = !bad && mx > 0.0 ? fix_start_exponent(mx) : 0;
        FixSum f;
        f.reset();
        for (int p = r0 + tid; p < r1; p += blockDim.x) {
            const double v = reinterpret_cast<double *>(ring0)[p];
            const long long X = bad ? 0 : __double2ll_rn(ldexp(v, k));
            const int2 x = fix_split(X);
            f.add_start(X, x);
            ring0[p] = x;
        }
        fix_warp_record(f, true, lane, s_pw[warp]);
        __syncthreads();
        if (warp == 0) publish(0, 0);
    }
    if (!grid_sync(&s_bar)) return;
    const int limit = bad ? 0 : (a.mode == 1 ? max(a.k_fixed, 0) : a.max_sweeps);
    if (warp == 0) {
        // ------------------------------------------------------ control warp
        const double omt = 1.0 - a.tol, omt2 = omt * omt;
        const float inv_n = 1.0f / (float)n;
        FixCtl c;
        unsigned m0;
        const long long v0 = read_acc(0, &m0);
        fix_ctl_start(a, lane, v0, omt2, n, c, s_slot);
        __syncthreads();
        int s = 0, rs = 0, code = 0, k0 = 0;   // k0 = s modulo 3
        bool counted = false;
        FixSlot nx;
        for (;; s++) {
            if (s_slot[(s + 1) & 1].stop) break;
            if (s >= limit) {
                counted = true;
                break;
            }
            const int k1 = k0 == 2 ? 0 : k0 + 1, k2 = k1 == 2 ? 0 : k1 + 1;
            if (s >= 1) {
                unsigned m;
                const long long v = read_acc(k0, &m);
                // the record of sweep s + 2 was last read before this sweep's barrier
                if (blockIdx.x == 0 && lane < kFixRec) acc[kFixRec * k2 + lane] = 0;
                code = fix_decide(a, lane, v, m, omt2, inv_n, c, &nx);
                rs = s;
                nx.stop = code == 2 || (code == 1 && a.mode == 0);
                if (lane == 0) s_slot[s & 1] = nx;
                __syncwarp();
            }
            __syncthreads();
            publish(1, k1);
            if (lane == 0) {
                // the CTA's rows and sums precede thread 0's release
                s_bar.ok = grid_arrive_wait(&s_bar);
            }
            __syncthreads();
            if (!s_bar.ok) return;
            k0 = k1;
        }
        if (counted && limit > 0) {
            unsigned m;
            const long long v = read_acc(k0, &m);
            code = fix_decide(a, lane, v, m, omt2, inv_n, c, &nx);
            rs = s;
        }
        fix_finish(a, lane, n, rs, code, counted, bad, blockIdx.x == 0, rs % 3, c, s_res);
    } else {
        // ------------------------------------------------------ row warps
        __syncthreads();
        int s = 0;
        int2 *x = ring0, *y = ring1, *z = ring2;
        for (;; s++) {
            const FixSlot sl = s_slot[(s + 1) & 1];
            if (sl.stop || s >= limit) break;
            if (STAGE) {
                // the whole iterate, in 16-byte pieces, then the row warps meet
                // (the control warp does not take part)
                const int nrt = (int)blockDim.x - 32;
                for (int k = tid - 32; k < n / 2; k += 4 * nrt) {
                    int4 v[4];
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (k + u * nrt < n / 2) v[u] = __ldcg(reinterpret_cast<const int4 *>(x) + k + u * nrt);
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (k + u * nrt < n / 2) reinterpret_cast<int4 *>(s_x)[k + u * nrt] = v[u];
                }
                if ((n & 1) && tid == 32) s_x[n - 1] = __ldcg(x + n - 1);
                bar_rows(nrt);
            }
            auto ldx = [&](int k) { return STAGE ? s_x[k] : LDXG(x + k); };
            FixSum f;
            f.reset();
            int4 nxt = !RES ? __ldg(a.items + min(ib + warp - 1, ie)) : make_int4(0, 0, 0, 0);
            for (int k = ib + warp - 1; k < ie; k += nw - 1) {
                const int4 it = RES ? s_item[k - ib] : nxt;
                if (!RES) nxt = __ldg(a.items + min(k + nw - 1, ie));
                const int lg = it.w & 7, rows = it.w >> 3, r = lane >> lg;
                const int i = it.x + (r < rows ? r : 0);
                const bool leads = r < rows && (lane & ((1 << lg) - 1)) == 0;
                const int2 xi = ldx(i);
                const int2 d = RES ? s_d[i - r0] : __ldg(a.fix_d + i);
                const int base = it.y + lane;
                FixAcc t;
                t.reset();
                if (RES) {
                    fix_quads(t, it.z, s_c + base, s_w + base, ldx);
                } else {
                    for (int t0 = 0; t0 < it.z; t0 += 8) {
                        int cc[8];
                        int2 ww[8], xx[8];
#pragma unroll
                        for (int u = 0; u < 8; u++) {
                            cc[u] = i;
                            ww[u] = make_int2(0, 0);
                            if (t0 + u < it.z) {
                                const int e = base + 32 * (t0 + u);
                                cc[u] = (int)(STREAM ? __ldcs(C + e) : C[e]);
                                ww[u] = STREAM ? __ldcs(W + e) : W[e];
                            }
                        }
#pragma unroll
                        for (int u = 0; u < 8; u++) xx[u] = ldx(cc[u]);
#pragma unroll
                        for (int u = 0; u < 8; u++) t.add(xx[u], ww[u]);
                        t.carry();
                    }
                }
                if (leads) {
                    t.add(xi, make_int2(-d.x, -d.y));
                    t.carry();
                }
                const long long pr = t.lanes(lg);
                if (leads) {
                    const long long X = fix_join(xi), Y = fix_row(X, pr, sl.M, sl.e);
                    const int2 yv = fix_split(Y);
                    y[i] = yv;
                    f.add(Y, yv, FixSum::narrow(Y), FixSum::narrow(X));
                }
            }
            __syncwarp();
            fix_warp_record(f, false, lane, s_pw[warp]);
            __syncthreads();   // the warps' sums are complete
            __syncthreads();   // the grid barrier has passed
            if (!s_bar.ok) return;
            int2 *t = x;
            x = y;
            y = z;
            z = t;
        }
    }
    __syncthreads();
    // the result as doubles, in place: no CTA reads the iterates any more
    const int rs = bad ? 0 : s_res[0], rb = s_res[1] ? (rs + 2) % 3 : rs % 3;
    int2 *res = pick3<int2 *>(ring0, ring1, ring2, rb);
    for (int p = r0 + tid; p < r1; p += blockDim.x) {
        const double v = fix_value(res[p]);
        reinterpret_cast<double *>(res)[p] = v;
    }
}

// (a staged iterate fits only where columns have 16 bits)
static const void *rows_kernel(const RowPlan &R) {
    if (R.resident) {
        if (R.stage) return (const void *)k_power_rows<uint16_t, true, true, false>;
        return R.col16 ? (const void *)k_power_rows<uint16_t, true, false, false>
                       : (const void *)k_power_rows<int, true, false, false>;
    }
    if (R.stream)
        return R.col16 ? (const void *)k_power_rows<uint16_t, false, false, true>
                       : (const void *)k_power_rows<int, false, false, true>;
    return R.col16 ? (const void *)k_power_rows<uint16_t, false, false, false>
                   : (const void *)k_power_rows<int, false, false, false>;
}

cmg_status_t launch_fill_small(const SmallJobs &jobs, int count, cudaStream_t s) {
    k_fill_small<<<dim3(64, count), 256, 0, s>>>(jobs);
    return launch_status();
}

cmg_status_t launch_plan_small(const SmallJobs &jobs, int count, cudaStream_t s) {
    k_plan_small<<<count, kPlanThreads, 0, s>>>(jobs);
    return launch_status();
}

static size_t rows_smem(int n, int col16, int stage, const PlanOut &o) {
    return 16 * (size_t)o.max_i + (col16 ? 10 : 12) * (size_t)o.max_e + (stage ? 8 * (size_t)((n + 1) & ~1) : 0) +
           8 * (size_t)((o.max_r + 1) & ~1) + 16;
}

// Shared memory the resident kernel may take.
static cmg_status_t rows_room(const RowPlan &R, size_t *room) {
    DeviceInfo d;
    CMG_TRY(device_info(&d));
    RowPlan q = R;
    q.resident = 1;
    cudaFuncAttributes fa;
    CMG_CUDA(cudaFuncGetAttributes(&fa, rows_kernel(q)));
    const long long v = (long long)d.max_smem_optin - (long long)fa.sharedSizeBytes - 512;
    *room = v > 0 ? (size_t)v : 0;
    return CMG_OK;
}

// Chooses between the resident and the streaming form from the plan's sizes.
static cmg_status_t rows_choose(int n, const PlanOut &o, RowPlan *R) {
    size_t room = 0;
    CMG_TRY(rows_room(*R, &room));
    R->resident = R->stage = 0;
    if (rows_smem(n, R->col16, 0, o) > room) return CMG_OK;
    R->resident = 1;
    // staging the iterate costs one trip to L2 and n / 8 cycles of copying per
    // SM; a scattered gather costs about 1.4 cycles more from L1 or L2 than from
    // shared memory.  (us per sweep unstaged and staged: 1,542 rows and 103K entries
    // 4.1 and 4.0, 5,688 and 129K 4.1 and 4.4, which the rule stages; 5,047 and 23K 3.4
    // and 4.3, 10K and 153K 3.5 and 5.2, 20K and 160K 3.7 and 5.9, which it does not.)
    if (R->col16 && rows_smem(n, 1, 1, o) <= room && (long long)n / 8 + 800 < (long long)o.max_e) R->stage = 1;
    R->res_e = o.max_e;
    R->res_i = o.max_i;
    R->res_r = o.max_r;
    R->smem = rows_smem(n, R->col16, R->stage, o);
    return CMG_OK;
}

bool rows_may_hold(int n) { return n <= kFixRowsMax; }

cmg_status_t build_row_plan(int n, long long nnz, const int *rp, const int *col, const double *w, double g,
                            const SweepLayout &L, RowPlan *R, size_t *bytes, cudaStream_t s) {
    unsigned long long ginv;
    int ge;
    if (!fix_reciprocal(g, &ginv, &ge)) return CMG_ERR_TOO_LARGE;
    DeviceInfo di;
    CMG_TRY(device_info(&di));
    R->col16 = n <= 65536 ? 1 : 0;
    Scratch scr(s);
    PlanOut *out_dev, o;
    CMG_TRY(scr.get(&out_dev, 1));
    // items: at most one per 32 rows plus one per 16 S entries and class
    const int S = nnz <= (long long)kWideEntries * di.sms ? 8 : 16;
    const long long cap = n / 32 + nnz / (8 * S) + 8;
    int4 *item;
    CMG_TRY(scr.get(&item, (size_t)cap + 1));
    CMG_TRY(dev_alloc_n(&R->range, (size_t)2 * di.sms + 1, s));
    auto plan = [&](int P, int quad) -> cmg_status_t {
        k_plan_units<<<1, kPlanThreads, 0, s>>>(n, rp, L.perm, S, quad, P, (int)cap, item, R->range, out_dev);
        CMG_TRY(launch_status());
        CMG_CUDA(cudaMemcpyAsync(&o, out_dev, sizeof(o), cudaMemcpyDeviceToHost, s));
        CMG_CUDA(cudaStreamSynchronize(s));
        return CMG_OK;
    };
    CMG_TRY(plan(di.sms, 1));
    if (o.entries >= 0x7fffffff || o.ni > cap || o.maxdeg > kRowsMaxRow) return CMG_ERR_TOO_LARGE;
    CMG_TRY(rows_choose(n, o, R));
    // (staging wants threads: each keeps 4 loads in flight)
    R->threads = std::max(R->stage ? 512 : 64, 32 * (1 + std::min(31, std::max(1, o.max_i))));
    if (!R->resident) {
        CMG_TRY(plan(2 * di.sms, 0));
        // only a layout that cannot stay in L2 is read evict-first
        R->stream = di.l2_bytes > 0 && o.entries * (R->col16 ? 10ll : 12ll) > (long long)di.l2_bytes;
        R->threads = kStreamThreads;
    }
    // a lane adds at most this many rows' sums
    if (o.max_i > 64 * (R->threads / 32 - 1)) return CMG_ERR_TOO_LARGE;
    R->P = o.P;
    R->ni = o.ni;
    R->entries = o.entries;
    CMG_TRY(dev_alloc_n(&R->item, (size_t)o.ni + 1, s));
    CMG_CUDA(cudaMemcpyAsync(R->item, item, sizeof(int4) * ((size_t)o.ni + 1), cudaMemcpyDeviceToDevice, s));
    const size_t ne = (size_t)std::max<long long>(o.entries, 1);
    CMG_TRY(dev_alloc(&R->ucol, ne * (R->col16 ? 2 : 4), s));
    CMG_TRY(dev_alloc_n(&R->uc, ne, s));
    CMG_TRY(dev_alloc_n(&R->ud, (size_t)n, s));
    CMG_TRY(dev_alloc_n(&R->acc, (size_t)kFixAccWords, s));
    const int fb = grid_for(32ll * o.ni, 256);
    if (R->col16)
        k_fill_units<<<fb, 256, 0, s>>>(o.ni, R->item, rp, col, w, ginv, ge, L.perm, L.inv, (uint16_t *)R->ucol, R->uc,
                                        R->ud);
    else
        k_fill_units<<<fb, 256, 0, s>>>(o.ni, R->item, rp, col, w, ginv, ge, L.perm, L.inv, (int *)R->ucol, R->uc, R->ud);
    CMG_TRY(launch_status());
    *bytes += 16 * ((size_t)o.ni + 1) + 4 * ((size_t)2 * di.sms + 1) + ne * (size_t)(R->col16 ? 10 : 12) +
              8 * (size_t)n + 8 * kFixAccWords;
    return CMG_OK;
}

void free_row_plan(RowPlan &R, cudaStream_t s) {
    dev_free(R.item, s);
    dev_free(R.range, s);
    dev_free(R.ucol, s);
    dev_free(R.uc, s);
    dev_free(R.ud, s);
    dev_free(R.acc, s);
    R = RowPlan();
}

cmg_status_t launch_power_rows(const RowPlan &R, const SweepLayout &L, PiArgs &a, GridSync *gs, cudaStream_t s) {
    a.perm = reinterpret_cast<const int *>(L.perm);
    a.items = R.item;
    a.item_range = R.range;
    a.res_entries = R.res_e;
    a.res_items = R.res_i;
    a.res_rows = R.res_r;
    a.lay_col = R.ucol;
    a.lay_w = R.uc;
    a.fix_d = R.ud;
    a.fix_acc = R.acc;
    const void *kern = rows_kernel(R);
    const int threads = R.threads;
    if (R.resident) CMG_TRY(allow_max_dynamic_smem(kern));
    int maxb = 0;
    CMG_TRY(coop_max_blocks(kern, threads, R.resident ? R.smem : 0, &maxb));
    if (maxb < R.P) return CMG_ERR_CUDA;
    CMG_CUDA(cudaMemsetAsync(R.acc, 0, 8 * kFixAccWords, s));
    void *args[] = {&a, &gs};
    return coop_launch(kern, R.P, threads, R.resident ? R.smem : 0, s, args, gs);
}

}  // namespace cmg
