// resident.cu -- the row kernel: power-iteration sweeps of a level spread over
// all SMs, with the level's matrix held in the SMs' shared memory for the
// whole launch where it fits (see k_power_rows), and the plan that deals the
// rows to the CTAs.
#include <algorithm>

#include "fixed.cuh"

namespace cmg {

// ------------------------------------------------------------------ plan
// Lanes per row by row length (FP64 items): steps of at most S entries per
// lane while the row fits a warp, S = 8 on levels with at most kWideEntries
// entries per SM (a sweep there is a chain of latencies: a row of 16 entries on
// one lane is two rounds of gathers, on two lanes one) and 16 above, where the
// FP64 pipe is the bound and every split row costs extra adds.
constexpr int kWideEntries = 8192;
constexpr int kItemCost = 256;     // per item, in entries: the rows' finish and stop sums
// Work of one CTA at least, in entries (an item counts kItemCost): below it more
// CTAs make the barrier dearer and the rows no faster, and leave no SM to the
// other streams of a server.
constexpr int kCtaWork = 2048;
constexpr int kPlanThreads = 1024;
constexpr int kRowsMaxRow = 4096;  // longest row the FP64 items take (one warp each)

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
template <typename DEG>
__device__ __forceinline__ int plan_units(int n, int S, DEG deg, int cap, int4 *item) {
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
                                                             const uint32_t *__restrict__ perm, int S, int P, int cap,
                                                             int4 *__restrict__ item, int *__restrict__ range,
                                                             PlanOut *__restrict__ out) {
    const int nu = plan_units(n, S, [&](int p) { return plan_deg(rp, perm, p); }, cap, item);
    if (threadIdx.x == 0) out->maxdeg = plan_deg(rp, perm, 0);
    plan_ranges(P, true, min(nu, cap), item, range, out);
}

// Everything k_power_fix needs of a level of at most kFixMaxN rows, one CTA per
// level and one launch for all of them: degree order (a stable counting sort),
// items and ranges, entries and diagonal in fixed point.  (The one-CTA and
// cluster kernels sorted and laid out their level in the sweep launch itself,
// and the cluster's plan read its row pointers back to the host.)
__global__ void __launch_bounds__(kPlanThreads) k_plan_small(const SmallJob *__restrict__ jobs) {
    __shared__ SmallJob J;
    __shared__ unsigned short s_perm[kFixMaxN], s_inv[kFixMaxN];
    __shared__ int s_hist[kFixMaxN + 1];
    __shared__ int s_md;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        J = jobs[blockIdx.x];
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
        s_inv[s_perm[p]] = (unsigned short)p;
        J.perm[p] = s_perm[p];
    }
    __syncthreads();
    // one item per row warp: of at most 8 steps where one CTA holds them all, else
    // of 16; beyond the warps, items of up to J.S steps dealt by their entries
    auto deg = [&](int p) { return len(s_perm[p]); };
    int nu = plan_units(n, 8, deg, J.cap_items, J.item);
    int steps = D <= 256 && nu <= J.one_cta ? 8 : 0;
    if (!steps) {
        nu = plan_units(n, 16, deg, J.cap_items, J.item);
        if (D <= 512 && nu <= J.cap_warps) steps = 16;
        else if (J.S != 16) nu = plan_units(n, J.S, deg, J.cap_items, J.item);
    }
    plan_ranges(J.C, false, min(nu, J.cap_items), J.item, J.range, J.out);
    const bool fits = nu <= J.cap_items && J.item[nu].y <= J.cap_entries;
    if (tid == 0) {
        J.out->by_warp = steps;
        J.out->maxdeg = fits ? 0 : -1;   // -1: beyond the capacities, not filled
        if (!fits) J.out->ni = 0;
    }
    if (!fits) return;
    for (int u = warp; u < nu; u += kPlanThreads / 32) {
        const int4 it = J.item[u];
        const int lg = it.w & 7, rows = it.w >> 3, r = lane >> lg, g = lane & ((1 << lg) - 1);
        const int p = it.x + (r < rows ? r : 0);
        int e0 = 0, deg = 0;
        if (r < rows) {
            e0 = J.rp[s_perm[p]];
            deg = len(s_perm[p]);
        }
        long long sum = 0;
        for (int t = 0; t < it.z; t++) {
            const int k = (t << lg) + g;
            const int d = it.y + 32 * t + lane;
            long long Cij = 0;
            int cl = p;
            if (k < deg) {
                Cij = fix_weight(J.w[e0 + k], J.ginv, J.ge);
                cl = s_inv[J.col[e0 + k]];
            }
            J.ucol[d] = (uint16_t)cl;
            J.uc[d] = fix_split(Cij);
            sum += Cij;
        }
        for (int o = (1 << lg) >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (r < rows && g == 0) J.ud[p] = fix_split(sum);
    }
}

// FP32 items are those of the sweep layout: its heavy rows (lw = -1, z their
// entries), then its slices (z their steps), in the layout's entry order.
__global__ void __launch_bounds__(kPlanThreads) k_plan_slices(int n, int h, int nsl, const int *__restrict__ meta, int P,
                                                              int4 *__restrict__ item, int *__restrict__ range,
                                                              PlanOut *__restrict__ out) {
    const int ni = h + nsl;
    for (int i = threadIdx.x; i < ni; i += blockDim.x) {
        const int o = meta[i], len = meta[i + 1] - o;
        if (i < h) item[i] = make_int4(i, o, len, -1);
        else item[i] = make_int4(h + 32 * (i - h), o, len >> 5, min(32, n - h - 32 * (i - h)) << 3);
    }
    if (threadIdx.x == 0) {
        item[ni] = make_int4(n, meta[ni], 0, 0);
        out->maxdeg = 0;
    }
    __syncthreads();
    plan_ranges(P, true, ni, item, range, out);
}

// Entries of the FP64 items, a warp per item; short rows and missing rows are
// padded with weight 0 and a valid column.
template <typename IDX>
__global__ void k_fill_units(int ni, const int4 *__restrict__ item, const int *__restrict__ rp,
                             const int *__restrict__ col, const double *__restrict__ w,
                             const uint32_t *__restrict__ perm, const int *__restrict__ inv, IDX *__restrict__ ucol,
                             double *__restrict__ uw) {
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < ni; u += warps) {
        const int4 it = item[u];
        const int lg = it.w & 7, rows = it.w >> 3, r = lane >> lg, g = lane & ((1 << lg) - 1);
        const int p = it.x + (r < rows ? r : 0);
        int e0 = 0, deg = 0;
        if (r < rows) {
            const int v = (int)perm[p];
            e0 = rp[v];
            deg = rp[v + 1] - e0;
        }
        for (int t = 0; t < it.z; t++) {
            const int k = (t << lg) + g;
            const size_t d = (size_t)it.y + 32 * t + lane;
            if (k < deg) {
                ucol[d] = (IDX)inv[col[e0 + k]];
                uw[d] = w[e0 + k];
            } else {
                ucol[d] = (IDX)p;
                uw[d] = 0.0;
            }
        }
    }
}

// ------------------------------------------------------------------ kernel
// Sweeps of a level over all SMs (cooperative, warp 0 the control warp, one
// grid barrier per sweep, iterates in degree order): the control path and the
// deferred stop decision are k_power_sell's.  A row warp takes items -- 32
// lanes on 32 / G rows, entry t of lane l at offset 32 t + l (FP64), or the
// sweep layout's heavy rows and slices (FP32: the same terms in the same order
// as k_power_sell, so the same bits).
//
// RES: one 1024-thread CTA per SM copies its items' columns, weights and g - d_i
// into shared memory once and sweeps from there.  On levels of a few million
// entries at most, what bounds a sweep is not bytes but the chain of
// dependent trips to L2 (columns and weights, then the iterate, per group of
// 8 entries, up to 16 groups on a 128-entry row) plus the barrier: from shared
// memory only the gathers remain, and with STAGE (the whole iterate copied to
// shared memory at the top of a sweep) one trip.  us per sweep on the slice
// kernel and here: FP64, 215 rows and 17K entries 14.0 and 4.4, 1,542 rows and
// 103K entries 17.3 and 6.3, 20K rows and 160K entries 16.0 and 5.2, 10K rows
// of a 3-D grid's hierarchy 8.3 and 4.9; FP32, 3,820 rows and 2.1M entries 14.5
// and 9.9.
// Otherwise: two 512-thread CTAs per SM stream the items (FP64 levels beyond
// shared memory): 100^3 grid levels 0 and 1 40.4 and 38.0, 23.6 and 22.5.
template <typename T, typename IDX, bool RES, bool STAGE, bool STREAM>
__global__ void __launch_bounds__(RES ? 1024 : 512, RES ? 1 : 2) k_power_rows(PiArgs a, GridSync *gs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool fp64 = sizeof(T) == 8;
    __shared__ Part s_pw[32];
    __shared__ Slot s_slot[2];
    __shared__ GridBar s_bar;
    __shared__ Ctl c;
    const int n = a.n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nw = (int)(blockDim.x >> 5);
    if (tid == 0) grid_bar_init(&s_bar, gs);
    T *const ring0 = (T *)a.buf[0], *const ring1 = (T *)a.buf[1], *const ring2 = (T *)a.buf[2];
    const T g = (T)a.g;
    const float inv_gf = 1.0f / (float)a.g;
    const int ib = a.item_range[blockIdx.x], ie = a.item_range[blockIdx.x + 1];
    const int4 first = a.items[ib], last = a.items[ie];
    const int r0 = first.x, r1 = last.x, e_lo = first.y;
    // shared memory (RES): items, weights, g - d_i, the staged iterate, columns
    int4 *s_item = reinterpret_cast<int4 *>(smem_raw);
    T *s_w = reinterpret_cast<T *>(s_item + a.res_items);
    T *s_x = s_w + a.res_entries;
    double *s_gd = reinterpret_cast<double *>(s_x + (STAGE ? ((n + 3) & ~3) : 0));
    IDX *s_c = reinterpret_cast<IDX *>(s_gd + (fp64 ? ((a.res_rows + 1) & ~1) : 0));
    if (RES) {
        const T *gw = reinterpret_cast<const T *>(a.lay_w) + e_lo;
        const IDX *gc = reinterpret_cast<const IDX *>(a.lay_col) + e_lo;
        const int ne = last.y - e_lo;   // a multiple of 8: 16-byte copies
        for (int k = tid; k < ne * (int)sizeof(T) / 16; k += blockDim.x)
            reinterpret_cast<uint4 *>(s_w)[k] = __ldg(reinterpret_cast<const uint4 *>(gw) + k);
        for (int k = tid; k < ne * (int)sizeof(IDX) / 16; k += blockDim.x)
            reinterpret_cast<uint4 *>(s_c)[k] = __ldg(reinterpret_cast<const uint4 *>(gc) + k);
        for (int k = tid; k < ie - ib; k += blockDim.x) {
            int4 it = a.items[ib + k];
            it.y -= e_lo;
            s_item[k] = it;
        }
    }
    const IDX *C = RES ? s_c : reinterpret_cast<const IDX *>(a.lay_col);
    const T *W = RES ? s_w : reinterpret_cast<const T *>(a.lay_w);

    // ---------------------------------------------------------- start phase
    {
        const void *cb = nullptr;
        double cmu = 0.0, cinv = 0.0;
        if (a.start == 1) {
            cb = a.cbuf[a.cres->buf];
            cmu = a.cres->mu;
            cinv = a.cres->inv_s;
        }
        Part acc = part_zero();
        for (int p = r0 + tid; p < r1; p += blockDim.x) {
            const int old = a.perm[p];
            const T xt = (T)start_value(a, old, cb, cmu, cinv);
            ring0[p] = xt;
            if (fp64) {
                double d = 0.0;
                for (int e = __ldg(a.rp + old), e1 = __ldg(a.rp + old + 1); e < e1; e++) d += __ldg(a.w + e);
                if (RES) s_gd[p - r0] = a.g - d;
                else a.gd[p] = a.g - d;
            }
            const ff v = fp64 ? ff_from_double((double)xt) : ff_make((float)xt, 0.f);
            acc.A = ff_add(acc.A, v);
            acc.B = ff_add(acc.B, ff_mul(v, v));
        }
        Part p = warp_sum_part(acc);
        if (lane == 0) s_pw[warp] = p;
        __syncthreads();
        if (warp == 0) {
            Part q = (lane < nw) ? s_pw[lane] : part_zero();
            q = warp_sum_part(q);
            if (lane == 0) store_part(a.partials + blockIdx.x, q);
        }
    }
    if (!grid_sync(&s_bar)) return;
    if (warp == 0) {
        const Part q = grid_part(a.partials, lane);
        const double mu0 = to_d(q.A) / (double)n;
        double ss0 = to_d(q.B) - (double)n * mu0 * mu0;
        if (ss0 < 0.0) ss0 = 0.0;
        const int e0 = start_exponent(ss0);
        if (lane == 0) {
            ctl_init(c, a, mu0, ss0, e0);
            s_slot[1] = slot_make(ff_from_double(mu0), e0, a.g, c.inv_g, fp64);
            s_slot[0] = slot_make(ff_zero(), 0, a.g, c.inv_g, fp64);
        }
    }
    __syncthreads();

    const bool no_sweeps = (a.mode == 1 && a.k_fixed <= 0);
    int s = 0;
    int exit_kind = no_sweeps ? 2 : 0;
    while (!no_sweeps) {
        const Slot sl = s_slot[(s + 1) & 1];
        if (sl.stop) {
            exit_kind = 1;
            break;
        }
        if ((a.mode == 1 && s >= a.k_fixed) || (a.mode == 0 && s >= a.max_sweeps)) {
            exit_kind = 2;
            break;
        }
        const T *x = pick3<T *>(ring0, ring1, ring2, s % 3);
        T *y = pick3<T *>(ring0, ring1, ring2, (s + 1) % 3);
        if (warp == 0) {
            if (s >= 1) {
                const Part q = grid_part(a.partials + (size_t)(s & 1) * gridDim.x, lane);
                if (lane == 0) ctrl_step(a, s, q, c, &s_slot[s & 1], false, fp64);
            }
        } else {
            const T m = fp64 ? (T)sl.m_d : (T)sl.m.hi;
            const T sig = fp64 ? (T)sl.sig_d : (T)scale2f(inv_gf, sl.e);
            const T gm = fp64 ? (T)sl.gm_d : g * m;
            Acc<T> acc;
            acc.reset();
            if (STAGE) {
                // the whole iterate, in 16-byte pieces, then the row warps
                // meet (the control warp does not take part)
                const int nrt = (int)blockDim.x - 32;
                const int nv = n * (int)sizeof(T) / 16;
                for (int k = tid - 32; k < nv; k += nrt)
                    reinterpret_cast<float4 *>(s_x)[k] = __ldcg(reinterpret_cast<const float4 *>(x) + k);
                for (int k = nv * (16 / (int)sizeof(T)) + tid - 32; k < n; k += nrt) s_x[k] = __ldcg(x + k);
                bar_rows(nrt);
            }
            auto ldx = [&](int k) { return STAGE ? s_x[k] : LDXG(x + k); };
            auto finish = [&](int i, T xi, T ac, double gd) {
                T yv;
                if (fp64) yv = (T)((fma(gd, (double)xi, (double)ac) - (double)gm) * (double)sig);
                else yv = (g * (xi - m) - ac) * sig;
                y[i] = yv;
                acc.add(yv, xi);
            };
            for (int k = ib + warp - 1; k < ie; k += nw - 1) {
                const int4 it = RES ? s_item[k - ib] : __ldg(a.items + k);
                if (fp64) {
                    const int lg = it.w & 7, rows = it.w >> 3, r = lane >> lg;
                    const int i = it.x + (r < rows ? r : 0);
                    const T xi = ldx(i);
                    const double gd = RES ? s_gd[i - r0] : LDX(a.gd + i);
                    const int base = it.y + lane;
                    T a0 = (T)0, a1 = (T)0;
                    for (int t0 = 0; t0 < it.z; t0 += 8) {
                        int cc[8];
                        T ww[8], xx[8];
#pragma unroll
                        for (int u = 0; u < 8; u++) {
                            cc[u] = i;
                            ww[u] = (T)0;
                            if (t0 + u < it.z) {
                                const int f = base + 32 * (t0 + u);
                                cc[u] = (int)(STREAM ? __ldcs(C + f) : C[f]);
                                ww[u] = STREAM ? __ldcs(W + f) : W[f];
                            }
                        }
#pragma unroll
                        for (int u = 0; u < 8; u++) xx[u] = (t0 + u < it.z) ? ldx(cc[u]) : (T)0;
#pragma unroll
                        for (int u = 0; u < 8; u++) {
                            if (t0 + u >= it.z) break;
                            if (u & 1) a1 = fma(ww[u], xx[u], a1);
                            else a0 = fma(ww[u], xx[u], a0);
                        }
                    }
                    T ac = a0 + a1;
                    for (int o = (1 << lg) >> 1; o > 0; o >>= 1) ac += __shfl_xor_sync(0xffffffffu, ac, o);
                    if (r < rows && (lane & ((1 << lg) - 1)) == 0) finish(i, xi, ac, gd);
                } else if (it.w < 0) {
                    // a heavy row: its chunks (as k_power_sell cuts them) one
                    // after the other, the partials added in chunk order
                    const int len = it.z, nc = (len + kHeavyChunk - 1) / kHeavyChunk;
                    const int per = (((len + nc - 1) / nc) + 7) & ~7;
                    const T xi = ldx(it.x);
                    T tot = (T)0, ac = (T)0;
                    for (int ch = 0; ch < nc; ch++) {
                        const int f0 = min(len, ch * per), f1 = min(len, f0 + per);
                        ac = row_sum_octets<T, IDX, 2>(C, W, ((it.y + f0) >> 3) + lane, (it.y + f1) >> 3, xi, ldx,
                                                       false);
                        ac = warp_sum(ac);
                        if (ch < nc - 1) tot += ac;
                    }
                    if (lane == 0) finish(it.x, xi, nc == 1 ? ac : tot + ac, 0.0);
                } else {
                    const int i = it.x + lane;
                    const bool ok = lane < (it.w >> 3);
                    const T xi = ok ? ldx(i) : (T)0;
                    const int so = it.y + lane;
                    const T ac = row_sum_grouped<T, IDX>(C, W, so, so + 32 * it.z, 32, xi, ldx, false);
                    if (ok) finish(i, xi, ac, 0.0);
                }
            }
            const Part p = warp_sum_part(acc.get());
            if (lane == 0) s_pw[warp] = p;
        }
        __syncthreads();
        if (warp == 0) {
            Part q = (lane >= 1 && lane < nw) ? s_pw[lane] : part_zero();
            q = warp_sum_part(q);
            if (lane == 0) {
                // the CTA's rows were stored before the CTA barrier above, so
                // thread 0 can arrive for the CTA at once
                store_part(a.partials + (size_t)((s + 1) & 1) * gridDim.x + blockIdx.x, q);
                s_bar.ok = grid_arrive_wait(&s_bar);
            }
        }
        __syncthreads();
        if (!s_bar.ok) return;
        s++;
    }
    // ---------------------------------------------------------- result
    if (warp == 0) {
        if (exit_kind == 2 && !no_sweeps) {
            const Part q = grid_part(a.partials + (size_t)(s & 1) * gridDim.x, lane);
            if (lane == 0) ctrl_step(a, s, q, c, nullptr, true, fp64);
        }
        if (blockIdx.x == 0 && lane == 0) {
            const int rs = c.res_sweep;
            const int rb = c.zero ? (rs - 1) % 3 : rs % 3;
            write_result(a, c, rb, (rs + 2) % 3);
        }
    }
}

template <typename T, typename IDX>
static const void *rows_kernel_t(const RowPlan &R) {
    if (R.resident)
        return R.stage ? (const void *)k_power_rows<T, IDX, true, true, false>
                       : (const void *)k_power_rows<T, IDX, true, false, false>;
    if constexpr (sizeof(T) == 8)
        return R.stream ? (const void *)k_power_rows<T, IDX, false, false, true>
                        : (const void *)k_power_rows<T, IDX, false, false, false>;
    return nullptr;
}

static const void *rows_kernel(const RowPlan &R) {
    if (R.fp32) return R.col16 ? rows_kernel_t<float, uint16_t>(R) : rows_kernel_t<float, int>(R);
    return R.col16 ? rows_kernel_t<double, uint16_t>(R) : rows_kernel_t<double, int>(R);
}

cmg_status_t launch_plan_small(const SmallJob *jobs_dev, int count, cudaStream_t s) {
    k_plan_small<<<count, kPlanThreads, 0, s>>>(jobs_dev);
    return launch_status();
}

int rows_threads(const RowPlan &R) { return R.resident ? 1024 : 512; }

static size_t rows_smem(int n, int fp32, int col16, int stage, const PlanOut &o) {
    const size_t e = fp32 ? 4 : 8, isz = col16 ? 2 : 4;
    return 16 * (size_t)o.max_i + (e + isz) * (size_t)o.max_e + (stage ? e * (size_t)((n + 3) & ~3) : 0) +
           (fp32 ? 0 : 8 * (size_t)((o.max_r + 1) & ~1)) + 16;
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
    const size_t e = R->fp32 ? 4 : 8;
    R->resident = R->stage = 0;
    if (rows_smem(n, R->fp32, R->col16, 0, o) > room) return CMG_OK;
    R->resident = 1;
    // staging the iterate costs one trip to L2 and n e / 64 cycles of copying
    // per SM; a scattered gather costs about 1.4 cycles more from L1 or L2 than
    // from shared memory
    if (rows_smem(n, R->fp32, R->col16, 1, o) <= room && (long long)n * e / 64 + 800 < (long long)o.max_e)
        R->stage = 1;
    R->res_e = o.max_e;
    R->res_i = o.max_i;
    R->res_r = o.max_r;
    R->smem = rows_smem(n, R->fp32, R->col16, R->stage, o);
    return CMG_OK;
}

cmg_status_t build_row_plan(int n, long long nnz, const int *rp, const int *col, const double *w,
                            const SweepLayout &L, int fp32, RowPlan *R, size_t *bytes, cudaStream_t s) {
    DeviceInfo di;
    CMG_TRY(device_info(&di));
    R->fp32 = fp32;
    R->col16 = n <= 65536 ? 1 : 0;
    Scratch scr(s);
    PlanOut *out_dev, o;
    CMG_TRY(scr.get(&out_dev, 1));
    // items: at most one per 32 rows plus one per S / 4 ... entries (a row on G
    // lanes holds more than G S / 2 entries and takes G / 32 of an item)
    const int S = nnz <= (long long)kWideEntries * di.sms ? 8 : 16;
    const long long cap = fp32 ? (long long)L.hheavy[0] + (n - L.hheavy[0] + 31) / 32
                               : n / 32 + nnz / (16 * (S / 2)) + 8;
    int4 *item;
    CMG_TRY(scr.get(&item, (size_t)cap + 1));
    CMG_TRY(dev_alloc_n(&R->range, (size_t)2 * di.sms + 1, s));
    auto plan = [&](int P) -> cmg_status_t {
        if (fp32) {
            const int h = L.hheavy[0];
            k_plan_slices<<<1, kPlanThreads, 0, s>>>(n, h, (n - h + 31) / 32, L.meta, P, item, R->range, out_dev);
        } else {
            k_plan_units<<<1, kPlanThreads, 0, s>>>(n, rp, L.perm, S, P, (int)cap, item, R->range, out_dev);
        }
        CMG_TRY(launch_status());
        CMG_CUDA(cudaMemcpyAsync(&o, out_dev, sizeof(o), cudaMemcpyDeviceToHost, s));
        CMG_CUDA(cudaStreamSynchronize(s));
        return CMG_OK;
    };
    CMG_TRY(plan(di.sms));
    if (o.entries >= 0x7fffffff || o.ni > cap || o.maxdeg > kRowsMaxRow) return CMG_ERR_TOO_LARGE;
    CMG_TRY(rows_choose(n, o, R));
    if (!R->resident) {
        if (fp32) return CMG_ERR_TOO_LARGE;   // FP32 levels are streamed by the slice kernel
        CMG_TRY(plan(2 * di.sms));
        const long long lay = o.entries * (long long)(R->col16 ? 2 + 8 : 4 + 8);
        R->stream = di.l2_bytes > 0 && lay > (long long)di.l2_bytes;
    }
    R->P = o.P;
    R->ni = o.ni;
    R->entries = o.entries;
    CMG_TRY(dev_alloc_n(&R->item, (size_t)o.ni + 1, s));
    CMG_CUDA(cudaMemcpyAsync(R->item, item, sizeof(int4) * ((size_t)o.ni + 1), cudaMemcpyDeviceToDevice, s));
    *bytes += 16 * ((size_t)o.ni + 1) + 4 * ((size_t)2 * di.sms + 1);
    if (!fp32) {
        const size_t ne = (size_t)std::max<long long>(o.entries, 1);
        CMG_TRY(dev_alloc(&R->ucol, ne * (R->col16 ? 2 : 4), s));
        CMG_TRY(dev_alloc_n(&R->uw, ne, s));
        const int fb = grid_for(32ll * o.ni, 256);
        if (R->col16)
            k_fill_units<<<fb, 256, 0, s>>>(o.ni, R->item, rp, col, w, L.perm, L.inv, (uint16_t *)R->ucol, R->uw);
        else
            k_fill_units<<<fb, 256, 0, s>>>(o.ni, R->item, rp, col, w, L.perm, L.inv, (int *)R->ucol, R->uw);
        CMG_TRY(launch_status());
        *bytes += ne * (size_t)((R->col16 ? 2 : 4) + 8);
    }
    return CMG_OK;
}

void free_row_plan(RowPlan &R, cudaStream_t s) {
    dev_free(R.item, s);
    dev_free(R.range, s);
    dev_free(R.ucol, s);
    dev_free(R.uw, s);
    R = RowPlan();
}

cmg_status_t launch_power_rows(const RowPlan &R, const SweepLayout &L, PiArgs &a, GridSync *gs, cudaStream_t s) {
    a.perm = reinterpret_cast<const int *>(L.perm);
    a.items = R.item;
    a.item_range = R.range;
    a.res_entries = R.res_e;
    a.res_items = R.res_i;
    a.res_rows = R.res_r;
    a.lay_col = R.fp32 ? L.bcol : R.ucol;
    a.lay_w = R.fp32 ? L.bw : (const void *)R.uw;
    const void *kern = rows_kernel(R);
    const int threads = rows_threads(R);
    if (R.resident) CMG_TRY(allow_max_dynamic_smem(kern));
    int maxb = 0;
    CMG_TRY(coop_max_blocks(kern, threads, R.resident ? R.smem : 0, &maxb));
    if (maxb < R.P) return CMG_ERR_CUDA;
    Scratch scr(s);
    PartRec *partials;
    CMG_TRY(scr.get(&partials, (size_t)2 * R.P));
    a.partials = partials;
    void *args[] = {&a, &gs};
    return coop_launch(kern, R.P, threads, R.resident ? R.smem : 0, s, args, gs);
}

}  // namespace cmg
