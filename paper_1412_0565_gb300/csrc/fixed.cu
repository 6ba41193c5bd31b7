// fixed.cu -- k_power_fix: FP64 power-iteration sweeps of a small level in fixed
// point (fixed.cuh), the level held in shared memory by one CTA or one
// thread-block cluster.
#include <math.h>

#include <algorithm>

#include "fixed.cuh"

namespace cmg {

constexpr int kFixMaxThreads = 1024;
constexpr int kFixMaxCtas = 8;

__device__ __forceinline__ unsigned fix_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned fix_ctas() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// address of a shared-memory object of this CTA in CTA `cta` of the cluster
__device__ __forceinline__ unsigned fix_peer(const void *local, unsigned cta) {
    unsigned ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(ra)
                 : "r"((unsigned)__cvta_generic_to_shared(local)), "r"(cta));
    return ra;
}
// all threads of all CTAs; orders the stores and reductions into other CTAs'
// shared memory before it with the reads after it
__device__ __forceinline__ void fix_barrier(int C) {
    if (C == 1) {
        asm volatile("bar.sync 0;" ::: "memory");
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// Result -> buf[0], previous iterate -> buf[1], in row order (res: fix_finish).
__device__ __forceinline__ void fix_write(const PiArgs &a, const int2 *ring, int nr, const int *res) {
    const int rs = res[0];
    const int2 *rr = ring + (size_t)(res[1] ? (rs + 2) % 3 : rs % 3) * nr, *rp = ring + (size_t)((rs + 2) % 3) * nr;
    double *o0 = (double *)a.buf[0], *o1 = (double *)a.buf[1];
    for (int i = threadIdx.x; i < a.n; i += blockDim.x) {
        const int v = a.perm[i];
        o0[v] = fix_value(rr[i]);
        o1[v] = rs > 0 ? fix_value(rp[i]) : 0.0;
    }
}

// Every CTA holds the whole iterate ring and its share of the items.  A sweep:
// warp 0 (control) turns the previous sweep's sums into decisions while the
// row warps compute their items from the local iterate and store each row's
// value into every CTA's ring; the row warps leave their lanes' stop sums in
// shared memory, meet, and one warp per sum adds them up and stores the total
// into every CTA's slot; then one barrier.  What bounds a sweep is this chain:
// an item's entries, a row's finish, the sums, the barrier; the control step
// runs beside it.  Six row warps reduce a sum each: a warp that reduced its
// own five sums spent 610 cycles on 16 warp reductions, and atomics into the
// other CTAs another 900 (3 CTAs) to 2,200 (8 CTAs).
// us per sweep in FP64 (one cluster) and here: the 3,048-row level of the 100^3
// grid 5.67 and 3.18.
__global__ void __launch_bounds__(kFixMaxThreads) k_power_fix(PiArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(16) long long s_acc[2][kFixMaxCtas][kFixSums];   // the CTAs' stop sums by sweep parity
    __shared__ __align__(16) long long s_rec[32][kFixSums];               // the start's sums by warp
    __shared__ FixSlot s_slot[2];
    __shared__ double s_mx[32];
    __shared__ int s_bad;
    __shared__ int s_res[2];       // sweeps of the result, annihilated
    const int n = a.n, nr = (n + 1) & ~1;
    const int C = (int)fix_ctas();
    const unsigned rank = fix_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nw = (int)(blockDim.x >> 5);
    int4 *s_item = reinterpret_cast<int4 *>(smem_raw);
    int2 *ring = reinterpret_cast<int2 *>(s_item + a.res_items);       // [3][nr]
    int2 *s_c = ring + 3 * (size_t)nr;
    int2 *s_d = s_c + a.res_entries;
    long long *s_lane = reinterpret_cast<long long *>(s_d + a.res_rows);   // [kFixSums][row threads]
    uint16_t *s_col = reinterpret_cast<uint16_t *>(s_lane + kFixSums * (blockDim.x - 32));
    const int ib = a.item_range[rank], ie = a.item_range[rank + 1];
    const int4 first = a.items[ib], last = a.items[ie];
    const int r0 = first.x, e_lo = first.y;
    {
        const int2 *gc = reinterpret_cast<const int2 *>(a.lay_w) + e_lo;
        const uint16_t *gcol = reinterpret_cast<const uint16_t *>(a.lay_col) + e_lo;
        const int ne = last.y - e_lo;   // a multiple of 32
        for (int k = tid; k < ne; k += blockDim.x) s_c[k] = __ldg(gc + k);
        for (int k = tid; k < ne / 2; k += blockDim.x)
            reinterpret_cast<unsigned *>(s_col)[k] = __ldg(reinterpret_cast<const unsigned *>(gcol) + k);
        for (int k = tid; k < last.x - r0; k += blockDim.x) s_d[k] = __ldg(a.fix_d + r0 + k);
        for (int k = tid; k < ie - ib; k += blockDim.x) {
            int4 it = a.items[ib + k];
            it.y -= e_lo;
            s_item[k] = it;
        }
    }
    fix_start(a, ring, s_mx, s_rec, &s_bad);

    const int limit = s_bad ? 0 : (a.mode == 1 ? max(a.k_fixed, 0) : a.max_sweeps);
    if (warp == 0) {
        // ------------------------------------------------------ control warp
        const double omt = 1.0 - a.tol, omt2 = omt * omt;
        const float inv_n = 1.0f / (float)n;
        FixCtl c;
        unsigned m;
        const long long v0 = fix_sum_records(&s_rec[0][0], nw, lane, &m);
        fix_ctl_start(a, lane, v0, omt2, n, c, s_slot);
        fix_barrier(C);   // every CTA is set up before another stores into it
        int s = 0, rs = 0, code = 0;
        bool counted = false;
        FixSlot nx;
        for (;; s++) {
            if (s_slot[(s + 1) & 1].stop) break;
            if (s >= limit) {
                counted = true;
                break;
            }
            if (s >= 1) {
                const long long v = fix_sum_records(&s_acc[s & 1][0][0], C, lane, &m);
                code = fix_decide(a, lane, v, m, omt2, inv_n, c, &nx);
                rs = s;
                nx.stop = code == 2 || (code == 1 && a.mode == 0);
                if (lane == 0) s_slot[s & 1] = nx;
                __syncwarp();
            }
            fix_barrier(C);
        }
        if (counted && limit > 0) {
            const long long v = fix_sum_records(&s_acc[s & 1][0][0], C, lane, &m);
            code = fix_decide(a, lane, v, m, omt2, inv_n, c, &nx);
            rs = s;
        }
        fix_finish(a, lane, n, rs, code, counted, s_bad != 0, rank == 0, 0, c, s_res);
        if (rank == 0 && lane == 0) {
            // written to buf[0], the previous iterate to buf[1]
            a.res->buf = 0;
            a.res->buf_prev = 1;
        }
    } else {
        // ------------------------------------------------------ row warps
        // shared-memory windows of the other CTAs, as offsets from this one's
        unsigned win[kFixMaxCtas - 1];
#pragma unroll
        for (int p = 0; p < kFixMaxCtas - 1; p++)
            win[p] = p < C - 1
                         ? fix_peer(smem_raw, p < (int)rank ? p : p + 1) - (unsigned)__cvta_generic_to_shared(smem_raw)
                         : 0u;
        const int nrw = nw - 1, rt = tid - 32, nrt = (int)blockDim.x - 32;
        fix_barrier(C);
        int k0 = 0, k1 = 1;   // s, s + 1 modulo 3
        for (int s = 0;; s++) {
            const FixSlot sl = s_slot[(s + 1) & 1];
            if (sl.stop || s >= limit) break;
            const int2 *x = ring + (size_t)k0 * nr;
            int2 *y = ring + (size_t)k1 * nr;
            FixSum f;
            f.reset();
            for (int k = ib + warp - 1; k < ie; k += nrw) {
                const int4 it = s_item[k - ib];
                const int lg = it.w & 7, rows = it.w >> 3, r = lane >> lg;
                const int i = it.x + (r < rows ? r : 0);
                const int2 xi = x[i];
                const int2 d = s_d[i - r0];
                FixAcc t;
                t.reset();
                fix_quads(t, it.z, s_col + it.y + lane, s_c + it.y + lane, [&](int q) { return x[q]; });
                const bool leads = r < rows && (lane & ((1 << lg) - 1)) == 0;
                if (leads) t.add(xi, make_int2(-d.x, -d.y));
                t.carry();
                const long long pr = t.lanes(lg);
                if (leads) {
                    const long long X = fix_join(xi), Y = fix_row(X, pr, sl.M, sl.e);
                    const int2 yv = fix_split(Y);
                    y[i] = yv;
                    const unsigned ya = (unsigned)__cvta_generic_to_shared(y + i);
#pragma unroll
                    for (int p = 0; p < kFixMaxCtas - 1; p++)
                        if (p < C - 1)
                            asm volatile("st.shared::cluster.v2.s32 [%0], {%1, %2};" ::"r"(ya + win[p]), "r"(yv.x), "r"(yv.y)
                                         : "memory");
                    f.add(Y, yv, FixSum::narrow(Y), FixSum::narrow(X));
                }
                __syncwarp();
            }
            const FixVals fv = fix_vals(f, false);
#pragma unroll
            for (int v = 0; v < 5; v++) s_lane[v * nrt + rt] = fv.v[v];
            s_lane[5 * nrt + rt] = (long long)f.mx;
            bar_rows(nrt);
            for (int v = warp - 1; v < kFixSums; v += nrw) {
                const long long *src = s_lane + v * nrt + lane;
                long long sum = 0;
                if (v < 5) {
                    for (int k = 0; k < nrw; k++) sum += src[32 * k];
                    sum = warp_sum(sum);
                } else {
                    unsigned m = 0;
                    for (int k = 0; k < nrw; k++) m = max(m, (unsigned)src[32 * k]);
                    sum = (long long)__reduce_max_sync(0xffffffffu, m);
                }
                // lane p: the sum into CTA p's slot of this rank
                if (lane < C)
                    asm volatile("st.shared::cluster.s64 [%0], %1;" ::"r"(fix_peer(&s_acc[(s + 1) & 1][rank][v], lane)), "l"(sum)
                                 : "memory");
                __syncwarp();
            }
            fix_barrier(C);
            k0 = k1;
            k1 = k1 == 2 ? 0 : k1 + 1;
        }
    }
    __syncthreads();
    if (rank == 0) fix_write(a, ring, nr, s_res);
}

// Row warps per CTA of the register form: 15 leave 128 registers a thread (with 31
// and 64 registers the 3,048-row level of the 100^3 grid took 4.0 us per sweep,
// from shared memory 3.3).
constexpr int kFixWarps = 15;

// The same sweeps with one item of at most U steps per row warp: a lane keeps its
// entries (column offsets and coefficients) in registers for the whole launch,
// so a sweep reads only the iterate; a leading lane keeps its row's value; the warp
// reduces its own five sums and stores them into every CTA's slots, where the
// control warps add them up.
// Row warps and control warp run separate loops that meet at the barrier.  What
// bounds a sweep is the longer of two chains: gathers, 32 multiply-adds, the
// lanes' sums, finish, warp sums (about 900 cycles), and the control step
// (about 1,000); then the barrier (60 cycles in one CTA, 420 in a cluster).
// us per sweep in FP64 (one CTA up to 512 rows, cluster above), from shared memory
// (k_power_fix, with three of the four products) and here, the 853-, 239-, 66- and
// 18-row levels of the 100^3 grid: 3.55 / 2.48 / 1.70 / 1.24, 2.85 / 2.05 / 1.37 /
// 1.23, and 1.44 / 1.22 / 1.05 / 0.95 (1.29 / 1.07 / 0.95 / 0.87 with three products
// and 57 bits: the fourth product and the wider sums are the price of the accuracy
// stated in fixed.cuh).
template <int U>
__global__ void __launch_bounds__(32 * (kFixWarps + 1)) k_power_fix_reg(PiArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(16) long long s_rec[kFixWarps + 1][kFixSums];   // the start's sums by warp
    __shared__ FixSlot s_slot[2];
    __shared__ int s_res[2];       // sweeps of the result, annihilated
    __shared__ double s_mx[32];
    __shared__ int s_bad;
    const int n = a.n, nr = (n + 1) & ~1;
    const int C = (int)fix_ctas();
    const unsigned rank = fix_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nw = (int)(blockDim.x >> 5), nrw = nw - 1;
    int2 *ring = reinterpret_cast<int2 *>(smem_raw);                        // [3][nr]
    long long *s_acc = reinterpret_cast<long long *>(ring + 3 * (size_t)nr);   // [2][C][nrw][kFixSums]
    for (int k = tid; k < 2 * C * nrw * kFixSums; k += blockDim.x) s_acc[k] = 0;
    fix_start(a, ring, s_mx, s_rec, &s_bad);

    const int limit = s_bad ? 0 : (a.mode == 1 ? max(a.k_fixed, 0) : a.max_sweeps);
    if (warp == 0) {
        // ------------------------------------------------------ control warp
        const double omt = 1.0 - a.tol, omt2 = omt * omt;
        const float inv_n = 1.0f / (float)n;
        const int N = C * nrw;
        FixCtl c;
        unsigned m;
        const long long v0 = fix_sum_records(&s_rec[0][0], nw, lane, &m);
        fix_ctl_start(a, lane, v0, omt2, n, c, s_slot);
        fix_barrier(C);   // every CTA is set up before another stores into it
        // totals of the sweep of parity par: a record per lane
        auto decide = [&](int par, FixSlot *next) -> int {
            unsigned mx;
            const long long v = fix_sum_records(s_acc + (size_t)par * N * kFixSums, N, lane, &mx);
            return fix_decide(a, lane, v, mx, omt2, inv_n, c, next);
        };
        int s = 0, rs = 0, code = 0;
        bool counted = false;
        FixSlot nx;
        for (;; s++) {
            if (s_slot[(s + 1) & 1].stop) break;
            if (s >= limit) {
                counted = true;
                break;
            }
            if (s >= 1) {
                code = decide(s & 1, &nx);
                rs = s;
                nx.stop = code == 2 || (code == 1 && a.mode == 0);
                if (lane == 0) s_slot[s & 1] = nx;
                __syncwarp();
            }
            fix_barrier(C);
        }
        if (counted && limit > 0) {
            code = decide(s & 1, &nx);
            rs = s;
        }
        fix_finish(a, lane, n, rs, code, counted, s_bad != 0, rank == 0, 0, c, s_res);
        if (rank == 0 && lane == 0) {
            // written to buf[0], the previous iterate to buf[1]
            a.res->buf = 0;
            a.res->buf_prev = 1;
        }
    } else {
        // ------------------------------------------------------ row warps
        const int k0 = (int)((long long)a.nitems * rank / C), k1 = (int)((long long)a.nitems * (rank + 1) / C);
        const int k = k0 + warp - 1;
        const bool have = k < k1;
        const int4 it = a.items[have ? k : a.nitems];
        const int lg = it.w & 7, rows = it.w >> 3, r = lane >> lg;
        const int i = have ? it.x + (r < rows ? r : 0) : 0;
        const bool leads = have && r < rows && (lane & ((1 << lg) - 1)) == 0;
        int off[U];
        int2 cf[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            off[u] = i;
            cf[u] = make_int2(0, 0);
            if (have && u < it.z) {
                const int f = it.y + 32 * u + lane;
                off[u] = reinterpret_cast<const uint16_t *>(a.lay_col)[f];
                cf[u] = reinterpret_cast<const int2 *>(a.lay_w)[f];
            }
        }
        // the diagonal: one more entry of the lane that leads the row
        int2 d = make_int2(0, 0);
        if (leads) {
            d = a.fix_d[i];
            d = make_int2(-d.x, -d.y);
        }
        unsigned win[kFixMaxCtas - 1];
#pragma unroll
        for (int p = 0; p < kFixMaxCtas - 1; p++)
            win[p] = p < C - 1
                         ? fix_peer(smem_raw, p < (int)rank ? p : p + 1) - (unsigned)__cvta_generic_to_shared(smem_raw)
                         : 0u;
        // lanes 4 g + j store value vi of the warp's sums into CTAs j and j + 4
        const int grp = lane >> 2, vi = grp < 3 ? grp : grp - 1;
        const bool sends = grp == 0 || grp == 1 || grp == 2 || grp == 4 || grp == 5 || grp == 6;
        const int p0 = lane & 3, p1 = p0 + 4;
        const size_t N = (size_t)C * nrw * kFixSums;
        long long *mine = s_acc + ((size_t)rank * nrw + warp - 1) * kFixSums + (sends ? vi : 0);
        const unsigned acc0 = sends && p0 < C ? fix_peer(mine, p0) : 0u, acc1 = sends && p1 < C ? fix_peer(mine, p1) : 0u;
        const unsigned pstep = (unsigned)(N * sizeof(long long));
        // a leading lane keeps its row's value from sweep to sweep
        int2 xi = ring[i];
        long long X = fix_join(xi);
        fix_barrier(C);
        int s = 0, b0 = 0, b1 = nr;   // ring slots of x and y
        for (;; s++) {
            const FixSlot sl = s_slot[(s + 1) & 1];
            if (sl.stop || s >= limit) break;
            if (have) {
                const int2 *x = ring + b0;
                FixAcc t;
                t.reset();
                t.add(xi, d);   // (while the gathers are in flight)
                // groups of four entries: loads first
#pragma unroll
                for (int u0 = 0; u0 < U; u0 += 4) {
                    if (u0 >= it.z) break;
                    int2 xv[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) xv[u] = x[off[u0 + u]];
#pragma unroll
                    for (int u = 0; u < 4; u++) t.add(xv[u], cf[u0 + u]);
                    if (u0 == 4 && U > 8) t.carry();
                }
                t.carry();
                const long long pr = t.lanes(lg);
                FixVals f;
                unsigned mx = 0;
#pragma unroll
                for (int j = 0; j < 5; j++) f.v[j] = 0;
                if (leads) {
                    const int2 xp = xi;
                    X = fix_row(X, pr, sl.M, sl.e);
                    xi = fix_split(X);
                    int2 *yp = ring + b1 + i;
                    *yp = xi;
                    const unsigned ya = (unsigned)__cvta_generic_to_shared(yp);
#pragma unroll
                    for (int p = 0; p < kFixMaxCtas - 1; p++)
                        if (p < C - 1)
                            asm volatile("st.shared::cluster.v2.s32 [%0], {%1, %2};" ::"r"(ya + win[p]), "r"(xi.x), "r"(xi.y)
                                         : "memory");
                    f = fix_vals_row(X, xi, xp);
                    mx = (unsigned)abs(xi.x);
                }
                __syncwarp();
                mx = __reduce_max_sync(0xffffffffu, mx);
                long long v = fix_warp_vals(f, lane);
                if (grp == 6) v = (long long)mx;
                const unsigned po = ((s + 1) & 1) ? pstep : 0u;
                if (acc0) asm volatile("st.shared::cluster.s64 [%0], %1;" ::"r"(acc0 + po), "l"(v) : "memory");
                if (acc1) asm volatile("st.shared::cluster.s64 [%0], %1;" ::"r"(acc1 + po), "l"(v) : "memory");
                __syncwarp();
            }
            fix_barrier(C);
            b0 = b1;
            b1 = b1 == 2 * nr ? 0 : b1 + nr;
        }
    }
    __syncthreads();
    if (rank == 0) fix_write(a, ring, nr, s_res);
}

// ------------------------------------------------------------------ host side
bool fix_reciprocal(double g, unsigned long long *ginv, int *ge) {
    if (!(g > 0.0) || !std::isfinite(g)) return false;
    int ex;
    const double m = frexp(g, &ex);   // g = m 2^ex, m in [0.5, 1)
    const unsigned long long G = (unsigned long long)ldexp(m, 64);
    *ge = ex - 64;                    // g = G 2^ge, G in [2^63, 2^64)
    const unsigned __int128 inv = ((unsigned __int128)1 << 127) / G;
    *ginv = inv >> 64 ? ~0ull : (unsigned long long)inv;
    return true;
}

bool fix_may_hold(int n, long long nnz) { return n >= 2 && n <= kFixMaxN && nnz <= (1 << 20); }

// CTAs of a level: one per kFixCtaWork of its work (an entry counts 1, a row 8),
// at least what its entries need of shared memory.  (1,500 and 6,000 give the same
// times; 12,000, fewer CTAs than a large level's eight, 3.9 us per sweep against 3.4
// on 4,096 rows and 16K entries and 3.7 against 3.2 on 3,048 rows and 44K entries.)
constexpr int kFixCtaWork = 3000;

static const void *fix_kernel(const FixPlan &F) {
    if (!F.by_warp) return (const void *)k_power_fix;
    return F.by_warp > 8 ? (const void *)k_power_fix_reg<16> : (const void *)k_power_fix_reg<8>;
}

static size_t fix_smem(int n, int threads, int res_i, int res_e, int res_r) {
    const size_t nr = (size_t)((n + 1) & ~1);
    return 16 * (size_t)res_i + 8 * (3 * nr + (size_t)res_e + (size_t)res_r + kFixSums * (size_t)(threads - 32)) +
           2 * (size_t)res_e + 16;
}

cmg_status_t build_fix_plans(std::vector<FixLevel> &lv, cudaStream_t s) {
    Scratch scr(s);
    SmallJobs jobs = {};
    std::vector<int> who;
    DeviceInfo di;
    CMG_TRY(device_info(&di));
    cudaFuncAttributes fa;
    CMG_CUDA(cudaFuncGetAttributes(&fa, (const void *)k_power_fix));
    const long long room = (long long)di.max_smem_optin - (long long)fa.sharedSizeBytes - 1024;
    for (size_t q = 0; q < lv.size(); q++) {
        FixLevel &L = lv[q];
        L.ok = 0;
        if (!fix_may_hold(L.n, L.nnz) || who.size() == kSmallJobs) continue;
        const long long work = L.nnz + 8ll * L.n;
        SmallJob J = {};
        J.n = L.n;
        // shared memory: ring and items, then about 13 bytes per entry (padding)
        const long long per_cta = room - 24ll * L.n - (56 << 10);
        if (per_cta <= 0) continue;
        const long long need = (13ll * L.nnz + per_cta - 1) / per_cta;
        const long long C = std::max(need, (work + kFixCtaWork - 1) / kFixCtaWork);
        if (need > L.max_ctas) continue;
        J.C = (int)std::min<long long>(std::max<long long>(1, C), L.max_ctas);
        const long long share = work / J.C;
        J.S = share <= 4096 ? 8 : (share <= 12288 ? 16 : 32);
        J.cap_items = (int)(L.n / 32 + L.nnz / 64 + 8);
        J.one_cta = kFixWarps;
        J.cap_warps = kFixWarps * L.max_ctas;
        J.rp = L.rp;
        J.col = L.col;
        J.w = L.w;
        if (!fix_reciprocal(L.g, &J.ginv, &J.ge)) continue;
        // items, range and perm in one allocation, the entries (exact) in another
        auto al = [](size_t x) { return (x + 15) & ~(size_t)15; };
        const size_t o1 = 16 * ((size_t)J.cap_items + 1), o2 = o1 + al(4 * ((size_t)J.C + 1)), o3 = o2 + al(4 * (size_t)L.n);
        FixPlan &F = L.plan;
        CMG_TRY(dev_alloc(&F.arena, o3, s));
        char *base = (char *)F.arena;
        F.C = J.C;
        J.item = F.item = (int4 *)base;
        J.range = F.range = (int *)(base + o1);
        J.perm = F.perm = (int *)(base + o2);
        CMG_TRY(scr.get(&J.inv, (size_t)L.n));
        F.bytes = o3;
        jobs.j[who.size()] = J;
        who.push_back((int)q);
    }
    const int count = (int)who.size();
    if (count == 0) return CMG_OK;
    PlanOut *out_dev;
    CMG_TRY(scr.get(&out_dev, (size_t)count));
    for (int k = 0; k < count; k++) jobs.j[k].out = out_dev + k;
    std::vector<PlanOut> out(count);
    CMG_TRY(launch_plan_small(jobs, count, s));
    CMG_CUDA(cudaMemcpyAsync(out.data(), out_dev, sizeof(PlanOut) * (size_t)count, cudaMemcpyDeviceToHost, s));
    CMG_CUDA(cudaStreamSynchronize(s));
    for (int k = 0; k < count; k++) {
        FixLevel &L = lv[who[k]];
        FixPlan &F = L.plan;
        F.res_e = out[k].max_e;
        F.res_i = out[k].max_i;
        F.res_r = out[k].max_r;
        F.ni = out[k].ni;
        F.by_warp = out[k].by_warp;
        bool fits = out[k].maxdeg == 0;
        if (F.by_warp) {
            // one CTA up to kFixWarps items, else about 8 warps per CTA: the warps
            // of one scheduler issue one after the other
            F.C = F.ni <= kFixWarps ? 1 : std::min(L.max_ctas, (F.ni + 7) / 8);
            const int per = std::max((F.ni + F.C - 1) / F.C, 1);
            F.threads = 32 * std::max(1 + per, std::min(kFixWarps + 1, (L.n / 16 + 31) / 32));
            F.smem = 24 * (size_t)((L.n + 1) & ~1) + 16 * (size_t)F.C * (F.threads / 32 - 1) * kFixSums + 16;
        } else {
            // one item per row warp where 31 warps hold them; enough threads that
            // no lane starts with more than 16 rows
            const int warps = std::max({1 + kFixSums, 1 + std::min(31, F.res_i), (L.n / 16 + 31) / 32});
            F.threads = 32 * std::min(32, warps);
            F.smem = fix_smem(L.n, F.threads, F.res_i, F.res_e, F.res_r);
            // a lane's sums take at most 8 rows
            fits = fits && F.res_i <= 8 * (F.threads / 32 - 1);
        }
        fits = fits && (long long)F.smem <= room;
        const void *kern = fix_kernel(F);
        CMG_TRY(allow_max_dynamic_smem(kern));
        if (fits && F.C > 1) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = (unsigned)F.C;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3((unsigned)F.C);
            cfg.blockDim = dim3((unsigned)F.threads);
            cfg.dynamicSmemBytes = F.smem;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int ncl = 0;
            if (cudaOccupancyMaxActiveClusters(&ncl, kern, &cfg) != cudaSuccess || ncl < 1) {
                cudaGetLastError();
                continue;
            }
        }
        if (!fits) continue;
        // exact entries, filled below
        const size_t ne = (size_t)std::max<long long>(out[k].entries, 1), o1 = 8 * ne, o2 = o1 + 8 * (size_t)L.n;
        CMG_TRY(dev_alloc(&F.entries, o2 + 2 * ne, s));
        jobs.j[k].uc = F.uc = (int2 *)F.entries;
        jobs.j[k].ud = F.ud = (int2 *)((char *)F.entries + o1);
        jobs.j[k].ucol = F.ucol = (uint16_t *)((char *)F.entries + o2);
        jobs.j[k].ni = F.ni;
        F.bytes += o2 + 2 * ne;
        L.ok = 1;
    }
    // (a level that does not fit keeps ni = 0 items to fill)
    return launch_fill_small(jobs, count, s);
}

void free_fix_plan(FixPlan &F, cudaStream_t s) {
    dev_free(F.arena, s);
    dev_free(F.entries, s);
    F = FixPlan();
}

cmg_status_t launch_power_fix(const FixPlan &F, PiArgs &a, cudaStream_t s) {
    a.items = F.item;
    a.item_range = F.range;
    a.perm = F.perm;
    a.lay_col = F.ucol;
    a.lay_w = F.uc;
    a.fix_d = F.ud;
    a.res_entries = F.res_e;
    a.res_items = F.res_i;
    a.res_rows = F.res_r;
    void *args[] = {&a};
    a.nitems = F.ni;
    const void *kern = fix_kernel(F);
    CMG_TRY(allow_max_dynamic_smem(kern));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)F.C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)F.C);
    cfg.blockDim = dim3((unsigned)F.threads);
    cfg.dynamicSmemBytes = F.smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    CMG_CUDA(cudaLaunchKernelExC(&cfg, kern, args));
    return launch_status();
}

}  // namespace cmg
