// refine.cu -- power iteration (Alg. 3 of arXiv 1412.0565), the final vector,
// its sign, and the Rayleigh quotient / residual of Sec. 4.
//
// Alg. 3 iterates u <- B_g v / ||B_g v|| with B_g = g I - L, after one
// Gram-Schmidt step against 1, and stops when cos(u^k, u^{k-1}) >= 1 - tol.
// Here the iterate is kept unnormalised, y_s = sigma_{s-1} (B_g y_{s-1} -
// g m_{s-1} 1), with sigma = 2^e / g (an exact power-of-two rescale keeps
// ||y|| near 1) and m an estimate of the mean of y_{s-1}, so that u_s is
// (y_s - mean(y_s)) / ||y_s - mean(y_s)||: the same vector as Alg. 3's in exact
// arithmetic, since 1 is an eigenvector of B_g.  Each sweep accumulates
//     A_s = sum y_s,  B_s = sum y_s^2,  C_s = sum y_s y_{s-1}
// from which mean, norm and the stopping cosine follow:
//     mu_s = A_s / n,  ss_s = B_s - n mu_s^2,
//     cos_s = (C_s - n mu_s mu_{s-1}) / sqrt(ss_s ss_{s-1}).
// Those sums are reduced by a dedicated control warp while the other warps
// compute the next sweep, so no reduction is on the critical path: the stop
// decision for sweep s is taken during sweep s+1 (whose result is then
// discarded; the iterates live in a ring of three buffers), and the mean
// estimate for sweep s+2 is m_{s+1} = 2^{e_s} (mu_s - m_s), the propagated
// 1-component of y_s, which keeps that component at rounding level.
//
// Sums and scalars are float-float (ffloat.cuh) on the FP32 pipe; FP64 is
// used where the FP64 form computes its sweeps, and for the final scalars.
//
// Kernels here (fixed.cu and resident.cu hold the others):
//   k_power_tiled  large levels: cooperative persistent kernel, one grid
//                  barrier per sweep.  Rows are cut into tiles (at most
//                  kTileRows rows, about kChunk entries); a tile's column
//                  indices and weights stream in with coalesced loads, all
//                  its x gathers are issued at once, and per-row sums run left
//                  to right in shared memory.
//   k_power_small  small levels: one CTA holds the CSR and the iterate ring in
//                  shared memory; one __syncthreads per sweep.
#include <algorithm>
#include <functional>
#include <math.h>

#include "pi_kernels.cuh"

namespace cmg {

#ifdef CMG_TRACE
// cycle stamps of the phases of the two-phase kernel's third sweep, per CTA
// and pass: [b][t][0] pass top, [2] phase 1 done, [3] after the barrier,
// [5] the last dest block's list summed, [6] its rows completed
__device__ long long g_x2t[160][32][8];
#define X2T(s, t, k) do { if ((s) == 2 && (t) < 32 && threadIdx.x == 32 && blockIdx.x < 160) g_x2t[blockIdx.x][(t)][(k)] = clock64(); } while (0)
extern "C" int cmg_debug_x2_trace(long long *host, int count) {
    return (int)cudaMemcpyFromSymbol(host, g_x2t, sizeof(long long) * (size_t)count);
}
#else
#define X2T(s, t, k) do { } while (0)
#endif

constexpr int kTileThreads = 512;                 // warp 0: control, 15 row warps
constexpr int kStageThreads = 1024;               // slice kernel with a staged iterate
#ifndef CMG_OCT32
#define CMG_OCT32 2
#endif
constexpr int kOct32 = CMG_OCT32;                 // FP32 heavy rows: octets per lane per round trip
constexpr int kRowThreads = kTileThreads - 32;
constexpr int kU = 8;                             // entries per row thread per chunk
constexpr int kChunk = kRowThreads * kU;          // 3840 entries
constexpr int kTileRows = 960;
constexpr int kTileCost = 3840;                   // entries + 4 * rows per tile
constexpr int kSmallMaxThreads = 1024;
constexpr int kFinThreads = 256;

// ================================================================== tiled kernel
template <typename T>
struct TileSmem;
// FP32: products; FP64: weights and gathered x (the row sum is an FMA chain)
template <>
struct TileSmem<float> {
    float prod[kChunk];
};
template <>
struct TileSmem<double> {
    double wv[kChunk];
    double xj[kChunk];
};

template <typename T>
__global__ void __launch_bounds__(kTileThreads, 2) k_power_tiled(PiArgs a, GridSync *gs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TileSmem<T> &ts = *reinterpret_cast<TileSmem<T> *>(smem_raw);
    T *s_x = reinterpret_cast<T *>(smem_raw + sizeof(TileSmem<T>));     // kTileRows
    T *s_acc = s_x + kTileRows;                                         // kTileRows
    int *s_rp = reinterpret_cast<int *>(s_acc + kTileRows);             // kTileRows + 1
    unsigned short *s_row = reinterpret_cast<unsigned short *>(s_rp + kTileRows + 4);  // kChunk
    __shared__ Part s_pw[kTileThreads / 32];
    __shared__ Slot s_slot[2];
    __shared__ GridBar s_bar;
    if (threadIdx.x == 0) grid_bar_init(&s_bar, gs);

    const int n = a.n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tb = (int)((long long)a.ntiles * blockIdx.x / gridDim.x);
    const int te = (int)((long long)a.ntiles * (blockIdx.x + 1) / gridDim.x);
    const int r0 = a.tile_row[tb], r1 = a.tile_row[te];
    T *const ring0 = (T *)a.buf[0], *const ring1 = (T *)a.buf[1], *const ring2 = (T *)a.buf[2];
    const T *__restrict__ wv = wsel<T>(a);
    const bool fp64 = sizeof(T) == 8;
    const T g = (T)a.g;
    const float inv_gf = 1.0f / (float)a.g;
    const double inv_gd = 1.0 / a.g;

    // ---------------------------------------------------------- start phase
    // y_0 (and g - d_i for the FP64 form); then one blocking reduction.
    {
        const void *cb = nullptr;
        double cmu = 0.0, cinv = 0.0;
        if (a.start == 1) {
            cb = a.cbuf[a.cres->buf];
            cmu = a.cres->mu;
            cinv = a.cres->inv_s;
        }
        // start sums: A = sum y_0 (not small after a prolongation), B = sum y_0^2
        Part acc = part_zero();
        for (int i = r0 + tid; i < r1; i += blockDim.x) {
            const T xt = (T)start_value(a, i, cb, cmu, cinv);
            ring0[i] = xt;
            if (fp64) {
                double d = 0.0;
                for (int e = __ldg(a.rp + i), e1 = __ldg(a.rp + i + 1); e < e1; e++) d += __ldg(a.w + e);
                a.gd[i] = a.g - d;
            }
            const ff v = fp64 ? ff_from_double((double)xt) : ff_make((float)xt, 0.f);
            acc.A = ff_add(acc.A, v);
            acc.B = ff_add(acc.B, ff_mul(v, v));
        }
        Part p = warp_sum_part(acc);
        if (lane == 0) s_pw[warp] = p;
        __syncthreads();
        if (warp == 0) {
            Part q = (lane < (int)(blockDim.x >> 5)) ? s_pw[lane] : part_zero();
            q = warp_sum_part(q);
            if (lane == 0) {
                store_part(a.partials + blockIdx.x, q);
            }
        }
    }
    if (!grid_sync(&s_bar)) return;
    __shared__ Ctl c;   // used by lane 0 of the control warp (in registers it would take every row thread's)
    if (warp == 0) {
        const Part q = grid_part(a.partials, lane);
        const double mu0 = to_d(q.A) / (double)n;
        double ss0 = to_d(q.B) - (double)n * mu0 * mu0;
        if (ss0 < 0.0) ss0 = 0.0;
        const int e0 = start_exponent(ss0);
        if (lane == 0) {
            ctl_init(c, a, mu0, ss0, e0);
            s_slot[1] = slot_make(ff_from_double(mu0), e0, a.g, c.inv_g, fp64);  // sweep 1: exact mean of y_0
            s_slot[0] = slot_make(ff_zero(), 0, a.g, c.inv_g, fp64);             // sweep 2: m_1 = 0
        }
    }
    __syncthreads();

    const bool no_sweeps = (a.mode == 1 && a.k_fixed <= 0);
    int s = 0;
    int exit_kind = no_sweeps ? 2 : 0;   // 1: decided stop, 2: count exit
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
            // ---- control: reduce sweep s over all CTAs, decide, plan sweep s+2
            if (s >= 1) {
                const Part q = grid_part(a.partials + (size_t)(s & 1) * gridDim.x, lane);
                if (lane == 0) ctrl_step(a, s, q, c, &s_slot[s & 1], false, fp64);
            }
        } else {
            // ---- rows of sweep s+1
            const int rt = tid - 32;
            const T m = fp64 ? (T)sl.m_d : (T)sl.m.hi;
            const T sig = fp64 ? (T)sl.sig_d : (T)scale2f(inv_gf, sl.e);
            const T gm = fp64 ? (T)sl.gm_d : g * m;
            Acc<T> acc;
            acc.reset();
            for (int t = tb; t < te; t++) {
                const int t0 = a.tile_row[t], t1 = a.tile_row[t + 1];
                const int nr = t1 - t0;
                if (nr <= 0) continue;
                const int e0 = __ldg(a.rp + t0);
                const int ne = __ldg(a.rp + t1) - e0;
                for (int k = rt; k < nr; k += kRowThreads) {
                    s_rp[k] = __ldg(a.rp + t0 + k) - e0;
                    s_x[k] = LDXG(x + t0 + k);
                    s_acc[k] = (T)0;
                }
                if (rt == 0) s_rp[nr] = ne;
                bar_rows(kRowThreads);
                for (int c0 = 0; c0 < ne; c0 += kChunk) {
                    const int cn = min(kChunk, ne - c0);
                    if (!fp64) {
                        for (int r = rt; r < nr; r += kRowThreads) {
                            const int lo = max(s_rp[r], c0), hi = min(s_rp[r + 1], c0 + cn);
                            for (int q = lo; q < hi; q++) s_row[q - c0] = (unsigned short)r;
                        }
                        bar_rows(kRowThreads);
                    }
                    int jj[kU];
                    T ww[kU], xj[kU];
#pragma unroll
                    for (int u = 0; u < kU; u++) {
                        const int k = rt + u * kRowThreads;
                        jj[u] = 0;
                        ww[u] = (T)0;
                        if (k < cn) {
                            jj[u] = __ldg(a.col + e0 + c0 + k);
                            ww[u] = __ldg(wv + e0 + c0 + k);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kU; u++) {
                        const int k = rt + u * kRowThreads;
                        xj[u] = (T)0;
                        if (k < cn) xj[u] = LDXG(x + jj[u]);
                    }
                    if (fp64) {
                        double *swv = reinterpret_cast<double *>(&ts);
                        double *sxj = swv + kChunk;
#pragma unroll
                        for (int u = 0; u < kU; u++) {
                            const int k = rt + u * kRowThreads;
                            if (k < cn) {
                                swv[k] = (double)ww[u];
                                sxj[k] = (double)xj[u];
                            }
                        }
                    } else {
                        float *sp = reinterpret_cast<float *>(&ts);
#pragma unroll
                        for (int u = 0; u < kU; u++) {
                            const int k = rt + u * kRowThreads;
                            if (k < cn) sp[k] = (float)ww[u] * ((float)s_x[s_row[k]] - (float)xj[u]);
                        }
                    }
                    bar_rows(kRowThreads);
                    for (int r = rt; r < nr; r += kRowThreads) {
                        const int lo = max(s_rp[r], c0), hi = min(s_rp[r + 1], c0 + cn);
                        T ac = s_acc[r];
                        if (fp64) {
                            const double *swv = reinterpret_cast<const double *>(&ts);
                            const double *sxj = swv + kChunk;
                            for (int q = lo; q < hi; q++) ac = fma((double)swv[q - c0], (double)sxj[q - c0], (double)ac);
                        } else {
                            const float *sp = reinterpret_cast<const float *>(&ts);
                            for (int q = lo; q < hi; q++) ac += (T)sp[q - c0];
                        }
                        s_acc[r] = ac;
                    }
                    bar_rows(kRowThreads);
                }
                for (int r = rt; r < nr; r += kRowThreads) {
                    const T xi = s_x[r];
                    T yv;
                    if (fp64) yv = (T)((fma(a.gd[t0 + r], (double)xi, (double)s_acc[r]) - (double)gm) * (double)sig);
                    else yv = (g * (xi - m) - s_acc[r]) * sig;
                    y[t0 + r] = yv;
                    acc.add(yv, xi);
                }
                bar_rows(kRowThreads);
            }
            Part p = warp_sum_part(acc.get());
            if (lane == 0) s_pw[warp] = p;
        }
        __syncthreads();
        if (warp == 0) {
            Part q = (lane >= 1 && lane < (int)(blockDim.x >> 5)) ? s_pw[lane] : part_zero();
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
            // the last sweep s ended the loop by count: reduce it now
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

// First entry and length (a multiple of 8) of chunk cidx of the heavy rows: a row
// of len entries is cut into nc chunks of equal length rounded up to octets.
__device__ __forceinline__ void sell_chunk(const PiArgs &a, const int *M, int cidx, int *f0, int *len) {
    const int r = a.crow[cidx], c0 = a.hchunk[r], nc = a.hchunk[r + 1] - c0;
    const int m0 = M[r], m1 = M[r + 1];
    const int per = (((m1 - m0 + nc - 1) / nc) + 7) & ~7;
    *f0 = min(m1, m0 + (cidx - c0) * per);
    *len = min(m1, *f0 + per) - *f0;
}

// First slice of CTA b of nb: slices starting at b / nb of the slice entries.
__device__ __forceinline__ int sell_first_slice(const int *SO, int nsl, int b, int nb) {
    if (b >= nb) return nsl;
    const long long target = SO[0] + ((long long)SO[nsl] - SO[0]) * b / nb;
    int lo = 0, hi = nsl;   // first slice starting at or after the target
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (SO[mid] < target) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// ================================================================== slice kernel
// Large levels with a sweep layout (rows renumbered by decreasing degree;
// heavy rows in CSR form, the rest in 32-row slices with interleaved entries):
// cooperative persistent kernel with the control warp of k_power_tiled.  A
// row warp takes a chunk of a heavy row (32 lanes over its octets) or a slice
// (one lane per row; entry k of the slice's rows is one coalesced load), so
// the loads of a sweep do not wait on one another and no CTA barrier is
// needed inside a sweep.  The iterates are stored in layout order.
//
// STAGE: one 1024-thread CTA per SM; at the top of each sweep the row warps
// copy the iterate's first stage_n entries (the highest-degree rows, which
// take the largest share of the gathers) into shared memory and gather from
// there.  A gather of 32 scattered words from L1 or L2 costs about one cycle
// per distinct line; from shared memory it costs the bank conflicts, a few
// cycles per 32 words.
//
// RES (FP32 levels that stage their whole iterate and whose layout fits beside it in
// the SMs' shared memory): the CTA copies its chunks and slices there once and
// sweeps from there, instead of reading them from L2 every sweep.  The rows stay
// with the CTA, warp and order that they have without RES -- the stop sums then
// round the same way, and with them the mean that every FP32 sweep subtracts: a
// level's thousands of sweeps turn one other rounding there into a different
// vector at the 1e-8 level.  16K rows and 3.2M entries: 23.9 us per sweep
// without, 18.8 with.  (The two-CTA form without a staged iterate measured the
// same or slower from shared memory: 3,820 rows and 2.1M entries 14.4 and 15.0,
// 100^3 grid levels 1 and 2 16.7 and 18.4, 9.7 and 10.2: it does not take it.)
template <typename T, typename IDX, bool CHUNKS, bool STREAM, bool STAGE, bool RES>
__global__ void __launch_bounds__(STAGE ? kStageThreads : kTileThreads, STAGE ? 1 : 2)
    k_power_sell(PiArgs a, GridSync *gs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // shared memory: the staged iterate; RES: weights, columns, chunk offsets
    T *const s_x = reinterpret_cast<T *>(smem_raw);
    T *const s_w = s_x + (STAGE ? ((a.stage_n + 7) & ~7) : 0);
    IDX *const s_c = reinterpret_cast<IDX *>(s_w + (RES ? a.res_entries : 0));
    int *const s_co = reinterpret_cast<int *>(s_c + (RES ? a.res_entries : 0));
    __shared__ Part s_pw[kStageThreads / 32];
    __shared__ Slot s_slot[2];
    __shared__ GridBar s_bar;
    if (threadIdx.x == 0) grid_bar_init(&s_bar, gs);
    const int n = a.n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    T *const ring0 = (T *)a.buf[0], *const ring1 = (T *)a.buf[1], *const ring2 = (T *)a.buf[2];
    const bool fp64 = sizeof(T) == 8;
    const T g = (T)a.g;
    const float inv_gf = 1.0f / (float)a.g;
    const double inv_gd = 1.0 / a.g;
    const int h = a.lay_h, nsl = a.lay_nsl;
    const int *__restrict__ M = a.lay_meta;
    const int *__restrict__ SO = M + h;
    const IDX *__restrict__ C = reinterpret_cast<const IDX *>(a.lay_col);
    const T *__restrict__ W = reinterpret_cast<const T *>(a.lay_w);
    // work of this CTA: a contiguous range of slices holding about 1/gridDim
    // of the slice entries (the slices are sorted by width, so equal slice
    // counts would not balance); heavy rows go round robin over all warps
    __shared__ int s_range[2];
    if (threadIdx.x < 2)
        s_range[threadIdx.x] = sell_first_slice(SO, nsl, (int)blockIdx.x + (int)threadIdx.x, (int)gridDim.x);
    __syncthreads();
    const int sb = s_range[0], se = s_range[1];
    const int r0 = (int)((long long)n * blockIdx.x / gridDim.x);
    const int r1 = (int)((long long)n * (blockIdx.x + 1) / gridDim.x);
    int sl_off = 0;   // RES: shared-memory entry of slice entry e is e + sl_off
    if (RES) {
        // this CTA's chunks (chunk b + grid j is the j-th), then its slices
        const int nj = CHUNKS && (int)blockIdx.x < a.nchunks ? (a.nchunks - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
        if (warp == 0) {
            int carry = 0;
            for (int j0 = 0; j0 < nj; j0 += 32) {
                int f0 = 0, len = 0;
                if (j0 + lane < nj) sell_chunk(a, M, (int)(blockIdx.x + gridDim.x * (j0 + lane)), &f0, &len);
                int incl = len;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                if (j0 + lane < nj) s_co[j0 + lane] = carry + incl - len;
                carry += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) s_co[nj] = carry;
        }
        __syncthreads();
        for (int j = warp; j < nj; j += (int)(blockDim.x >> 5)) {
            int f0, len;
            sell_chunk(a, M, (int)(blockIdx.x + gridDim.x * j), &f0, &len);
            const int d = s_co[j];
            for (int k = lane; k < len; k += 32) {
                s_w[d + k] = W[f0 + k];
                s_c[d + k] = C[f0 + k];
            }
        }
        sl_off = s_co[nj] - (sb < se ? SO[sb] : 0);
        for (int k = (sb < se ? SO[sb] : 0) + tid; k < (sb < se ? SO[se] : 0); k += blockDim.x) {
            s_w[k + sl_off] = W[k];
            s_c[k + sl_off] = C[k];
        }
    }

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
                a.gd[p] = a.g - d;
            }
            const ff v = fp64 ? ff_from_double((double)xt) : ff_make((float)xt, 0.f);
            acc.A = ff_add(acc.A, v);
            acc.B = ff_add(acc.B, ff_mul(v, v));
        }
        Part p = warp_sum_part(acc);
        if (lane == 0) s_pw[warp] = p;
        __syncthreads();
        if (warp == 0) {
            Part q = (lane < (int)(blockDim.x >> 5)) ? s_pw[lane] : part_zero();
            q = warp_sum_part(q);
            if (lane == 0) {
                store_part(a.partials + blockIdx.x, q);
            }
        }
    }
    if (!grid_sync(&s_bar)) return;
    __shared__ Ctl c;   // used by lane 0 of the control warp (in registers it would take every row thread's)
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
    const int rw = warp - 1, nrw = (int)(blockDim.x >> 5) - 1;            // row warps of this CTA
    // heavy-row chunks are dealt CTA by CTA (chunk k to CTA k mod grid), so
    // a level with few chunks still spreads them over all SMs
    const int gw = rw * (int)gridDim.x + blockIdx.x, ngw = (int)gridDim.x * nrw;
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
            auto finish = [&](int i, T xi, T ac) {
                T yv;
                if (fp64) yv = (T)((fma(a.gd[i], (double)xi, (double)ac) - (double)gm) * (double)sig);
                else yv = (g * (xi - m) - ac) * sig;
                y[i] = yv;
                acc.add(yv, xi);
            };
            const int S = STAGE ? a.stage_n : 0;
            if (STAGE) {
                // 16-byte copies of x[0, S) into shared memory, then the row
                // warps meet (the control warp does not take part)
                const int nrt = (int)blockDim.x - 32;
                const int nv = ((reinterpret_cast<uintptr_t>(x) & 15) == 0) ? (int)(((long long)S * sizeof(T)) / 16) : 0;
                const float4 *src = reinterpret_cast<const float4 *>(x);
                float4 *dst = reinterpret_cast<float4 *>(s_x);
                for (int k = tid - 32; k < nv; k += nrt) dst[k] = __ldcg(src + k);
                for (int k = nv * (16 / (int)sizeof(T)) + tid - 32; k < S; k += nrt) s_x[k] = __ldcg(x + k);
                bar_rows(nrt);
            }
            auto ldx = [&](int c) { return (STAGE && c < S) ? s_x[c] : LDXG(x + c); };
            // heavy rows: a row of len entries (a multiple of 8) is cut into
            // nc = ceil(len / kHeavyChunk) chunks of equal length rounded up
            // to whole octets, a warp per chunk, lanes taking octets; the
            // warp of a row's last chunk waits for the row's other chunks,
            // sums the chunk partials in chunk order and completes the row
            const bool vec = ((reinterpret_cast<uintptr_t>(C) | reinterpret_cast<uintptr_t>(W)) & 15) == 0;
            for (int cidx = gw, j = rw; CHUNKS && cidx < a.nchunks; cidx += ngw, j += nrw) {
                const int r = a.crow[cidx], c0 = a.hchunk[r], nc = a.hchunk[r + 1] - c0;
                int f0, flen;
                sell_chunk(a, M, cidx, &f0, &flen);
                const T xi = ldx(r);
                T ac;
                if (RES) {
                    const int d = s_co[j] >> 3;
                    ac = row_sum_octets<T, IDX, sizeof(T) == 4 ? kOct32 : 1>(s_c, s_w, d + lane, d + (flen >> 3), xi, ldx,
                                                                             false);
                } else {
                    const int f1 = f0 + flen;
                    ac = vec ? row_sum_octets<T, IDX, sizeof(T) == 4 ? kOct32 : 1>(C, W, (f0 >> 3) + lane, f1 >> 3, xi,
                                                                                  ldx, STREAM)
                             : row_sum_grouped<T, IDX>(C, W, f0 + lane, f1, 32, xi, ldx, STREAM);
                }
                ac = warp_sum(ac);
                if (nc == 1) {
                    if (lane == 0) finish(r, xi, ac);
                } else if (lane == 0) {
                    // the warp of the row's last chunk completes the row (a
                    // fixed thread, so the sweep's partial sums group the
                    // same way in every run); the others publish their partial
                    T *cp = reinterpret_cast<T *>(a.cpart);
                    unsigned int *cnt = reinterpret_cast<unsigned int *>(a.hcount + r);
                    if (cidx < c0 + nc - 1) {
                        cp[cidx] = ac;
                        red_add_release_gpu(cnt, 1u);
                    } else {
                        // the other chunks have lower indices: their warps
                        // never wait on this one, so the wait ends; bounded
                        // all the same (GridSync::err, like a barrier)
                        const unsigned int want = (unsigned int)((s + 1) * (nc - 1));
                        unsigned long long t0 = 0;
                        for (unsigned int spin = 0; ld_acquire_gpu(cnt) < want; spin++) {
                            if ((spin & 255u) == 255u) {
                                const unsigned long long t = global_ns();
                                if (t0 == 0) {
                                    t0 = t;
                                } else if (t - t0 > kBarrierTimeoutNs || ld_relaxed_gpu(&gs->err)) {
                                    atomicExch(&gs->err, 1u);
                                    s_bar.err = 1;   // the CTA leaves at its next barrier
                                    break;
                                }
                            }
                        }
                        T tot = (T)0;
                        for (int c = c0; c < c0 + nc - 1; c++) tot += __ldcg(cp + c);
                        finish(r, xi, tot + ac);
                    }
                }
                __syncwarp();
            }
            // slices: a lane per row, entries in groups of 8 (row_sum_grouped)
            for (int q = sb + rw; q < se; q += nrw) {
                const int i = h + 32 * q + lane;
                const int so = SO[q] + lane, wd = (SO[q + 1] - SO[q]) >> 5;
                const T xi = (i < n) ? ldx(i) : (T)0;
                const T ac = RES ? row_sum_grouped<T, IDX>(s_c, s_w, so + sl_off, so + sl_off + 32 * wd, 32, xi, ldx, false)
                                 : row_sum_grouped<T, IDX>(C, W, so, so + 32 * wd, 32, xi, ldx, STREAM);
                if (i < n) finish(i, xi, ac);
            }
            Part p = warp_sum_part(acc.get());
            if (lane == 0) s_pw[warp] = p;
        }
        __syncthreads();
        if (warp == 0) {
            Part q = (lane >= 1 && lane < (int)(blockDim.x >> 5)) ? s_pw[lane] : part_zero();
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

// ================================================================== two-phase kernel
// Sweeps of a level with a two-phase layout (XLayout, internal.h): one
// 1024-thread CTA per SM (grid = the layout's P), warp 0 the control warp,
// warps 1..31 the row warps.  Per pass: phase 1 (source blocks staged in
// shared memory, xbuf written in list order), a grid barrier, phase 2 (the
// CTA's dest blocks: terms added into 64-bit fixed-point row accumulators in
// shared memory, then the rows completed).  The two xbufs alternate between
// passes, so phase 1 of pass t+1 follows phase 2 of pass t without a
// barrier: the buffer it overwrites was last read in pass t-1, which every
// CTA finished before the barrier of pass t.
//
// Fixed point: a sweep's terms are w x_c (FP64 form) or w (x_r - x_c) (FP32
// form), so every partial sum of a row is at most g max|x| in magnitude (g
// is twice the largest weighted degree).  With sc = 61 - e, g max|x| < 2^e,
// the terms scaled by 2^sc and rounded to integers sum in int64 without
// overflow; integer addition is associative, so the sum does not depend on
// the order of the shared-memory atomics.  max|x| of the sweep's iterate is
// the exact maximum of the previous sweep's per-CTA maxima.
constexpr int kXRows = kStageThreads / 32 - 1;   // row warps

// round(v 2^sc) for a double, by integer arithmetic (round half away from
// zero; values below 2^-sc / 2 and subnormals give 0): the FP64 pipe is
// left to the product that forms v
__device__ __forceinline__ long long fix64(double v, int sc) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int ef = (int)((b >> 52) & 0x7ffu);
    if (ef == 0) return 0;
    const long long mant = (long long)((b & 0xfffffffffffffull) | 0x10000000000000ull);
    const int sh = ef - 1075 + sc;   // v 2^sc = mant 2^sh; sh <= 8 by the choice of sc
    long long r;
    if (sh >= 0) r = mant << min(sh, 10);
    else if (sh > -64) r = (mant + (1ll << (-sh - 1))) >> (-sh);
    else r = 0;
    return (b >> 63) ? -r : r;
}

__device__ __forceinline__ long long fix_term(float v, int sc, float scf) { return __float2ll_rn(v * scf); }
__device__ __forceinline__ long long fix_term(double v, int sc, float) { return fix64(v, sc); }

__device__ __forceinline__ int fix_scale(double g, double xmax) {
    if (!(xmax > 0.0)) return 0;
    int ex;
    frexp(g * xmax, &ex);   // g xmax < 2^ex
    return max(-120, min(120, 61 - ex));
}

template <typename T>
__global__ void __launch_bounds__(kStageThreads, 1) k_power_2p(PiArgs a, GridSync *gs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *const sm = reinterpret_cast<T *>(smem_raw);
    __shared__ Part s_pw[kStageThreads / 32];
    __shared__ double s_mx[kStageThreads / 32];
    __shared__ Slot s_slot[2];
    __shared__ GridBar s_bar;
    if (threadIdx.x == 0) grid_bar_init(&s_bar, gs);
    __shared__ int s_sc;
    __shared__ Ctl s_ctl;   // the control warp's state (kept out of every thread's registers)
    const int n = a.n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rt = tid - 32, nrt = (int)blockDim.x - 32, rw = warp - 1;   // row threads and warps
    T *const ring0 = (T *)a.buf[0], *const ring1 = (T *)a.buf[1], *const ring2 = (T *)a.buf[2];
    const bool fp64 = sizeof(T) == 8;
    const T g = (T)a.g;
    const float inv_gf = 1.0f / (float)a.g;
    const int P = (int)gridDim.x, b = (int)blockIdx.x;
    const int r0 = (int)((long long)n * b / P), r1 = (int)((long long)n * (b + 1) / P);
    const T *__restrict__ XW = reinterpret_cast<const T *>(a.x_w);
    auto cta_max = [&](double v, double *dst) {   // max over the CTA into *dst (thread 0 writes)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (lane == 0) s_mx[warp] = v;
        __syncthreads();
        if (warp == 0) {
            double u = lane < (int)(blockDim.x >> 5) ? s_mx[lane] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) u = fmax(u, __shfl_xor_sync(0xffffffffu, u, o));
            if (lane == 0) *dst = u;
        }
    };
    auto grid_max = [&](const double *src) {      // warp 0: max of the P per-CTA values
        double u = 0.0;
        for (int k = lane; k < P; k += 32) u = fmax(u, __ldcg(src + k));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) u = fmax(u, __shfl_xor_sync(0xffffffffu, u, o));
        return u;
    };

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
        double mx = 0.0;
        for (int p = r0 + tid; p < r1; p += blockDim.x) {
            const int old = a.perm[p];
            const T xt = (T)start_value(a, old, cb, cmu, cinv);
            ring0[p] = xt;
            mx = fmax(mx, fabs((double)xt));
            if (fp64) {
                double d = 0.0;
                for (int e = __ldg(a.rp + old), e1 = __ldg(a.rp + old + 1); e < e1; e++) d += __ldg(a.w + e);
                a.gd[p] = a.g - d;
            }
            const ff v = fp64 ? ff_from_double((double)xt) : ff_make((float)xt, 0.f);
            acc.A = ff_add(acc.A, v);
            acc.B = ff_add(acc.B, ff_mul(v, v));
        }
        Part p = warp_sum_part(acc);
        if (lane == 0) s_pw[warp] = p;
        cta_max(mx, a.x_pmax + b);   // its __syncthreads also publishes s_pw
        if (warp == 0) {
            Part q = (lane < (int)(blockDim.x >> 5)) ? s_pw[lane] : part_zero();
            q = warp_sum_part(q);
            if (lane == 0) {
                store_part(a.partials + blockIdx.x, q);
            }
        }
    }
    if (!grid_sync(&s_bar)) return;
    if (warp == 0) {
        Ctl c;
        const Part q = grid_part(a.partials, lane);
        const double xmax = grid_max(a.x_pmax);
        const double mu0 = to_d(q.A) / (double)n;
        double ss0 = to_d(q.B) - (double)n * mu0 * mu0;
        if (ss0 < 0.0) ss0 = 0.0;
        const int e0 = start_exponent(ss0);
        ctl_init(c, a, mu0, ss0, e0);
        if (lane == 0) {
            s_ctl = c;
            s_slot[1] = slot_make(ff_from_double(mu0), e0, a.g, c.inv_g, fp64);
            s_slot[0] = slot_make(ff_zero(), 0, a.g, c.inv_g, fp64);
            s_sc = fix_scale(a.g, xmax);
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
        if (warp == 0 && s >= 1) {
            // decisions of sweep s-1 and the fixed-point scale of sweep s,
            // overlapped with phase 1 of pass 0 (published by its barrier)
            const Part q = grid_part(a.partials + (size_t)(s & 1) * P, lane);
            Slot nx;
            Ctl c = s_ctl;
            ctrl_step(a, s, q, c, &nx, false, fp64);
            const double xmax = grid_max(a.x_pmax + (size_t)(s & 1) * P);
            __syncwarp();
            if (lane == 0) {
                s_ctl = c;
                s_slot[s & 1] = nx;
                s_sc = fix_scale(a.g, xmax);
            }
        }
        const T m = fp64 ? (T)sl.m_d : (T)sl.m.hi;
        const T sig = fp64 ? (T)sl.sig_d : (T)scale2f(inv_gf, sl.e);
        const T gm = fp64 ? (T)sl.gm_d : g * m;
        Acc<T> acc;
        acc.reset();
        T ymax = (T)0;
        auto finish = [&](int i, T xi, T ac) {
            T yv;
            if (fp64) yv = (T)((fma(a.gd[i], (double)xi, (double)ac) - (double)gm) * (double)sig);
            else yv = (g * (xi - m) - ac) * sig;
            y[i] = yv;
            acc.add(yv, xi);
            ymax = max(ymax, abs(yv));
        };
        for (int t = 0; t < a.x_T; t++) {
            // xbuf holds pass t's list positions from ps0 & ~7 on, so that 8
            // list entries at a multiple of 8 sit at a multiple of 8 there
            T *const xb = reinterpret_cast<T *>(a.x_buf[t & 1]);
            const int ps0 = __ldg(a.x_ps + t), xsh = ps0 & 7, xb0 = ps0 - xsh;
            X2T(s, t, 0);
            if (warp > 0) {
                // ------------------------------------------------ phase 1
                // this CTA's share of the pass's stream, source block by
                // source block; entry j goes to its list position, found
                // from its 32-entry chunk's cell and cell-start bits
                const long long Et = (long long)__ldg(a.x_ps + t + 1) - ps0;
                int e = (int)(Et * b / P);
                const int e1 = (int)(Et * (b + 1) / P);
                const int *qo = a.x_qoff + (size_t)t * (a.x_Q + 1);
                const uint2 *chk = a.x_chk + __ldg(a.x_choff + t);
                const uint16_t *srcp = a.x_src + __ldg(a.x_sal + t);
                int lo = 0, hi = a.x_Q - 1;   // last block q with qo[q] <= e
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (__ldg(qo + mid) <= e) lo = mid;
                    else hi = mid - 1;
                }
                for (int q = lo; e < e1; q++) {
                    const int qe = min(e1, __ldg(qo + q + 1));
                    if (qe > e) {
                        const int base = q * a.x_SB, cnt = min(a.x_SB, n - base);
                        const T *xs = x + base;
                        // 16-byte asynchronous copies (L2 only: x was written
                        // by other CTAs before the last barrier), then the tail
                        const int nv16 = ((reinterpret_cast<uintptr_t>(xs) & 15) == 0) ? (int)((cnt * sizeof(T)) / 16) : 0;
                        for (int k = rt; k < nv16; k += nrt) {
                            const unsigned dsm = (unsigned)__cvta_generic_to_shared(reinterpret_cast<char *>(sm) + 16 * (size_t)k);
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dsm),
                                         "l"(reinterpret_cast<const char *>(xs) + 16 * (size_t)k)
                                         : "memory");
                        }
                        asm volatile("cp.async.wait_all;" ::: "memory");
                        for (int k = nv16 * (int)(16 / sizeof(T)) + rt; k < cnt; k += nrt) sm[k] = __ldcg(xs + k);
                        bar_rows(nrt);
                        // 8 consecutive stream entries per row thread (one
                        // vector load of their source offsets); an entry's
                        // cell comes from its 32-entry chunk's bits
                        for (int gi = (e >> 3) + rt; 8 * gi < qe; gi += nrt) {
                            const int j0 = 8 * gi;
                            const uint4 sv = __ldcs(reinterpret_cast<const uint4 *>(srcp + j0));
                            const uint2 ci = __ldg(chk + (j0 >> 5));
                            const unsigned sw[4] = {sv.x, sv.y, sv.z, sv.w};
                            int lastc = -1, dl = 0;
#pragma unroll
                            for (int u = 0; u < 8; u++) {
                                const int j = j0 + u;
                                if (j < e || j >= qe) continue;
                                const int cell = (int)ci.x + __popc(ci.y & ((2u << (j & 31)) - 1u));
                                if (cell != lastc) {
                                    dl = __ldg(a.x_cdel + cell);
                                    lastc = cell;
                                }
                                xb[j + xsh + dl] = sm[(sw[u >> 1] >> (16 * (u & 1))) & 0xffffu];
                            }
                        }
                        bar_rows(nrt);
                    }
                    e = qe;
                }
            }
            X2T(s, t, 2);
            if (!grid_sync(&s_bar)) return;
            X2T(s, t, 3);
            if (warp > 0) {
                // ------------------------------------------------ phase 2
                const int sc = s_sc;
                const float scf = ldexpf(1.0f, sc);
                long long *const accs = reinterpret_cast<long long *>(smem_raw);
                T *const xv = reinterpret_cast<T *>(accs + a.x_VMAX);
                const int g0 = __ldg(a.x_ndb + t), g1 = __ldg(a.x_ndb + t + 1);
                for (int gb = g0 + b; gb < g1; gb += P) {
                    const int R0 = __ldg(a.x_dbr + gb), R1 = __ldg(a.x_dbr + gb + 1);
                    const int L0 = __ldg(a.x_dbl + gb), L1 = __ldg(a.x_dbl + gb + 1);
                    for (int p = R0 + rt; p < R1; p += nrt) {
                        xv[p - R0] = __ldcg(x + p);
                        accs[p - R0] = 0;
                    }
                    bar_rows(nrt);
                    // 8 consecutive list entries per lane (vector loads from
                    // a multiple of 8); a run of one row's entries is summed
                    // in a register and added to its accumulator once
                    for (int pb = (L0 & ~7) + 256 * rw; pb < L1; pb += 256 * kXRows) {
                        const int base = pb + 8 * lane;
                        if (base + 8 <= L0 || base >= L1) continue;
                        const uint4 dv = __ldcs(reinterpret_cast<const uint4 *>(a.x_dst + base));
                        const unsigned dw[4] = {dv.x, dv.y, dv.z, dv.w};
                        T wv[8], xvv[8];
                        if (fp64) {
#pragma unroll
                            for (int h = 0; h < 4; h++) {
                                const double2 w2 = __ldcs(reinterpret_cast<const double2 *>(XW + base) + h);
                                const double2 x2 = __ldcg(reinterpret_cast<const double2 *>(xb + (base - xb0)) + h);
                                wv[2 * h] = (T)w2.x;
                                wv[2 * h + 1] = (T)w2.y;
                                xvv[2 * h] = (T)x2.x;
                                xvv[2 * h + 1] = (T)x2.y;
                            }
                        } else {
#pragma unroll
                            for (int h = 0; h < 2; h++) {
                                const float4 w4 = __ldcs(reinterpret_cast<const float4 *>(XW + base) + h);
                                const float4 x4 = __ldcg(reinterpret_cast<const float4 *>(xb + (base - xb0)) + h);
                                wv[4 * h] = (T)w4.x;
                                wv[4 * h + 1] = (T)w4.y;
                                wv[4 * h + 2] = (T)w4.z;
                                wv[4 * h + 3] = (T)w4.w;
                                xvv[4 * h] = (T)x4.x;
                                xvv[4 * h + 1] = (T)x4.y;
                                xvv[4 * h + 2] = (T)x4.z;
                                xvv[4 * h + 3] = (T)x4.w;
                            }
                        }
                        int rd = -1;
                        long long ra = 0;
#pragma unroll
                        for (int k = 0; k < 8; k++) {
                            const int pos = base + k;
                            if (pos < L0 || pos >= L1) continue;
                            const int d = (int)((dw[k >> 1] >> (16 * (k & 1))) & 0xffffu);
                            const T v = fp64 ? wv[k] * xvv[k] : wv[k] * (xv[d] - xvv[k]);
                            const long long iv = fix_term(v, sc, scf);
                            if (d != rd) {
                                if (rd >= 0) atomicAdd(reinterpret_cast<unsigned long long *>(accs + rd), (unsigned long long)ra);
                                rd = d;
                                ra = iv;
                            } else {
                                ra += iv;
                            }
                        }
                        if (rd >= 0) atomicAdd(reinterpret_cast<unsigned long long *>(accs + rd), (unsigned long long)ra);
                    }
                    bar_rows(nrt);
                    X2T(s, t, 5);
                    for (int p = R0 + rt; p < R1; p += nrt) {
                        T ac;
                        if (fp64) ac = (T)((double)accs[p - R0] * ldexp(1.0, -sc));
                        else ac = (T)(__ll2float_rn(accs[p - R0]) * ldexpf(1.0f, -sc));
                        finish(p, xv[p - R0], ac);
                    }
                    bar_rows(nrt);
                }
                X2T(s, t, 6);
            }
        }
        if (warp > 0) {
            Part p = warp_sum_part(acc.get());
            if (lane == 0) s_pw[warp] = p;
        }
        cta_max((double)ymax, a.x_pmax + (size_t)((s + 1) & 1) * P + b);   // its __syncthreads publishes s_pw
        if (warp == 0) {
            Part q = (lane >= 1 && lane < (int)(blockDim.x >> 5)) ? s_pw[lane] : part_zero();
            q = warp_sum_part(q);
            if (lane == 0) {
                store_part(a.partials + (size_t)((s + 1) & 1) * P + blockIdx.x, q);
            }
        }
        if (!grid_sync(&s_bar)) return;
        s++;
    }
    // ---------------------------------------------------------- result
    if (warp == 0) {
        Ctl c = s_ctl;
        if (exit_kind == 2 && !no_sweeps) {
            const Part q = grid_part(a.partials + (size_t)(s & 1) * P, lane);
            if (lane == 0) ctrl_step(a, s, q, c, nullptr, true, fp64);
        }
        if (blockIdx.x == 0 && lane == 0) {
            const int rs = c.res_sweep;
            const int rb = c.zero ? (rs - 1) % 3 : rs % 3;
            write_result(a, c, rb, (rs + 2) % 3);
        }
    }
}

// ================================================================== small kernel
// Levels one CTA can hold that have no fixed-point plan (step entry points,
// geometric levels): shared memory holds ring[3][n], g - d_i [n], w[nnz],
// rp[n + 1], col[nnz].
template <int G>
__global__ void __launch_bounds__(kSmallMaxThreads) k_power_small(PiArgs a, GridSync *) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n;
    const int m = a.rp[n];
    double *ring0 = reinterpret_cast<double *>(smem_raw);
    double *s_gd = ring0 + 3 * (size_t)n;
    double *s_w = s_gd + n;
    // every row thread's stop sums (A, B, C), by sweep parity; the control warp
    // reduces them (one float-float conversion per control lane, instead of
    // one per row thread)
    double *s_dacc = s_w + m;
    int *s_rp = reinterpret_cast<int *>(s_dacc + 6 * (size_t)blockDim.x);
    int *s_col = s_rp + n + 1;
    __shared__ Part s_pw[32];
    __shared__ Slot s_slot[2];
    __shared__ Ctl c;   // used by lane 0 of the control warp (in registers it would take every row thread's)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nw = blockDim.x >> 5;
    // the control warp's sums of the row warps' partials of parity `par`, in
    // a fixed order (rows warps in order per lane, then the lanes' xor tree)
    auto ctl_part = [&](int par) -> Part {
        double A = 0.0, B = 0.0, C = 0.0;
        for (int w = 1; w < nw; w++) {
            const double *src = s_dacc + ((size_t)par * blockDim.x + 32 * w + lane) * 3;
            A += src[0];
            B += src[1];
            C += src[2];
        }
        Part p;
        p.A = ff_from_double(A);
        p.B = ff_from_double(B);
        p.C = ff_from_double(C);
        return warp_sum_part(p);
    };

    for (int i = tid; i <= n; i += blockDim.x) s_rp[i] = a.rp[i];
    for (int e = tid; e < m; e += blockDim.x) {
        s_col[e] = a.col[e];
        s_w[e] = a.w[e];
    }
    {
        const void *cb = nullptr;
        double cmu = 0.0, cinv = 0.0;
        if (a.start == 1) {
            cb = a.cbuf[a.cres->buf];
            cmu = a.cres->mu;
            cinv = a.cres->inv_s;
        }
        Part acc = part_zero();
        for (int i = tid; i < n; i += blockDim.x) {
            const double xt = start_value(a, i, cb, cmu, cinv);
            ring0[i] = xt;
            double d = 0.0;
            for (int e = a.rp[i], e1 = a.rp[i + 1]; e < e1; e++) d += a.w[e];
            s_gd[i] = a.g - d;
            const ff v = ff_from_double(xt);
            acc.A = ff_add(acc.A, v);
            acc.B = ff_add(acc.B, ff_mul(v, v));
        }
        Part p = warp_sum_part(acc);
        if (lane == 0) s_pw[warp] = p;
    }
    __syncthreads();
    if (warp == 0) {
        Part q = (lane < nw) ? s_pw[lane] : part_zero();
        q = warp_sum_part(q);
        const double mu0 = to_d(q.A) / (double)n;
        double ss0 = to_d(q.B) - (double)n * mu0 * mu0;
        if (ss0 < 0.0) ss0 = 0.0;
        const int e0 = start_exponent(ss0);
        if (lane == 0) {
            ctl_init(c, a, mu0, ss0, e0);
            s_slot[1] = slot_make(ff_from_double(mu0), e0, a.g, c.inv_g, true);
            s_slot[0] = slot_make(ff_zero(), 0, a.g, c.inv_g, true);
        }
    }
    __syncthreads();

    const bool no_sweeps = (a.mode == 1 && a.k_fixed <= 0);
    int s = 0;
    int exit_kind = no_sweeps ? 2 : 0;
    const int rt = tid - 32, nrt = blockDim.x - 32;
    const int rlane = rt & (G - 1);
    const int groups = nrt / G;
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
        const double *x = ring0 + (size_t)(s % 3) * n;
        double *y = ring0 + (size_t)((s + 1) % 3) * n;
        if (warp == 0) {
            if (s >= 1) {
                const Part q = ctl_part(s & 1);
                if (lane == 0) ctrl_step(a, s, q, c, &s_slot[s & 1], false, true);
            }
        } else {
            Acc<double> acc;
            acc.reset();
            for (int base = rt / G;; base += groups) {
                if (__shfl_sync(0xffffffffu, base, 0) >= n) break;
                const int i = base;
                double ac = 0.0, xi = 0.0;
                if (i < n) {
                    xi = x[i];
                    // four independent accumulators: the loads of four entries
                    // are in flight together
                    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
                    int e = s_rp[i] + rlane;
                    const int e1 = s_rp[i + 1];
                    for (; e + 3 * G < e1; e += 4 * G) {
                        const int c0 = s_col[e], c1 = s_col[e + G], c2 = s_col[e + 2 * G], c3 = s_col[e + 3 * G];
                        const double w0 = s_w[e], w1 = s_w[e + G], w2 = s_w[e + 2 * G], w3 = s_w[e + 3 * G];
                        a0 = fma(w0, x[c0], a0);
                        a1 = fma(w1, x[c1], a1);
                        a2 = fma(w2, x[c2], a2);
                        a3 = fma(w3, x[c3], a3);
                    }
                    for (; e < e1; e += G) a0 = fma(s_w[e], x[s_col[e]], a0);
                    ac = (a0 + a1) + (a2 + a3);
                }
                ac = group_sum<G>(ac);
                // only the lanes leading a row group hold sums
                if (i < n && rlane == 0) {
                    const double yv = (fma(s_gd[i], xi, ac) - sl.gm_d) * sl.sig_d;
                    y[i] = yv;
                    acc.add(yv, xi);
                }
            }
            double *dst = s_dacc + ((size_t)((s + 1) & 1) * blockDim.x + tid) * 3;
            dst[0] = acc.A;
            dst[1] = acc.B;
            dst[2] = acc.C;
        }
        __syncthreads();
        s++;
    }
    __shared__ int s_rb, s_rbp;
    if (warp == 0) {
        if (exit_kind == 2 && !no_sweeps) {
            const Part q = ctl_part(s & 1);
            if (lane == 0) ctrl_step(a, s, q, c, nullptr, true, true);
        }
        if (lane == 0) {
            const int rs = c.res_sweep;
            s_rb = c.zero ? (rs + 2) % 3 : rs % 3;
            s_rbp = (rs + 2) % 3;
            write_result(a, c, 0, 1);
        }
    }
    __syncthreads();
    // result -> buf[0], previous iterate -> buf[1]
    double *o0 = (double *)a.buf[0], *o1 = (double *)a.buf[1];
    const double *rr = ring0 + (size_t)s_rb * n, *rp = ring0 + (size_t)s_rbp * n;
    for (int i = tid; i < n; i += blockDim.x) {
        o0[i] = rr[i];
        o1[i] = rp[i];
    }
}

// ================================================================== host side
__global__ void k_tiles(int n, const int *__restrict__ rp, int ntiles, int *__restrict__ tile_row) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k <= ntiles; k += gridDim.x * blockDim.x) {
        if (k == ntiles) {
            tile_row[k] = n;
            continue;
        }
        const long long target = (long long)k * kTileCost;
        int lo = 0, hi = n;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((long long)rp[mid] + 4ll * mid < target) lo = mid + 1;
            else hi = mid;
        }
        tile_row[k] = lo;
    }
}

int tile_count(int n, long long nnz) { return (int)((nnz + 4ll * n + kTileCost - 1) / kTileCost); }

cmg_status_t build_tiles(int n, long long nnz, const int *rp, int *tile_row, cudaStream_t s) {
    const int nt = tile_count(n, nnz);
    k_tiles<<<grid_for(nt + 1, 256), 256, 0, s>>>(n, rp, nt, tile_row);
    return launch_status();
}

static size_t tiled_smem(bool fp32) {
    const size_t e = fp32 ? sizeof(float) : sizeof(double);
    const size_t ts = fp32 ? sizeof(TileSmem<float>) : sizeof(TileSmem<double>);
    return ts + e * 2 * kTileRows + sizeof(int) * (kTileRows + 4) + 2 * kChunk;
}

template <typename T, typename IDX, bool STAGE>
static const void *sell_kernel_tis(bool chunks, bool stream) {
    if (chunks)
        return stream ? (const void *)k_power_sell<T, IDX, true, true, STAGE, false>
                      : (const void *)k_power_sell<T, IDX, true, false, STAGE, false>;
    return stream ? (const void *)k_power_sell<T, IDX, false, true, STAGE, false>
                  : (const void *)k_power_sell<T, IDX, false, false, STAGE, false>;
}

template <typename T, typename IDX>
static const void *sell_kernel_ti(bool chunks, bool stream, bool stage) {
    return stage ? sell_kernel_tis<T, IDX, true>(chunks, stream) : sell_kernel_tis<T, IDX, false>(chunks, stream);
}

static const void *sell_kernel(int fp32, int col16, bool chunks, bool stream, bool stage) {
    if (fp32)
        return col16 ? sell_kernel_ti<float, uint16_t>(chunks, stream, stage)
                     : sell_kernel_ti<float, int>(chunks, stream, stage);
    return col16 ? sell_kernel_ti<double, uint16_t>(chunks, stream, stage)
                 : sell_kernel_ti<double, int>(chunks, stream, stage);
}

// (a level that stages its whole iterate has 16-bit columns)
static const void *sell_res_kernel(bool chunks) {
    return chunks ? (const void *)k_power_sell<float, uint16_t, true, false, true, true>
                  : (const void *)k_power_sell<float, uint16_t, false, false, true, true>;
}

// Launch of the slice kernel over a level's layout: CTAs and threads (the
// resident form takes them over, so that the sums group the same way).
static cmg_status_t sell_geometry(const SweepLayout &L, int n, int fp32, int *blocks, int *threads, const void **kern,
                                  size_t *smem, bool *stream) {
    DeviceInfo di;
    CMG_TRY(device_info(&di));
    // only a layout that cannot stay in L2 is read evict-first
    const long long lay_bytes = L.entries * (long long)((L.col16 ? 2 : 4) + (fp32 ? 4 : 8));
    *stream = di.l2_bytes > 0 && lay_bytes > (long long)di.l2_bytes;
    const int stage_n = std::min(L.stage_n, n);
    const bool stage = stage_n > 0;
    *kern = sell_kernel(fp32, L.col16, L.hheavy[0] > 0, *stream, stage);
    *threads = stage ? kStageThreads : kTileThreads;
    *smem = stage ? (size_t)((stage_n + 7) & ~7) * (fp32 ? sizeof(float) : sizeof(double)) : 0;
    if (stage) CMG_TRY(allow_max_dynamic_smem(*kern));
    int maxb = 0;
    CMG_TRY(coop_max_blocks(*kern, *threads, *smem, &maxb));
    const int row_warps = *threads / 32 - 1;
    const long long tasks = (long long)(n - L.hheavy[0] + 31) / 32 + L.nchunks;
    *blocks = (int)std::max<long long>(1, std::min<long long>(maxb, (tasks + row_warps - 1) / row_warps));
    return CMG_OK;
}

// Most entries and chunks of one CTA of the slice kernel: out[0], out[1].
__global__ void k_sell_share(PiArgs a, int nb, int *out) {
    const int *M = a.lay_meta, *SO = M + a.lay_h;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
        int e = 0, j = 0;
        for (int c = b; c < a.nchunks; c += nb, j++) {
            int f0, len;
            sell_chunk(a, M, c, &f0, &len);
            e += len;
        }
        e += SO[sell_first_slice(SO, a.lay_nsl, b + 1, nb)] - SO[sell_first_slice(SO, a.lay_nsl, b, nb)];
        atomicMax(out, e);
        atomicMax(out + 1, j);
    }
}

static void sell_args(const SweepLayout &L, int n, PiArgs &a) {
    a.perm = reinterpret_cast<const int *>(L.perm);
    a.lay_h = L.hheavy[0];
    a.lay_nsl = (n - a.lay_h + 31) / 32;
    a.lay_meta = L.meta;
    a.lay_col = L.bcol;
    a.lay_w = L.bw;
    a.hchunk = L.hchunk;
    a.crow = L.crow;
    a.hcount = L.hcount;
    a.cpart = L.cpart;
    a.nchunks = L.nchunks;
}

cmg_status_t sell_share_async(const SweepLayout &L, int n, int *out_dev, cudaStream_t s) {
    CMG_CUDA(cudaMemsetAsync(out_dev, 0, 2 * sizeof(int), s));
    PiArgs a = {};
    sell_args(L, n, a);
    int blocks, threads;
    const void *kern;
    size_t smem;
    bool stream;
    CMG_TRY(sell_geometry(L, n, 1, &blocks, &threads, &kern, &smem, &stream));
    k_sell_share<<<div_up(blocks, 32), 32, 0, s>>>(a, blocks, out_dev);
    return launch_status();
}

cmg_status_t sell_choose_resident(SweepLayout *L, int n, int max_entries, int max_chunks) {
    L->res_e = 0;
    int blocks, threads;
    const void *kern;
    size_t smem;
    bool stream;
    CMG_TRY(sell_geometry(*L, n, 1, &blocks, &threads, &kern, &smem, &stream));
    if (L->stage_n < n || !L->col16) return CMG_OK;
    const size_t need = 4 * (size_t)((n + 7) & ~7) + (size_t)max_entries * (4 + 2) +
                        4 * ((size_t)max_chunks + 2) + 16;
    const void *k = sell_res_kernel(L->hheavy[0] > 0);
    DeviceInfo di;
    CMG_TRY(device_info(&di));
    cudaFuncAttributes fa;
    CMG_CUDA(cudaFuncGetAttributes(&fa, k));
    if ((long long)need > (long long)di.max_smem_optin - (long long)fa.sharedSizeBytes) return CMG_OK;
    CMG_TRY(allow_max_dynamic_smem(k));
    int maxb = 0;
    CMG_TRY(coop_max_blocks(k, threads, need, &maxb));
    if (maxb < blocks) return CMG_OK;
    L->res_e = max_entries;
    L->res_smem = need;
    return CMG_OK;
}

static const void *small_kernel(int G) {
    switch (G) {
        case 1: return (const void *)k_power_small<1>;
        case 2: return (const void *)k_power_small<2>;
        case 4: return (const void *)k_power_small<4>;
        case 8: return (const void *)k_power_small<8>;
        case 16: return (const void *)k_power_small<16>;
        default: return (const void *)k_power_small<32>;
    }
}

// Lanes per row in the small kernel: every lane-operation costs FP64 issue
// slots, so the fewest lanes that keep each lane's dependent FMA chain short.
static int small_lanes(int n, long long nnz) {
    const double avg = (double)nnz / (double)std::max(1, n);
    int g = 1;
    while (g < 32 && g * 16 < avg) g <<= 1;
    return g;
}

// Threads of the small kernel: the control warp plus enough row warps for
// one row per lane group (at most 31 row warps).
static int small_threads(int n, int G) {
    long long lanes = (long long)n * G;
    int w = (int)std::min<long long>(31, std::max<long long>(1, (lanes + 31) / 32));
    return 32 * (w + 1);
}

static size_t small_bytes(const PiLevel &lv, int G) {
    return 8 * (4 * (size_t)lv.n + (size_t)lv.nnz + 6 * (size_t)small_threads(lv.n, G)) +
           4 * ((size_t)lv.n + 1 + (size_t)lv.nnz) + 16;
}

size_t xsweep_smem(int fp32) {
    DeviceInfo d;
    if (device_info(&d) != CMG_OK) return 0;
    cudaFuncAttributes fa;
    const void *k = fp32 ? (const void *)k_power_2p<float> : (const void *)k_power_2p<double>;
    if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) return 0;
    const long long room = (long long)d.max_smem_optin - (long long)fa.sharedSizeBytes - 256;
    // 192 KB: a 48K-vertex FP32 (24K FP64) source block, 24K (12K) vrows
    const long long want = 192ll << 10;
    if (room < (64ll << 10)) return 0;
    return (size_t)(std::min(room, want) & ~255ll);
}

int stage_capacity(int fp32) {
    DeviceInfo d;
    if (device_info(&d) != CMG_OK) return 0;
    cudaFuncAttributes fa;
    const void *k = fp32 ? (const void *)k_power_sell<float, int, true, true, true, false>
                         : (const void *)k_power_sell<double, int, true, true, true, false>;
    if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) return 0;
    const long long room = (long long)d.max_smem_optin - (long long)fa.sharedSizeBytes - 256;
    if (room <= 0) return 0;
    const long long cap = room / (fp32 ? (long long)sizeof(float) : (long long)sizeof(double));
    return (int)(cap & ~3ll);
}

// Lanes per row with which the small kernel holds the level (0: it cannot).
static int small_config(const PiLevel &lv) {
    DeviceInfo d;
    if (device_info(&d) != CMG_OK) return 0;
    const int G = small_lanes(lv.n, lv.nnz);
    return small_bytes(lv, G) + 4096 <= (size_t)d.max_smem_optin ? G : 0;
}

bool small_level_fits(const PiLevel &lv, int fp32) { return !fp32 && small_config(lv) > 0; }

cmg_status_t power_iteration(const PiRun &run, GridSync *gs, cudaStream_t s, const PiWorkspace *ws) {
    const PiLevel &lv = *run.lv;
    Scratch scr(s);
    PiArgs a;
    a.n = lv.n;
    a.rp = lv.rp;
    a.col = lv.col;
    a.w = lv.w;
    a.w32 = lv.w32;
    a.g = lv.g;
    a.tile_row = lv.tile_row;
    a.ntiles = lv.ntiles;
    a.mode = run.mode;
    a.k_fixed = run.k_fixed;
    a.max_sweeps = run.max_sweeps;
    a.tol = run.tol;
    a.seed = run.seed;
    a.start = run.x_init ? 2 : (run.coarse_res ? 1 : 0);
    for (int k = 0; k < 3; k++) {
        a.cbuf[k] = run.coarse_bufs[k];
        a.cfp64 = run.coarse_fp64;
        a.buf[k] = run.bufs[k];
    }
    a.cres = run.coarse_res;
    a.agg = run.coarse_agg;
    a.x_init = run.x_init;
    a.gd = run.gd;
    a.res = run.res;
    a.partials = nullptr;
    a.zero_tol2 = run.fp32 ? kZeroTol2_32 : kZeroTol2_64;
    a.cinvp = run.coarse_inv;
    a.perm = nullptr;
    a.lay_h = a.lay_nsl = 0;
    a.lay_meta = nullptr;
    a.lay_col = a.lay_w = nullptr;
    a.hchunk = nullptr;
    a.crow = nullptr;
    a.hcount = nullptr;
    a.cpart = nullptr;
    a.nchunks = 0;
    a.stage_n = 0;
    void *args[] = {&a, &gs};
    if (lv.fix && !run.fp32) return launch_power_fix(*lv.fix, a, s);
    if (small_level_fits(lv, run.fp32)) {
        const int G = small_config(lv);
        const void *kern = small_kernel(G);
        const size_t smem = small_bytes(lv, G);
        CMG_TRY(allow_max_dynamic_smem(kern));
        return coop_launch(kern, 1, small_threads(lv.n, G), smem, s, args, gs);
    }
    if (lv.rows && lv.lay) return launch_power_rows(*lv.rows, *lv.lay, a, gs, s);
    if (!run.fp32 && !run.gd) return CMG_ERR_INVALID_ARG;
    if (lv.xl && lv.lay) {
        // two-phase kernel: one 1024-thread CTA per SM, the layout's P CTAs
        const XLayout &X = *lv.xl;
        a.perm = reinterpret_cast<const int *>(lv.lay->perm);
        a.x_T = X.T;
        a.x_Q = X.Q;
        a.x_SB = X.SB;
        a.x_VMAX = X.VMAX;
        a.x_src = X.src;
        a.x_dst = X.dst;
        a.x_w = X.w;
        a.x_ps = X.pass_s;
        a.x_sal = X.sal;
        a.x_qoff = X.qoff;
        a.x_ndb = X.ndb;
        a.x_dbr = X.dbr;
        a.x_dbl = X.dbl;
        a.x_cdel = X.cdel;
        a.x_choff = X.choff;
        a.x_chk = X.chk;
        a.x_pmax = X.pmax;
        a.x_buf[0] = X.xbuf[0];
        a.x_buf[1] = X.xbuf[1];
        const void *kern = run.fp32 ? (const void *)k_power_2p<float> : (const void *)k_power_2p<double>;
        CMG_TRY(allow_max_dynamic_smem(kern));
        int maxb = 0;
        CMG_TRY(coop_max_blocks(kern, kStageThreads, X.smem, &maxb));
        if (maxb < X.P) return CMG_ERR_TOO_LARGE;
        double *partials;
        if (ws) {
            if (2 * X.P * kPartDoubles > ws->partials_cap) return CMG_ERR_TOO_LARGE;
            partials = ws->partials;
        } else {
            CMG_TRY(scr.get(&partials, (size_t)2 * X.P * kPartDoubles));
        }
        a.partials = reinterpret_cast<PartRec *>(partials);
        return coop_launch(kern, X.P, kStageThreads, X.smem, s, args, gs);
    }
    if (lv.lay) {
        // slice kernel over the level's sweep layout (one graph)
        const SweepLayout &L = *lv.lay;
        sell_args(L, lv.n, a);
        if (a.lay_h > 0) {
            if (!L.hchunk) return CMG_ERR_INVALID_ARG;
            CMG_CUDA(cudaMemsetAsync(L.hcount, 0, sizeof(int) * (size_t)a.lay_h, s));
        }
        a.stage_n = std::min(L.stage_n, lv.n);
        int blocks, threads;
        const void *kern;
        size_t smem;
        bool stream;
        CMG_TRY(sell_geometry(L, lv.n, run.fp32, &blocks, &threads, &kern, &smem, &stream));
        if (run.fp32 && L.res_e > 0) {
            kern = sell_res_kernel(a.lay_h > 0);
            CMG_TRY(allow_max_dynamic_smem(kern));
            smem = L.res_smem;
            a.res_entries = L.res_e;
        }
        double *partials;
        if (ws) {
            if (2 * blocks * kPartDoubles > ws->partials_cap) return CMG_ERR_TOO_LARGE;
            partials = ws->partials;
        } else {
            CMG_TRY(scr.get(&partials, (size_t)2 * blocks * kPartDoubles));
        }
        a.partials = reinterpret_cast<PartRec *>(partials);
        return coop_launch(kern, blocks, threads, smem, s, args, gs);
    }
    if (!a.tile_row) {
        int *tr;
        if (ws) {
            if (tile_count(lv.n, lv.nnz) + 1 > ws->tile_cap) return CMG_ERR_TOO_LARGE;
            tr = ws->tile_row;
        } else {
            CMG_TRY(scr.get(&tr, (size_t)tile_count(lv.n, lv.nnz) + 1));
        }
        CMG_TRY(build_tiles(lv.n, lv.nnz, lv.rp, tr, s));
        a.tile_row = tr;
        a.ntiles = tile_count(lv.n, lv.nnz);
    }
    const void *kern = run.fp32 ? (const void *)k_power_tiled<float> : (const void *)k_power_tiled<double>;
    const size_t smem = tiled_smem(run.fp32 != 0);
    CMG_TRY(allow_max_dynamic_smem(kern));
    int maxb = 0;
    CMG_TRY(coop_max_blocks(kern, kTileThreads, smem, &maxb));
    // one tile per CTA where possible (each tile's phases are latency-bound),
    // never more CTAs than co-resident
    const int blocks = std::max(1, std::min(maxb, a.ntiles));
    double *partials;
    if (ws) {
        if (2 * blocks * kPartDoubles > ws->partials_cap) return CMG_ERR_TOO_LARGE;
        partials = ws->partials;
    } else {
        CMG_TRY(scr.get(&partials, (size_t)2 * blocks * kPartDoubles));
    }
    a.partials = reinterpret_cast<PartRec *>(partials);
    return coop_launch(kern, blocks, kTileThreads, smem, s, args, gs);
}

// Sum of K per-thread doubles over the CTA, result in out[] of every thread
// (fixed order).  sm: 32*K doubles.  Two __syncthreads.  (Used once per
// solve by the final pass.)
template <int K>
__device__ __forceinline__ void block_allsum(double (&v)[K], double *sm, double (&out)[K]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < K; k++) v[k] = warp_sum(v[k]);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; k++) sm[warp * K + k] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; k++) {
        double t = (lane < nw) ? sm[lane * K + k] : 0.0;
        out[k] = warp_sum(t);
    }
    __syncthreads();
}

// Grid-wide sum of K doubles per thread, result in out[] of every thread.
template <int K>
__device__ __forceinline__ bool grid_allsum(double (&v)[K], double *sm, double *part,
                                            double (&out)[K], GridBar *bar) {
    double tot[K];
    block_allsum<K>(v, sm, tot);
    if (gridDim.x == 1) {
#pragma unroll
        for (int k = 0; k < K; k++) out[k] = tot[k];
        return true;
    }
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < K; k++) part[blockIdx.x * K + k] = tot[k];
    if (!grid_sync(bar)) return false;
    const int lane = threadIdx.x & 31;
    double s[K];
#pragma unroll
    for (int k = 0; k < K; k++) s[k] = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32)
#pragma unroll
        for (int k = 0; k < K; k++) s[k] += LDX(part + b * K + k);
#pragma unroll
    for (int k = 0; k < K; k++) out[k] = warp_sum(s[k]);
    return true;
}

// ================================================================== finalisation
// Rows [r0, r1) of CTA b out of nb, balanced by 3 * nnz + 5 * rows.
__device__ __forceinline__ void cta_rows(const int *rp, int n, int b, int nb, int *r0, int *r1) {
    const long long total = 3ll * rp[n] + 5ll * n;
    auto first_at = [&](long long target) {
        int lo = 0, hi = n;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (3ll * rp[mid] + 5ll * mid < target) lo = mid + 1;
            else hi = mid;
        }
        return lo;
    };
    *r0 = (b == 0) ? 0 : first_at((total * b + nb - 1) / nb);
    *r1 = (b == nb - 1) ? n : first_at((total * (b + 1) + nb - 1) / nb);
}

struct FinArgs {
    int n;
    const int *rp;
    const int *col;
    const double *w;
    double g;
    int fp32;
    const void *buf[3];
    const PiResult *res;
    double *u;
    double *tmp;
    double *part;      // [3][gridDim.x][4]
    double *out;       // [2]: lambda, residual
    int sign;          // apply the canonical sign
    int fresh;         // u already holds the vector (skip the vector phase)
    const int *inv;    // the iterates are in layout order: row i is at inv[i] (nullptr: natural)
};

// (|v|, index) order of the sign rule: larger magnitude first, lower index on ties.
__device__ __forceinline__ bool better(double v, int i, double bv, int bi) {
    return v > bv || (v == bv && i < bi);
}

template <int G>
__global__ void __launch_bounds__(kFinThreads) k_finalize(FinArgs a, GridSync *gs) {
    __shared__ double sm[32 * 4];
    __shared__ double s_best[32], s_bval[32];
    __shared__ int s_bidx[32];
    __shared__ GridBar s_bar;
    if (threadIdx.x == 0) grid_bar_init(&s_bar, gs);
    const int n = a.n;
    int r0, r1;
    cta_rows(a.rp, n, blockIdx.x, gridDim.x, &r0, &r1);
    const int lane = threadIdx.x & (G - 1);
    const int groups = blockDim.x / G;
    double *part0 = a.part, *part1 = a.part + (size_t)gridDim.x * 4,
           *part2 = a.part + (size_t)gridDim.x * 8;
    double p[4], S[4];

    if (!a.fresh) {
        const PiResult r = *a.res;
        const bool recompute = a.fp32 && r.sweeps > 0 && !r.zero;
        if (recompute) {
            // FP64 recomputation of the last sweep from the previous (FP32) iterate
            const float *x = (const float *)a.buf[r.buf_prev];
            p[0] = p[1] = p[2] = p[3] = 0.0;
            for (int base = r0 + threadIdx.x / G;; base += groups) {
                if (__shfl_sync(0xffffffffu, base, 0) >= r1) break;
                const int i = base;
                double acc = 0.0, xi = 0.0;
                if (i < r1) {
                    xi = ((double)x[a.inv ? a.inv[i] : i] - r.mu_prev) * r.inv_s_prev;
                    const int e1 = __ldg(a.rp + i + 1);
                    for (int e = __ldg(a.rp + i) + lane; e < e1; e += G) {
                        const int j = __ldg(a.col + e);
                        const double xj = ((double)x[a.inv ? a.inv[j] : j] - r.mu_prev) * r.inv_s_prev;
                        acc += __ldg(a.w + e) * (xi - xj);
                    }
                }
                acc = group_sum<G>(acc);
                if (i < r1 && lane == 0) {
                    const double yv = a.g * xi - acc;
                    a.tmp[i] = yv;
                    p[0] += yv;
                    p[1] += yv * yv;
                }
            }
            if (!grid_allsum<4>(p, sm, part0, S, &s_bar)) return;
            const double mu = S[0] / (double)n;
            const double ss = S[1] - (double)n * mu * mu;
            const double inv = ss > 0.0 ? 1.0 / sqrt(ss) : 0.0;
            for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) a.u[i] = (a.tmp[i] - mu) * inv;
        } else if (a.fp32) {
            const float *y = (const float *)a.buf[r.buf];
            for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x)
                a.u[i] = ((double)y[a.inv ? a.inv[i] : i] - r.mu) * r.inv_s;
        } else {
            const double *y = (const double *)a.buf[r.buf];
            for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x)
                a.u[i] = (y[a.inv ? a.inv[i] : i] - r.mu) * r.inv_s;
        }
    }
    // ---- canonical sign: the entry of largest |u_i| (lowest index on ties) is
    // made positive.  Its signed value travels with the reduction, so no CTA
    // reads u after another may have negated it.
    if (a.sign) {
        double best = -1.0, bval = 0.0;
        int bidx = 0x7fffffff;
        for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
            const double v = a.u[i];
            if (better(fabs(v), i, best, bidx)) {
                best = fabs(v);
                bidx = i;
                bval = v;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
            const double ov = __shfl_xor_sync(0xffffffffu, bval, o);
            if (better(ob, oi, best, bidx)) {
                best = ob;
                bidx = oi;
                bval = ov;
            }
        }
        if ((threadIdx.x & 31) == 0) {
            s_best[threadIdx.x >> 5] = best;
            s_bidx[threadIdx.x >> 5] = bidx;
            s_bval[threadIdx.x >> 5] = bval;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < (int)blockDim.x / 32; q++)
                if (better(s_best[q], s_bidx[q], best, bidx)) {
                    best = s_best[q];
                    bidx = s_bidx[q];
                    bval = s_bval[q];
                }
            part1[blockIdx.x * 4 + 0] = best;
            part1[blockIdx.x * 4 + 1] = (double)bidx;
            part1[blockIdx.x * 4 + 2] = bval;
        }
        if (!grid_sync(&s_bar)) return;
        __syncthreads();
        if (threadIdx.x == 0) {
            double bb = -1.0, bv = 0.0;
            int bi = 0x7fffffff;
            for (int b = 0; b < (int)gridDim.x; b++) {
                const double v = LDX(part1 + b * 4 + 0);
                const int ii = (int)LDX(part1 + b * 4 + 1);
                if (better(v, ii, bb, bi)) {
                    bb = v;
                    bi = ii;
                    bv = LDX(part1 + b * 4 + 2);
                }
            }
            s_bval[0] = bv;
        }
        __syncthreads();
        if (s_bval[0] < 0.0)
            for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) a.u[i] = -a.u[i];
        if (!grid_sync(&s_bar)) return;
    } else if (!a.fresh) {
        if (!grid_sync(&s_bar)) return;
    }
    // ---- Rayleigh quotient: lambda = (1/2) sum_i sum_j w_ij (u_i - u_j)^2 / ||u||^2
    p[0] = p[1] = p[2] = p[3] = 0.0;
    for (int base = r0 + threadIdx.x / G;; base += groups) {
        if (__shfl_sync(0xffffffffu, base, 0) >= r1) break;
        const int i = base;
        double acc = 0.0, ui = 0.0;
        if (i < r1) {
            ui = LDX(a.u + i);
            const int e1 = __ldg(a.rp + i + 1);
            for (int e = __ldg(a.rp + i) + lane; e < e1; e += G) {
                const double d = ui - LDX(a.u + __ldg(a.col + e));
                acc += __ldg(a.w + e) * d * d;
            }
        }
        acc = group_sum<G>(acc);
        if (i < r1 && lane == 0) {
            p[0] += acc;
            p[1] += ui * ui;
        }
    }
    if (!grid_allsum<4>(p, sm, part2, S, &s_bar)) return;
    const double uu = S[1];
    const double lam = 0.5 * S[0] / uu;
    // ---- residual ||(L - lambda I) u|| / ||u||, (L u)_i = sum_j w_ij (u_i - u_j)
    p[0] = p[1] = p[2] = p[3] = 0.0;
    for (int base = r0 + threadIdx.x / G;; base += groups) {
        if (__shfl_sync(0xffffffffu, base, 0) >= r1) break;
        const int i = base;
        double acc = 0.0, ui = 0.0;
        if (i < r1) {
            ui = LDX(a.u + i);
            const int e1 = __ldg(a.rp + i + 1);
            for (int e = __ldg(a.rp + i) + lane; e < e1; e += G)
                acc += __ldg(a.w + e) * (ui - LDX(a.u + __ldg(a.col + e)));
        }
        acc = group_sum<G>(acc);
        if (i < r1 && lane == 0) {
            const double rr = acc - lam * ui;
            p[0] += rr * rr;
        }
    }
    if (!grid_allsum<4>(p, sm, part0, S, &s_bar)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.out[0] = lam;
        a.out[1] = sqrt(S[0] / uu);
    }
}

static const void *finalize_kernel(int G) {
    switch (G) {
        case 2: return (const void *)k_finalize<2>;
        case 4: return (const void *)k_finalize<4>;
        case 8: return (const void *)k_finalize<8>;
        case 16: return (const void *)k_finalize<16>;
        default: return (const void *)k_finalize<32>;
    }
}

cmg_status_t finalize(const PiLevel &lv, int fp32, void *const bufs[3], const PiResult *res,
                      double *u, int sign, int fresh, double *out2, GridSync *gs, cudaStream_t s,
                      const PiWorkspace *ws) {
    const int G = lanes_for_avg((double)lv.nnz / (double)std::max(1, lv.n));
    const void *kern = finalize_kernel(G);
    int maxb = 0;
    CMG_TRY(coop_max_blocks(kern, kFinThreads, 0, &maxb));
    DeviceInfo d;
    CMG_TRY(device_info(&d));
    const long long bytes = 12 * lv.nnz + 20ll * lv.n;
    int blocks = (int)std::min<long long>((bytes + 65535) / 65536, (long long)std::min(maxb, 2 * d.sms));
    blocks = std::max(1, blocks);
    Scratch scr(s);
    double *part, *tmp = nullptr;
    if (ws) {
        if (12 * blocks > ws->fin_part_cap || (fp32 && !fresh)) return CMG_ERR_TOO_LARGE;
        part = ws->fin_part;
    } else {
        CMG_TRY(scr.get(&part, (size_t)12 * blocks));
        if (fp32 && !fresh) CMG_TRY(scr.get(&tmp, (size_t)lv.n));
    }
    FinArgs a;
    a.n = lv.n;
    a.rp = lv.rp;
    a.col = lv.col;
    a.w = lv.w;
    a.g = lv.g;
    a.fp32 = fp32;
    for (int k = 0; k < 3; k++) a.buf[k] = bufs ? bufs[k] : nullptr;
    a.res = res;
    a.u = u;
    a.tmp = tmp;
    a.part = part;
    a.out = out2;
    a.sign = sign;
    a.fresh = fresh;
    a.inv = lv.lay ? lv.lay->inv : nullptr;
    void *args[] = {&a, &gs};
    return coop_launch(kern, blocks, kFinThreads, 0, s, args, gs);
}

}  // namespace cmg
