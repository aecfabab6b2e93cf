// Vector kernels of an outer iteration (BiCG updates, deferred updates, pass-2 MR
// update, and the FP64 kernels with inner products).
//
// Deferred updates (FP32 and double-float, double-pass forms).  Sub-step j of
// the BiCG part updates u_i <- r_i - beta_j u_i and r_i <- r_i - alpha_j u_{i+1}
// for every i <= j, but the next sweep reads only u_j and r_j.  So a sub-step can
// update those two alone, and the updates of i < j, which are local to a site,
// are made up in order by whoever needs the vectors next (deferred()): in FP32
// the MR step, and for the Gram matrix the kernel that forms it (in registers);
// in double-float, where doing them twice would cost more than the traffic, a
// kernel before the Gram matrix (k_deferred).  Each vector is then read and
// written once per outer iteration instead of once per sub-step: per site 2 l
// instead of l (l + 1) updates of 3 spinors.  Where it is done: defer_updates
// in solver.cu.  In pass 2 (always) the updated r_j goes to another vector
// (rb_j, rb_at), so that the MR step still has every occurrence of the weighted sum and
// adds to y once instead of l + 1 times.  Every number is formed by the same
// operations in the same order as without.
//
// Spread over components and chains (FP64).  On small and medium lattices the
// FP64 kernels are bound by the FP64 pipe (76 cycles per warp instruction and
// sub-partition), not by memory: one thread per site in 256-thread blocks used
// 2 SMs on 4^3 x 8 and 32 on 8^3 x 16.  Here
//   * elementwise updates take one thread per 16 bytes of a vector, the shift
//     vectors of single-pass solves one warp per shift and 32 pairs;
//   * kernels with inner products take a tile of 32 sites per block (or per
//     cluster): a warp per component, and for the products one warp per real
//     chain, which adds a site's 12 components in order.
// Tiles follow the site ranges and warps that 256-thread blocks of a grid of
// `nbx` blocks would have (tile 8 b + w: warp w of block b), and their partials
// are added eight by eight in a shuffle tree's order (tile_group), so every sum
// has one order whatever the launch.  (Double-float kernels with inner products
// were slower this way: 16^3 x 32, l = 2, Gram 43 -> 104 us, MR 59 -> 128 us; a
// product chain of 24 dependent double-float FMAs keeps 3 of 12 warps busy.)
#pragma once

#include "solver_kernels.cuh"

namespace fa {

constexpr int kFlat = 256;        // threads of the elementwise kernels
constexpr int kFlatShift = 32;    // pairs per block of the update with shift vectors (one warp per shift)
constexpr int kMrThreads = 384;   // one warp per component of a tile
template <typename R> constexpr int flat_elems(int V) { return Ch<R>::N * V; }
inline int flat_blocks(int n, int per) { return (n + per - 1) / per; }

__device__ __forceinline__ cx<double> ldc(const double2* p) {
    const double2 t = *p;
    return {t.x, t.y};
}
__device__ __forceinline__ void stc(double2* p, cx<double> v) { *p = make_double2(v.r, v.i); }

// 16 bytes of a vector: element e of its Ch<R>::N * V
template <typename R> __device__ __forceinline__ Ch<R> lde(const typename Ch<R>::T* p) { return Ch<R>::ld(p, 0, 0, 0); }
template <typename R> __device__ __forceinline__ void ste(typename Ch<R>::T* p, const Ch<R>& v) { v.stv(p, 0, 0, 0); }
template <typename R> __device__ __forceinline__ void ste_cs(typename Ch<R>::T* p, const Ch<R>& v) { v.stv_cs(p, 0, 0, 0); }

// sites of a tile: first site of lane 0 and the end of its block's range; a
// lane takes s, s + 256, ... below the end
struct TileSites {
    int s, end;
};
__device__ __forceinline__ TileSites tile_sites(int V, int tile, int ntile) {
    int s0, s1;
    site_range(V, tile >> 3, ntile >> 3, s0, s1);
    return {s0 + 32 * (tile & 7) + (int)(threadIdx.x & 31), s1};
}

// sum over the warp's lanes in the order of the block reductions' shuffle tree
__device__ __forceinline__ double warp_sum(double a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a = __dadd_rn(a, __shfl_down_sync(0xffffffffu, a, o));
    return a;
}
// u_i <- r_i - beta u_i, i = i0..j (i0 = j where the others are deferred)
template <typename R, int EPT>
__global__ void __launch_bounds__(kFlat)
k_update_u(const SolverDev* __restrict__ ds, int i0, int j, int pass2, const int4* tab) {
    dep_wait();
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, pass2)) return;
    const TraceScope trace_(trace_kind<R>(FA_TK_UPDATE_U));
    const int n = flat_elems<R>(d.V), e0 = w.bx * (kFlat * EPT) + threadIdx.x;
    const cx<R> nb = nweight<R>(d.rec_beta, d.rec_beta4, d.st->m * d.L + j);
    for (int i = i0; i <= j; ++i) {
        const typename Ch<R>::T* r = Vec<R>::r(d) + (size_t)i * n;
        typename Ch<R>::T* u = Vec<R>::u(d) + (size_t)i * n;
        Ch<R> a[EPT], b[EPT];
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
            const int e = e0 + k * kFlat;
            if (e < n) {
                a[k] = lde<R>(r + e);
                b[k] = lde<R>(u + e);
            }
        }
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
            const int e = e0 + k * kFlat;
            if (e >= n) continue;
#pragma unroll
            for (int c = 0; c < Ch<R>::W; ++c) b[k].c[c] = cfma(nb, b[k].c[c], a[k].c[c]);
            ste<R>(u + e, b[k]);
        }
    }
}

// r_i <- r_i - alpha u_{i+1}, i = i0..j (FP32, double-float).  Pass 1: in place,
// the occurrences stored where the iteration is stored; with i0 = 0 the seed
// solution x too (else the deferred updates accumulate it).  Pass 2: i0 = j, into
// rb_j.  XS (pass 1): block 0 runs the shift part of sub-step j beside the
// vector blocks.
template <typename R, bool PASS2, bool XS, int EPT>
__global__ void __launch_bounds__(kFlat)
k_update_r(const SolverDev* __restrict__ ds, int i0, int j, int seed_x, const int4* tab) {
    dep_wait();
    const Where w = where<XS>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, PASS2)) return;
    const TraceScope trace_(trace_kind<R>(FA_TK_UPDATE_R, XS));
    if (XS && w.bx < 0) {
        sc_alpha_shifts(d, j);
        return;
    }
    using T = typename Ch<R>::T;
    const int n = flat_elems<R>(d.V), e0 = w.bx * (kFlat * EPT) + threadIdx.x, m = d.st->m;
    const cx<R> na = nweight<R>(d.rec_alpha, d.rec_alpha4, m * d.L + j);
    T* store = PASS2 ? nullptr : store_at<R>(d, m);
    for (int i = i0; i <= j; ++i) {
        T* r = Vec<R>::r(d) + (size_t)i * n;
        const T* u = Vec<R>::u(d) + (size_t)(i + 1) * n;
        T* out = PASS2 ? rb_at<R>(d, i) : r;
        Ch<R> a[EPT], b[EPT];
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
            const int e = e0 + k * kFlat;
            if (e < n) {
                a[k] = lde<R>(r + e);
                b[k] = lde<R>(u + e);
            }
        }
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
            const int e = e0 + k * kFlat;
            if (e >= n) continue;
            if (store != nullptr) ste_cs<R>(store + (size_t)slot_old(j, i) * n + e, a[k]);
#pragma unroll
            for (int c = 0; c < Ch<R>::W; ++c) a[k].c[c] = cfma(na, b[k].c[c], a[k].c[c]);
            ste<R>(out + e, a[k]);
        }
    }
    if (!PASS2 && seed_x && d.x64 != nullptr) {
        for (int k = 0; k < EPT; ++k) {
            const int e = e0 + k * kFlat;
            if (e < n) acc_x<R>(d.x64, e / d.V, d.V, e % d.V, d.rec_alpha[m * d.L + j], lde<R>(Vec<R>::u(d) + e));
        }
    }
}

// Double-float, l > 2: the deferred updates of pass 1 before the Gram matrix.
// Leaves r_i and u_i final for i < L - 1 (the others are).
template <int L>
__global__ void __launch_bounds__(kFlat)
k_deferred(const SolverDev* __restrict__ ds, const int4* tab) {
    using R = df;
    dep_wait();
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, 0)) return;
    const TraceScope trace_(trace_kind<R>(FA_TK_UPDATE_R, true));
    const int n = 12 * d.V, e = w.bx * kFlat + threadIdx.x, m = d.st->m;
    if (e >= n) return;
    float4 *rp = Vec<R>::r(d) + e, *up = Vec<R>::u(d) + e;
    const StepScalars<R, L> sc(d, m);
    Ch<R> r[L + 1], u[L];
#pragma unroll
    for (int i = 0; i < L; ++i) r[i] = lde<R>(rp + (size_t)i * n);
#pragma unroll
    for (int i = 0; i < L; ++i) u[i] = lde<R>(up + (size_t)i * n);
    deferred<R, L>(d, m, sc, r, u, store_at<R>(d, m), e / d.V, e % d.V);
#pragma unroll
    for (int i = 0; i < L - 1; ++i) {
        ste<R>(rp + (size_t)i * n, r[i]);
        ste<R>(up + (size_t)i * n, u[i]);
    }
}

// Pass 2, FP32 and double-float: the deferred updates, y += every weighted
// occurrence of the outer iteration, and the MR update of r_0 and u_0.
template <typename R, int L>
__global__ void __launch_bounds__(kFlat)
k_mr_acc(const SolverDev* __restrict__ ds, const int4* tab) {
    dep_wait();
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, 1)) return;
    const TraceScope trace_(trace_kind<R>(FA_TK_MR));
    const int V = d.V, n = flat_elems<R>(V), e = w.bx * kFlat + threadIdx.x, m = d.st->m;
    if (e >= n) return;
    const int q = e / V, s = e - q * V;
    using T = typename Ch<R>::T;
    T *rp = Vec<R>::r(d) + e, *up = Vec<R>::u(d) + e;
    Ch<R> r[L + 1], u[L + 1];
#pragma unroll
    for (int i = 0; i <= L; ++i) r[i] = lde<R>(rp + (size_t)i * n);
#pragma unroll
    for (int i = 0; i <= L; ++i) u[i] = lde<R>(up + (size_t)i * n);
    const StepScalars<R, L> sc(d, m);
    double2 y[Ch<R>::W];
    double2* yp = d.y + (size_t)(q * Ch<R>::W) * V + s;
#pragma unroll
    for (int c = 0; c < Ch<R>::W; ++c) y[c] = yp[(size_t)c * V];
    deferred_acc<R, L>(d, m, sc, r, u, q, s, y);
    acc_mr<R, L>(d, m, r, y);
#pragma unroll
    for (int c = 0; c < Ch<R>::W; ++c) yp[(size_t)c * V] = y[c];
    Ch<R> r0 = r[0], u0 = u[0];
#pragma unroll
    for (int j = 1; j <= L; ++j) {
        if (d.x64 != nullptr) acc_x<R>(d.x64, q, V, s, d.rec_gamma[m * (L + 1) + j], r[j - 1]);
        const cx<R> ng = nweight<R>(d.rec_gamma, d.rec_gamma4, m * (L + 1) + j);
#pragma unroll
        for (int c = 0; c < Ch<R>::W; ++c) {
            r0.c[c] = cfma(ng, r[j].c[c], r0.c[c]);
            u0.c[c] = cfma(ng, u[j].c[c], u0.c[c]);
        }
    }
    ste<R>(rp, r0);
    ste<R>(up, u0);
}

// FP64: r_i <- r_i - alpha u_{i+1}, i = 0..j.  ACC (pass 2): y += sum_i
// coef[m][slot_old(j,i)] r_i (before the update).  Bound by the FP64 pipe in pass 2 (14
// instructions per element on average at l = 2).  Measured on GB300, 32^3 x 64, l = 2, pass 2, us per
// launch with 1 / 4 elements per thread: 630 / 709; a loop that returns early past
// the end, 64 registers instead of 54: 800; the next pair loaded ahead: 753.
constexpr int kUpdateElems64 = 1;
template <bool ACC, bool XS>
__global__ void __launch_bounds__(kFlat)
k_update_r64(const SolverDev* __restrict__ ds, int j, int pass2, const int4* tab) {
    dep_wait();
    const Where w = where<XS>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, pass2)) return;
    const TraceScope trace_(trace_kind<double>(FA_TK_UPDATE_R, XS));
    if (XS && w.bx < 0) {
        sc_alpha_shifts(d, j);
        return;
    }
    const int n = 12 * d.V, m = d.st->m, L = d.L;
    const double2 al = d.rec_alpha[m * L + j];
    const cx<double> na = negcx<double>(al);
    double2* store = pass2 ? nullptr : store_at<double>(d, m);
    constexpr int EPT = kUpdateElems64;
    const int e0 = w.bx * (kFlat * EPT) + (int)threadIdx.x;
    cx<double> t[EPT];
#pragma unroll
    for (int k = 0; k < EPT; ++k) t[k] = czero<double>();
    for (int i = 0; i <= j; ++i) {
        double2* r = d.r64 + (size_t)i * n;
        const double2* u = d.u64 + (size_t)(i + 1) * n;
        const cx<double> cf = ACC ? tocx<double>(d.coef[(size_t)m * nc_slots(L) + slot_old(j, i)]) : czero<double>();
        cx<double> a[EPT], b[EPT];
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
            const int e = e0 + k * kFlat;
            if (e < n) {
                a[k] = ldc(r + e);
                b[k] = ldc(u + e);
            }
        }
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
            const int e = e0 + k * kFlat;
            if (e >= n) continue;
            if (store != nullptr) __stcs(store + (size_t)slot_old(j, i) * n + e, make_double2(a[k].r, a[k].i));
            if (ACC) t[k] = cfma(cf, a[k], t[k]);
            stc(r + e, cfma(na, b[k], a[k]));
        }
    }
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
        const int e = e0 + k * kFlat;
        if (e >= n) continue;
        if (ACC) {
            const double2 y = d.y[e];
            d.y[e] = make_double2(__dadd_rn(y.x, t[k].r), __dadd_rn(y.y, t[k].i));
        }
        if (d.x64 != nullptr) acc_x1(d.x64 + e, al, ldc(d.u64 + e));
    }
}

// The same with shift vectors (single pass), W pairs per block.  W = 32: warp 0
// updates r, and warp w the vectors of the shifts w, w + 8, ...  W = 256: a thread
// takes a pair through all shifts (rule: set_forms64 in solver.cu).  The r before
// the update stay in shared memory.
template <int W>
__global__ void __launch_bounds__(kFlat)
k_update_shifts64(const SolverDev* __restrict__ ds, int j, const int4* tab) {
    dep_wait();
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, 0)) return;
    const TraceScope trace_(trace_kind<double>(FA_TK_UPDATE_R));
    const int n = 12 * d.V, m = d.st->m, L = d.L;
    const int lane = threadIdx.x % W, part = threadIdx.x / W;
    const int e = w.bx * W + lane;
    __shared__ double2 old[kMaxEll][W], now[W];
    if (e < n && part == 0) {
        const double2 al = d.rec_alpha[m * L + j];
        const cx<double> na = negcx<double>(al);
        for (int i = 0; i <= j; ++i) {
            double2* ri = d.r64 + (size_t)i * n + e;
            const cx<double> a = ldc(ri), b = ldc(d.u64 + (size_t)(i + 1) * n + e);
            const cx<double> v = cfma(na, b, a);
            stc(ri, v);
            old[i][lane] = make_double2(a.r, a.i);
            if (i == j) now[lane] = make_double2(v.r, v.i);
        }
        if (d.x64 != nullptr) acc_x1(d.x64 + e, al, ldc(d.u64 + e));
    }
    if (W < kFlat) __syncthreads();
    if (e >= n) return;
    const cx<double> rj = ldc(&old[j][lane]), rn = ldc(&now[lane]);
    for (int sh = part; sh < d.ns; sh += kFlat / W) {
        if (!d.active[sh]) continue;
        const double2* P = d.prec + ((size_t)sh * d.max_outer + m) * ps_stride(L) + 5 * j;
        const cx<double> as = tocx<double>(P[0]), bs = negcx<double>(P[1]), iz = tocx<double>(P[2]);
        const cx<double> iaz = tocx<double>(P[3]), niazn = negcx<double>(P[4]);
        double2* us = d.us + (size_t)sh * (L + 1) * n + e;
        double2* xs = d.xs + (size_t)sh * n + e;
        const cx<double> xv = ldc(xs);
        // u^s_i <- r_old_i/zeta - beta_s u^s_i
        cx<double> v0, vj;
        for (int i = 0; i <= j; ++i) {
            vj = cfma(bs, ldc(us + (size_t)i * n), cmul(iz, ldc(&old[i][lane])));
            stc(us + (size_t)i * n, vj);
            if (i == 0) v0 = vj;
        }
        // u^s_{j+1} <- r_old_j/(alpha_s zeta) - r_j/(alpha_s zeta_new) - sigma u^s_j; x_s += alpha_s u^s_0
        cx<double> t = cmul(iaz, rj);
        t = cfma(niazn, rn, t);
        stc(us + (size_t)(j + 1) * n, crfma(-d.sigma[sh], vj, t));
        stc(xs, cfma(as, v0, xv));
    }
}

// Gram matrix <r_i, r_k>, 0 <= i <= k <= L (FP64): a warp per chain (real or
// imaginary part of one product); l <= 2 needs no imaginary part of the
// diagonal.  Last block: the MR coefficients, and with `shifts` their shift part.
// Measured on GB300 (tracer, us per launch, one thread per site with all
// products -> this): l = 2, 8^3 x 16 30 -> 8.7.  (Nine warps and two blocks per SM, 113
// registers instead of 148: 32^3 x 64 1522 -> 1347, 8^3 x 16 11 -> 21.)
constexpr int kGramWarps = 12;
template <int L>
__global__ void __launch_bounds__(32 * kGramWarps)
k_gram_tile(const SolverDev* __restrict__ ds, int shifts, const int4* tab) {
    dep_wait();
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, 0)) return;
    const TraceScope trace_(trace_kind<double>(FA_TK_GRAM));
    constexpr int NG = n_gram(L), NW = kGramWarps;
    constexpr int NCH = L <= 2 ? 2 * NG - (L + 1) : 2 * NG;
    const int V = d.V, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const TileSites ts = tile_sites(V, w.bx, w.nbx);
    // chains in the order: real parts of the NG products, then imaginary parts
    // (l <= 2: of the off-diagonal ones only)
    for (int ch = warp; ch < NCH; ch += NW) {
        const int im = ch >= NG, lo = (im && L <= 2) ? 1 : 0;
        int i = 0, c = im ? ch - NG : ch;   // the c-th product with k >= i (or k > i)
        for (; c >= L + 1 - i - lo; ++i) c -= L + 1 - i - lo;
        const int k = i + lo + c;
        const double2* a = d.r64 + (size_t)i * 12 * V;
        const double2* b = d.r64 + (size_t)k * 12 * V;
        double acc = 0.0;
        for (int s = ts.s; s < ts.end; s += 256) {
#pragma unroll
            for (int q = 0; q < 12; ++q) {
                const double2 x = a[(size_t)q * V + s], y = b[(size_t)q * V + s];
                acc = __fma_rn(x.x, im ? y.y : y.x, acc);
                acc = __fma_rn(im ? -x.y : x.y, im ? y.x : y.y, acc);
            }
        }
        acc = warp_sum(acc);
        if (lane == 0) {
            double* p = &d.part[(size_t)(i * (L + 1) - i * (i - 1) / 2 + (k - i)) * w.nbx + w.bx].x;
            p[im] = acc;
            if (L <= 2 && !im && i == k) p[1] = 0.0;
        }
    }
    if (last_block(d.st, w.ntk) == LB_LAST) {
        sc_mr_seed<L, false>(d, w.nbx, false);
        if (shifts) {
            __syncthreads();
            sc_mr_shifts<L>(d);
        }
    }
}

// MR update of a tile (FP64): warp q takes component q; then three warps form
// <rt, r_0> (two chains) and |r_0|^2.  SHIFTS (single pass): the C blocks of a
// cluster take the shifts rank, rank + C, ...; block 0 of the cluster
// overwrites r_0 and u_0 once all of them hold the old r.  Only block 0 takes a
// ticket, so the convergence step may run while the others are still at their
// shifts: whatever it writes (the active flags, the outer iteration) they read
// before the cluster's barrier, which comes before the ticket.  ACC (pass 2): y +=
// sum_k coef[m][slot_mr(k)] r_k.
// Measured on GB300 (tracer, us per launch, one thread per site -> this): l = 2,
// 8^3 x 16 28 -> 12.8 (pass 1), 30 -> 8.3 (pass 2).
template <int L, bool ACC, bool SHIFTS, bool DOT, bool XS, int C>
__global__ void __launch_bounds__(kMrThreads)
k_mr_tile(const SolverDev* __restrict__ ds, int pass2, ScalarStep step, const int4* tab) {
    static_assert(C == 1 || (SHIFTS && !XS), "clusters split the shifts");
    dep_wait();
    Where w = where<XS>(tab);
    int rank = 0;
    if constexpr (C > 1) {
        rank = w.bx % C;
        w.bx /= C;
        w.nbx /= C;
        w.ntk /= C;
    }
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, pass2)) return;
    const TraceScope trace_(trace_kind<double>(FA_TK_MR, XS));
    if (XS && w.bx < 0) {
        mr_shifts<L>(d, [&] {
            __threadfence();   // the new zeta of every thread before the ticket
            run_step<false>(d, step, w.nbx, w.ntk);
        });
        return;
    }
    const int V = d.V, n = 12 * V, m = d.st->m;
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const TileSites ts = tile_sites(V, w.bx, w.nbx);
    __shared__ double2 rnew[12][32];
    cx<double> ng[L + 1];
    ng[0] = czero<double>();
#pragma unroll
    for (int k = 1; k <= L; ++k) ng[k] = negcx<double>(d.rec_gamma[m * (L + 1) + k]);
    double2* store = pass2 ? nullptr : store_at<double>(d, m);
    unsigned long long live = 0ull;   // the shifts still active
    if constexpr (SHIFTS) {
        static_assert(kMaxShifts == 64, "one bit per shift");
        live = __ballot_sync(0xffffffffu, lane < d.ns && d.active[lane] != 0);
        live |= (unsigned long long)__ballot_sync(0xffffffffu, 32 + lane < d.ns && d.active[32 + lane] != 0) << 32;
    }
    double acc = 0.0;
    // every lane makes the same number of rounds (barriers); its site may lie past the end
    const int first = ts.s - lane;
    for (int sb = first; sb < ts.end || sb == first; sb += 256) {
        const int s = sb + lane;
        const bool valid = s < ts.end;
        const size_t e = (size_t)q * V + s;
        cx<double> rv[L + 1];
        if (valid) {
#pragma unroll
            for (int i = 0; i <= L; ++i) rv[i] = ldc(d.r64 + (size_t)i * n + e);
        }
        if constexpr (C > 1) tile_sync<C>();
        if (valid && rank == 0) {
            if (store != nullptr) {
#pragma unroll
                for (int k = 0; k < L; ++k) __stcs(store + (size_t)slot_mr(L, k) * n + e, make_double2(rv[k].r, rv[k].i));
            }
            if (ACC) {
                cx<double> t = czero<double>();
#pragma unroll
                for (int k = 0; k < L; ++k)
                    t = cfma(tocx<double>(d.coef[(size_t)m * nc_slots(L) + slot_mr(L, k)]), rv[k], t);
                const double2 y = d.y[e];
                d.y[e] = make_double2(__dadd_rn(y.x, t.r), __dadd_rn(y.y, t.i));
            }
            if (d.x64 != nullptr) {
#pragma unroll
                for (int k = 1; k <= L; ++k) acc_x1(d.x64 + e, d.rec_gamma[m * (L + 1) + k], rv[k - 1]);
            }
            cx<double> r0 = rv[0], u0 = ldc(d.u64 + e);
#pragma unroll
            for (int k = 1; k <= L; ++k) {
                r0 = cfma(ng[k], rv[k], r0);
                u0 = cfma(ng[k], ldc(d.u64 + (size_t)k * n + e), u0);
            }
            stc(d.r64 + e, r0);
            stc(d.u64 + e, u0);
            if (DOT) rnew[q][lane] = make_double2(r0.r, r0.i);
        }
        if (SHIFTS && valid) {
            for (int sh = rank; sh < d.ns; sh += C) {
                if (!((live >> sh) & 1ull)) continue;
                const double2* P = d.prec + ((size_t)sh * d.max_outer + m) * ps_stride(L) + 5 * L;
                double2* us = d.us + (size_t)sh * (L + 1) * n + e;
                double2* xs = d.xs + (size_t)sh * n + e;
                cx<double> xv = ldc(xs), u0 = ldc(us);
#pragma unroll
                for (int k = 0; k < L; ++k) xv = cfma(tocx<double>(P[1 + k]), rv[k], xv);
#pragma unroll
                for (int k = 1; k <= L; ++k) u0 = cfma(ng[k], ldc(us + (size_t)k * n), u0);
                stc(xs, xv);
                stc(us, cmul(tocx<double>(P[0]), u0));
            }
        }
        if (DOT) {
            __syncthreads();
            // warp 0, 1: real and imaginary part of <rt, r_0>; warp 2: |r_0|^2
            if (q < 3 && valid && rank == 0) {
#pragma unroll
                for (int k = 0; k < 12; ++k) {
                    const double2 r = rnew[k][lane];
                    const double2 t = q == 2 ? r : d.rt64[(size_t)k * V + s];
                    acc = __fma_rn(t.x, q == 1 ? r.y : r.x, acc);
                    acc = __fma_rn(q == 1 ? -t.y : t.y, q == 1 ? r.x : r.y, acc);
                }
            }
            __syncthreads();
        }
    }
    if (DOT) {
        if (rank != 0) return;
        if (q < 3) {
            acc = warp_sum(acc);
            if (lane == 0) {
                double* p = &d.part[(size_t)(q == 2 ? w.nbx : 0) + w.bx].x;
                p[q == 1] = acc;
                if (q == 2) p[1] = 0.0;
            }
        }
        run_step<false>(d, step, w.nbx, w.ntk);
    }
}

// ------------------------------------------------------------------ FP64, a thread per site
// From site64_min sites per SM on (a wave and a quarter of 256-thread blocks, half of
// that for the few products of l <= 2) there is FP64 work for every SM without a split by component and chain, and the tile
// kernels lose to their barriers, to products formed from vectors loaded once per
// chain, and to the few blocks that 148 registers x 384 threads leave.  The same
// chains in the same order: the same bits.  Measured on GB300 (tracer, us per launch,
// l = 2, tiles / a thread per site): Gram matrix 32^3 x 64 1522 / 776, 16^3 x 32 196 /
// 92, 41,472 sites 69 / 50, 24,576 44 / 29, 16,384 32 / 29; MR step of a double pass 1851 /
// 1136, 158 / 101, 55 / 53, 34 / 30, 24 / 29 (l = 4 at 24,576 sites: 52 / 69); k_update_shifts64 with 8 shifts (W = 32 / 256) 10444 /
// 9183, 628 / 585, 198 / 187, 78 / 87.  At l = 8 and 41,472 sites they draw (507 / 511,
// 119 / 126).  With many shifts a warp per shift is even or better (16^3 x 32, 24
// shifts: 1661 / 1692), as is the tile form of the single-pass MR step (1386 / 1627),
// whose site form takes whole waves of one block per SM (8 shifts: 155,648 sites, 4.0
// waves, 660 / 616; 196,608, 5.05, 832 / 892; 32^3 x 64 8568 / 7940).
constexpr int site64_min(int L) { return L <= 2 ? 160 : 320; }
constexpr int kFewShifts = 16;

// the Gram matrix
template <int L>
__global__ void __launch_bounds__(kThreads, L <= 2 ? 4 : 1)
k_gram_site(const SolverDev* __restrict__ ds, int shifts, const int4* tab) {
    dep_wait();
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, 0)) return;
    const TraceScope trace_(trace_kind<double>(FA_TK_GRAM));
    constexpr int NG = n_gram(L);
    const int V = d.V, n = 12 * V;
    cx<double> acc[NG];
#pragma unroll
    for (int k = 0; k < NG; ++k) acc[k] = czero<double>();
    int s0, s1;
    site_range(V, w.bx, w.nbx, s0, s1);
    for (int s = s0 + threadIdx.x; s < s1; s += kThreads) {
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            cx<double> v[L + 1];
#pragma unroll
            for (int i = 0; i <= L; ++i) v[i] = ldc(d.r64 + (size_t)i * n + (size_t)q * V + s);
            int g = 0;
#pragma unroll
            for (int i = 0; i <= L; ++i)
#pragma unroll
                for (int k = i; k <= L; ++k, ++g) {
                    if (L <= 2 && i == k) {
                        acc[g].r = __fma_rn(v[i].r, v[i].r, acc[g].r);
                        acc[g].r = __fma_rn(v[i].i, v[i].i, acc[g].r);
                    } else {
                        acc[g] = cjfma(v[i], v[k], acc[g]);
                    }
                }
        }
    }
    reduce_store<NG, double>(acc, d.part, w.nbx, w.bx);
    if (last_block(d.st, w.ntk) == LB_LAST) {
        sc_mr_seed<L, false>(d, n_partials<double>(w.nbx), false);
        if (shifts) {
            __syncthreads();
            sc_mr_shifts<L>(d);
        }
    }
}

// the MR update of pass 1
template <int L, bool SHIFTS, bool XS>
__global__ void __launch_bounds__(kThreads)
k_mr_site(const SolverDev* __restrict__ ds, ScalarStep step, const int4* tab) {
    dep_wait();
    const Where w = where<XS>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, 0)) return;
    const TraceScope trace_(trace_kind<double>(FA_TK_MR, XS));
    if (XS && w.bx < 0) {
        mr_shifts<L>(d, [&] {
            __threadfence();   // the new zeta of every thread before the ticket
            run_step<false>(d, step, n_partials<double>(w.nbx), w.ntk);
        });
        return;
    }
    const int V = d.V, n = 12 * V, m = d.st->m;
    cx<double> ng[L + 1];
    ng[0] = czero<double>();
#pragma unroll
    for (int k = 1; k <= L; ++k) ng[k] = negcx<double>(d.rec_gamma[m * (L + 1) + k]);
    double2* store = store_at<double>(d, m);
    cx<double> dots[2] = {czero<double>(), czero<double>()};
    int s0, s1;
    site_range(V, w.bx, w.nbx, s0, s1);
    for (int s = s0 + threadIdx.x; s < s1; s += kThreads) {
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            const size_t e = (size_t)q * V + s;
            cx<double> rv[L + 1];
#pragma unroll
            for (int i = 0; i <= L; ++i) rv[i] = ldc(d.r64 + (size_t)i * n + e);
            if (store != nullptr) {
#pragma unroll
                for (int k = 0; k < L; ++k) __stcs(store + (size_t)slot_mr(L, k) * n + e, make_double2(rv[k].r, rv[k].i));
            }
            if (SHIFTS) {
                for (int sh = 0; sh < d.ns; ++sh) {
                    if (!d.active[sh]) continue;
                    const double2* P = d.prec + ((size_t)sh * d.max_outer + m) * ps_stride(L) + 5 * L;
                    double2* us = d.us + (size_t)sh * (L + 1) * n + e;
                    double2* xs = d.xs + (size_t)sh * n + e;
                    cx<double> xv = ldc(xs), u0 = ldc(us);
#pragma unroll
                    for (int k = 0; k < L; ++k) xv = cfma(tocx<double>(P[1 + k]), rv[k], xv);
#pragma unroll
                    for (int k = 1; k <= L; ++k) u0 = cfma(ng[k], ldc(us + (size_t)k * n), u0);
                    stc(xs, xv);
                    stc(us, cmul(tocx<double>(P[0]), u0));
                }
            }
            if (d.x64 != nullptr) {
#pragma unroll
                for (int k = 1; k <= L; ++k) acc_x1(d.x64 + e, d.rec_gamma[m * (L + 1) + k], rv[k - 1]);
            }
            cx<double> r0 = rv[0], u0 = ldc(d.u64 + e);
#pragma unroll
            for (int k = 1; k <= L; ++k) {
                r0 = cfma(ng[k], rv[k], r0);
                u0 = cfma(ng[k], ldc(d.u64 + (size_t)k * n + e), u0);
            }
            stc(d.r64 + e, r0);
            stc(d.u64 + e, u0);
            const cx<double> t = ldc(d.rt64 + e);
            dots[0] = cjfma(t, r0, dots[0]);
            dots[1].r = __fma_rn(r0.r, r0.r, dots[1].r);
            dots[1].r = __fma_rn(r0.i, r0.i, dots[1].r);
        }
    }
    reduce_store<2, double>(dots, d.part, w.nbx, w.bx);
    run_step<false>(d, step, n_partials<double>(w.nbx), w.ntk);
}

}  // namespace fa
