// Device kernels of the multi-shift BiCGstab(l) solver (single-pass and
// double-pass forms of Sec. 2), shared by solver.cu.
//
// Seed recurrence (BiCGstab(l), Sleijpen-Fokkema, cited in Sec. 2):
//   outer m: rho0 <- -omega rho0; for j = 0..l-1:
//     rho1 = <rt, r_j>, beta = alpha rho1/rho0, rho0 = rho1
//     u_i <- r_i - beta u_i (i <= j);  u_{j+1} = A u_j;  alpha = rho0/<rt, u_{j+1}>
//     r_i <- r_i - alpha u_{i+1} (i <= j);  r_{j+1} = A r_j
//   MR: gamma minimises |r_0 - sum gamma_j r_j| (normal equations, pivoted elimination),
//     r_0 <- r_0 - sum gamma_j r_j, u_0 <- u_0 - sum gamma_j u_j, omega = gamma_l.
// Shifted systems (shift invariance, Sec. 1) carry zeta_s with r^s = r_0/zeta_s:
//   BiCG: zeta_new = (1 + alpha sigma) zeta + (alpha beta/alpha_prev)(zeta' - zeta),
//         alpha_s = alpha zeta/zeta_new, beta_s = beta (zeta'/zeta)^2,
//         u^s_i <- r_old_i/zeta - beta_s u^s_i, u^s_{j+1} <- (r_old_j/zeta - r_j/zeta_new)/alpha_s
//         - sigma u^s_j, x_s <- x_s + alpha_s u^s_0
//   MR:   p_s = 1 - sum gamma_j (-sigma)^j, c_k = sum_{j>k} gamma_j (-sigma)^{j-1-k},
//         x_s <- x_s + sum_k c_k r_k/(zeta p_s), u^s_0 <- (u^s_0 - sum gamma_j u^s_j)/p_s,
//         zeta <- zeta p_s, zeta' <- zeta' p_s.
// All scalars are FP64 and live on the device; vector kernels read the
// current outer iteration m and their scalars from the device record, so
// pass 1, pass 2 and any replay run the same kernels with the same
// arithmetic (explicit fma intrinsics, no contraction by the compiler).
#pragma once

#include "hop64.cuh"
#include "hop_device.cuh"
#include "trace.cuh"

namespace fa {

// ------------------------------------------------------------------ solver state
struct DevState {
    double2 rho0, alpha, omega, alpha_prev;
    double bnorm2, tol2b, theta2b, rnorm2;
    int m;           // current outer iteration
    int done;        // nonzero: pass-1 kernels return at once
    int status;      // fa_status of the solve
    int n_active;    // shifts not frozen
    int n_outer;     // M, set when pass 1 ends
    int switch_req;  // FA_MIXED: head residuals below the switch threshold
    int max_outer;
    unsigned ticket; // blocks of the current reduction that have stored their partials
};

// Per-shift record of pass 1 at outer iteration m (complex FP64):
//   sub-step j: [5j+0] alpha_s, [5j+1] beta_s, [5j+2] 1/zeta, [5j+3] 1/(alpha_s zeta),
//               [5j+4] 1/(alpha_s zeta_new)
//   MR:         [5l] 1/p_s, [5l+1+k] c_k/(zeta p_s), k < l
__host__ __device__ constexpr int ps_stride(int L) { return 6 * L + 1; }
// Pass-2 weights per outer iteration: slot (j, i) of the BiCG sub-step j for the
// occurrence r_i before its update (i <= j), then l MR slots for r_0..r_{l-1}.
__host__ __device__ constexpr int nc_slots(int L) { return L * (L + 1) / 2 + L; }
__host__ __device__ constexpr int slot_old(int j, int i) { return j * (j + 1) / 2 + i; }
__host__ __device__ constexpr int slot_mr(int L, int k) { return L * (L + 1) / 2 + k; }
__host__ __device__ constexpr int n_gram(int L) { return (L + 1) * (L + 2) / 2; }

// Everything one system needs on the device.  Kernels read their system's
// descriptor from an array (ds[blockIdx.y] for site kernels, ds[blockIdx.x]
// for the kernels with one block per system), so one launch serves a batch of
// systems of the same lattice shape; a single solve is a batch of one.
struct SolverDev {
    DevState* st;
    int ns, L, max_outer, V;
    Geom g;
    const double2* links64;
    const float4* links32;
    const float4* linksdf;            // double-float links [4][9][V]
    double diag, ef, eb, bc, scale;   // 4+m, e^{+mu}, e^{-mu}, time-boundary sign, c
    // the same operator scalars rounded to FP32 (multi-RHS sweep): 4+m and -1/2 for the
    // first hop of A, c (4+m) and -c/2 for the second, e^{+-mu}, the boundary sign
    float fdiag1, fhop1, fdiag2, fhop2, fef, feb, fbc;
    const double* sigma;   // [ns]
    const double* omega;   // [ns]
    double2* zeta;         // [ns]
    double2* zeta_p;       // [ns]
    int* active;           // [ns]
    int* iters;            // [ns]
    double2* rec_alpha;    // [max_outer][L]
    double2* rec_beta;     // [max_outer][L]
    double2* rec_gamma;    // [max_outer][L+1]
    // the same scalars as FP32 pairs (hi, lo) per part, which the FP32 and double-float
    // kernels load: a conversion per thread costs more than an element's update
    float4 *rec_alpha4, *rec_beta4, *rec_gamma4;
    double2* prec;         // [ns][max_outer][ps_stride]
    double2* coef;         // [max_outer][nc_slots]
    float4* coef4;         // the same weights as FP32 pairs (hi, lo) per part
    double2* cs;           // [ns][max_outer][nc_slots]   per-shift sweep output
    // seed vectors: r_0..r_l and u_0..u_l contiguous, the shadow vector, scratch
    double2 *r64, *u64, *rt64, *tmp64;
    float4 *r32, *u32, *rt32, *tmp32;
    // pass 2, FP32 and double-float: r_j after sub-step j's update, j < l - 1 (r_j itself
    // keeps the value before it for the MR step; the last one goes to r_l, which the
    // sub-step's second hop overwrites).  In memory that pass 2 does not use: place_rb
    double2* rb64;
    float4* rb32;
    double2* y;            // FP64 [12][V] result
    double2* xs;           // single-pass x_s   [ns][12][V]
    double2* us;           // single-pass u^s_i [ns][l+1][12][V]
    // pseudo-double-pass occurrence stores: outer iteration m is stored in the
    // FP64 store if m < cap64, in the FP32 store if 0 <= m - m0_32 < cap32
    char* store64;
    char* store32;
    int cap64, cap32, m0_32;
    double2* part;         // this system's reduction partials
    // reliable updates: seed solution x (FP64, [12][V], accumulated alongside the
    // recurrence when not null) and the packed source b (FP64)
    double2* x64;
    const double2* b64;
    // nonzero: max_outer is the planned number of outer iterations, reaching it
    // freezes the remaining shifts instead of failing (fixed-cost runs)
    int fixed_iters;
};

template <typename R> struct Vec;
template <> struct Vec<double> {
    using T = double2;
    __device__ static T* r(const SolverDev& d) { return d.r64; }
    __device__ static T* u(const SolverDev& d) { return d.u64; }
    __device__ static T* rt(const SolverDev& d) { return d.rt64; }
    __device__ static T* tmp(const SolverDev& d) { return d.tmp64; }
    __device__ static T* rb(const SolverDev&) { return nullptr; }
    __device__ static LinkView<double> links(const SolverDev& d) { return {d.links64, d.V}; }
};
// double-float vectors live in the FP64 buffers (same bytes: one float4 per complex)
template <> struct Vec<df> {
    using T = float4;
    __device__ static T* r(const SolverDev& d) { return reinterpret_cast<T*>(d.r64); }
    __device__ static T* u(const SolverDev& d) { return reinterpret_cast<T*>(d.u64); }
    __device__ static T* rt(const SolverDev& d) { return reinterpret_cast<T*>(d.rt64); }
    __device__ static T* tmp(const SolverDev& d) { return reinterpret_cast<T*>(d.tmp64); }
    __device__ static T* rb(const SolverDev& d) { return reinterpret_cast<T*>(d.rb64); }
    __device__ static LinkView<df> links(const SolverDev& d) { return {d.linksdf, d.V}; }
};
template <> struct Vec<float> {
    using T = float4;
    __device__ static T* r(const SolverDev& d) { return d.r32; }
    __device__ static T* u(const SolverDev& d) { return d.u32; }
    __device__ static T* rt(const SolverDev& d) { return d.rt32; }
    __device__ static T* tmp(const SolverDev& d) { return d.tmp32; }
    __device__ static T* rb(const SolverDev& d) { return d.rb32; }
    __device__ static LinkView<float> links(const SolverDev& d) { return {d.links32, d.V}; }
};

// Position of a block in a launch that serves one or several systems.  Without
// a work table: system blockIdx.y, block blockIdx.x of gridDim.x (every system of
// the launch has the same lattice shape).  With a table (systems of different
// lattice shapes in one launch): tab[blockIdx.x] = (system, block within the
// system, vector blocks of the system, blocks of the system in this launch =
// the tickets of its reductions).  XS kernels: block -1 is the system's shift
// block (block 0 of the launch without a table).
struct Where {
    int sys, bx, nbx, ntk;
};
template <bool XS>
__device__ __forceinline__ Where where(const int4* tab) {
    if (tab != nullptr) {
        const int4 t = tab[blockIdx.x];
        return {t.x, t.y, t.z, t.w};
    }
    return {(int)blockIdx.y, (int)blockIdx.x - (XS ? 1 : 0), (int)gridDim.x - (XS ? 1 : 0), (int)gridDim.x};
}

// pass 1: the system has finished (converged, failed or max_outer);
// pass 2: the system has replayed all its outer iterations.
__device__ __forceinline__ bool sys_idle(const SolverDev& d, int pass2) {
    return pass2 ? (d.st->m >= d.st->n_outer) : (d.st->done != 0);
}

// ------------------------------------------------------------------ chunk IO
// A chunk is the vector unit of one load: FP64 one complex (double2, 12 per
// site), FP32 two complex (float4, 6 per site).
template <typename R> struct Ch;
template <> struct Ch<double> {
    static constexpr int W = 1, N = 12;
    using T = double2;
    cx<double> c[1];
    __device__ __forceinline__ static Ch ld(const T* b, int q, int V, int s) {
        double2 t = b[(size_t)q * V + s];
        Ch r; r.c[0] = {t.x, t.y}; return r;
    }
    __device__ __forceinline__ void stv(T* b, int q, int V, int s) const {
        b[(size_t)q * V + s] = make_double2(c[0].r, c[0].i);
    }
    // evict-first store / load (occurrence store: written once, read once by the gather)
    __device__ __forceinline__ void stv_cs(T* b, int q, int V, int s) const {
        __stcs(b + (size_t)q * V + s, make_double2(c[0].r, c[0].i));
    }
    __device__ __forceinline__ static Ch ld_cs(const T* b, int q, int V, int s) {
        double2 t = __ldcs(b + (size_t)q * V + s);
        Ch r; r.c[0] = {t.x, t.y}; return r;
    }
};
template <> struct Ch<df> {
    static constexpr int W = 1, N = 12;
    using T = float4;
    cx<df> c[1];
    __device__ __forceinline__ static Ch ld(const T* b, int q, int V, int s) {
        float4 t = b[(size_t)q * V + s];
        Ch r; r.c[0] = {df(t.x, t.y), df(t.z, t.w)}; return r;
    }
    __device__ __forceinline__ void stv(T* b, int q, int V, int s) const {
        b[(size_t)q * V + s] = make_float4(c[0].r.hi, c[0].r.lo, c[0].i.hi, c[0].i.lo);
    }
    __device__ __forceinline__ void stv_cs(T* b, int q, int V, int s) const {
        __stcs(b + (size_t)q * V + s, make_float4(c[0].r.hi, c[0].r.lo, c[0].i.hi, c[0].i.lo));
    }
    __device__ __forceinline__ static Ch ld_cs(const T* b, int q, int V, int s) {
        float4 t = __ldcs(b + (size_t)q * V + s);
        Ch r; r.c[0] = {df(t.x, t.y), df(t.z, t.w)}; return r;
    }
};
template <> struct Ch<float> {
    static constexpr int W = 2, N = 6;
    using T = float4;
    cx<float> c[2];
    __device__ __forceinline__ static Ch ld(const T* b, int q, int V, int s) {
        float4 t = b[(size_t)q * V + s];
        Ch r; r.c[0] = {t.x, t.y}; r.c[1] = {t.z, t.w}; return r;
    }
    __device__ __forceinline__ void stv(T* b, int q, int V, int s) const {
        b[(size_t)q * V + s] = make_float4(c[0].r, c[0].i, c[1].r, c[1].i);
    }
    __device__ __forceinline__ void stv_cs(T* b, int q, int V, int s) const {
        __stcs(b + (size_t)q * V + s, make_float4(c[0].r, c[0].i, c[1].r, c[1].i));
    }
    __device__ __forceinline__ static Ch ld_cs(const T* b, int q, int V, int s) {
        float4 t = __ldcs(b + (size_t)q * V + s);
        Ch r; r.c[0] = {t.x, t.y}; r.c[1] = {t.z, t.w}; return r;
    }
};

template <typename R> __device__ __forceinline__ size_t vstride(const SolverDev& d) {
    return (size_t)Ch<R>::N * d.V;
}
// pass 2: r_j after its own update
template <typename R> __device__ __forceinline__ typename Ch<R>::T* rb_at(const SolverDev& d, int j) {
    return j == d.L - 1 ? Vec<R>::r(d) + (size_t)d.L * vstride<R>(d) : Vec<R>::rb(d) + (size_t)j * vstride<R>(d);
}

// store slots of outer iteration m, or nullptr when m is not stored
template <typename R>
__device__ __forceinline__ typename Ch<R>::T* store_at(const SolverDev& d, int m) {
    const size_t per = (size_t)nc_slots(d.L) * vstride<R>(d) * sizeof(typename Ch<R>::T);
    if (sizeof(R) == 8) {
        if (m < d.cap64) return reinterpret_cast<typename Ch<R>::T*>(d.store64 + (size_t)m * per);
    } else {
        const int k = m - d.m0_32;
        if (d.m0_32 >= 0 && k >= 0 && k < d.cap32) return reinterpret_cast<typename Ch<R>::T*>(d.store32 + (size_t)k * per);
    }
    return nullptr;
}

template <typename R> __device__ __forceinline__ cx<R> tocx(double2 v) { return {fromdbl<R>(v.x), fromdbl<R>(v.y)}; }
template <typename R> __device__ __forceinline__ cx<R> negcx(double2 v) {
    return {fromdbl<R>(-v.x), fromdbl<R>(-v.y)};
}
// scalar k of a record (or pass-2 weight) in R from its FP64 and FP32-pair copies:
// the same value as tocx<R>(cf[k]) without an FP64 conversion per thread
template <typename R> __device__ __forceinline__ cx<R> weight(const double2* cf, const float4* cf4, size_t k) {
    if constexpr (std::is_same<R, double>::value) {
        return tocx<double>(cf[k]);
    } else {
        const float4 t = cf4[k];
        if constexpr (std::is_same<R, float>::value) return {t.x, t.z};
        else return {df(t.x, t.y), df(t.z, t.w)};
    }
}
template <typename R> __device__ __forceinline__ cx<R> nweight(const double2* cf, const float4* cf4, size_t k) {
    const cx<R> t = weight<R>(cf, cf4, k);
    return {-t.r, -t.i};
}
// a record's FP64 scalar and its FP32-pair copy
__device__ __forceinline__ void put_scalar(double2* rec, float4* rec4, size_t k, dcx v) {
    rec[k] = make_double2(v.r, v.i);
    const float2 r = d2df_int(v.r), i = d2df_int(v.i);
    rec4[k] = make_float4(r.x, r.y, i.x, i.y);
}

// x (FP64) += a v for the W components of chunk q
template <typename R>
__device__ __forceinline__ void acc_x(double2* x, int q, int V, int s, double2 a, const Ch<R>& v) {
#pragma unroll
    for (int w = 0; w < Ch<R>::W; ++w) {
        double2* p = x + (size_t)(q * Ch<R>::W + w) * V + s;
        double2 t = *p;
        const double vr = todbl(v.c[w].r), vi = todbl(v.c[w].i);
        t.x = __fma_rn(a.x, vr, t.x);
        t.x = __fma_rn(-a.y, vi, t.x);
        t.y = __fma_rn(a.x, vi, t.y);
        t.y = __fma_rn(a.y, vr, t.y);
        *p = t;
    }
}

// x (FP64) += a v for one complex number
__device__ __forceinline__ void acc_x1(double2* x, double2 a, cx<double> v) {
    double2 t = *x;
    t.x = __fma_rn(a.x, v.r, t.x);
    t.x = __fma_rn(-a.y, v.i, t.x);
    t.y = __fma_rn(a.x, v.i, t.y);
    t.y = __fma_rn(a.y, v.r, t.y);
    *x = t;
}

template <typename R> __device__ __forceinline__ cx<double> dbl(cx<R> v) { return {todbl(v.r), todbl(v.i)}; }

// ------------------------------------------------------------------ deferred updates
// The updates of i < j that the sub-steps leave out (see vec_tile.cuh), for one
// 16-byte chunk q of site s, in the order of the sub-steps j = 1..L-1:
//   u_i <- r_i - beta_j u_i, then r_i <- r_i - alpha_j u_{i+1}   (i < j),
// from r_i and u_i as their own sub-step i left them (u_j and r_j enter at step j).
template <typename R, int L> struct StepScalars {   // -alpha_j, -beta_j of the outer iteration
    cx<R> na[L], nb[L];
    __device__ __forceinline__ StepScalars(const SolverDev& d, int m) {
#pragma unroll
        for (int j = 0; j < L; ++j) {
            na[j] = nweight<R>(d.rec_alpha, d.rec_alpha4, m * L + j);
            nb[j] = nweight<R>(d.rec_beta, d.rec_beta4, m * L + j);
        }
    }
};
template <typename R, int NU>
__device__ __forceinline__ void defer_u(cx<R> nb, const Ch<R>* r, Ch<R> (&u)[NU], int i) {
#pragma unroll
    for (int w = 0; w < Ch<R>::W; ++w) u[i].c[w] = cfma(nb, u[i].c[w], r[i].c[w]);
}
template <typename R, int NU>
__device__ __forceinline__ void defer_r(cx<R> na, Ch<R>* r, const Ch<R> (&u)[NU], int i) {
#pragma unroll
    for (int w = 0; w < Ch<R>::W; ++w) r[i].c[w] = cfma(na, u[i + 1].c[w], r[i].c[w]);
}
// pass 1: with the occurrences of stored iterations and the seed solution x
template <typename R, int L, int NU>
__device__ __forceinline__ void deferred(const SolverDev& d, int m, const StepScalars<R, L>& sc, Ch<R> (&r)[L + 1],
                                         Ch<R> (&u)[NU], typename Ch<R>::T* store, int q, int s) {
    const size_t vs = vstride<R>(d);
    if (d.x64 != nullptr) acc_x<R>(d.x64, q, d.V, s, d.rec_alpha[m * L], u[0]);
#pragma unroll
    for (int j = 1; j < L; ++j) {
#pragma unroll
        for (int i = 0; i < j; ++i) defer_u(sc.nb[j], r, u, i);
        if (d.x64 != nullptr) acc_x<R>(d.x64, q, d.V, s, d.rec_alpha[m * L + j], u[0]);
#pragma unroll
        for (int i = 0; i < j; ++i) {
            if (store != nullptr) r[i].stv_cs(store + slot_old(j, i) * vs, q, d.V, s);
            defer_r(sc.na[j], r, u, i);
        }
    }
}
// r alone (the Gram matrix; u_0 is not needed)
template <typename R, int L>
__device__ __forceinline__ void deferred_r(const StepScalars<R, L>& sc, Ch<R> (&r)[L + 1], Ch<R> (&u)[L]) {
#pragma unroll
    for (int j = 1; j < L; ++j) {
#pragma unroll
        for (int i = 1; i < j; ++i) defer_u(sc.nb[j], r, u, i);
#pragma unroll
        for (int i = 0; i < j; ++i) defer_r(sc.na[j], r, u, i);
    }
}
// y += t for the W complex numbers of a chunk
template <typename R>
__device__ __forceinline__ void add_y(double2 (&y)[Ch<R>::W], const cx<R> (&t)[Ch<R>::W]) {
#pragma unroll
    for (int w = 0; w < Ch<R>::W; ++w) {
        y[w].x = __dadd_rn(y[w].x, todbl(t[w].r));
        y[w].y = __dadd_rn(y[w].y, todbl(t[w].i));
    }
}
// pass 2: r holds r_j before sub-step j's update (j < L), u the vectors as
// their sub-steps left them; y += the weighted occurrences of every sub-step
template <typename R, int L>
__device__ __forceinline__ void deferred_acc(const SolverDev& d, int m, const StepScalars<R, L>& sc, Ch<R> (&r)[L + 1],
                                             Ch<R> (&u)[L + 1], int q, int s, double2 (&y)[Ch<R>::W]) {
    const size_t vs = vstride<R>(d), cf0 = (size_t)m * nc_slots(L);
#pragma unroll
    for (int j = 0; j < L; ++j) {
#pragma unroll
        for (int i = 0; i < j; ++i) defer_u(sc.nb[j], r, u, i);
        if (d.x64 != nullptr) acc_x<R>(d.x64, q, d.V, s, d.rec_alpha[m * L + j], u[0]);
        cx<R> t[Ch<R>::W];
#pragma unroll
        for (int w = 0; w < Ch<R>::W; ++w) t[w] = czero<R>();
#pragma unroll
        for (int i = 0; i <= j; ++i) {
            const cx<R> c = weight<R>(d.coef, d.coef4, cf0 + slot_old(j, i));
#pragma unroll
            for (int w = 0; w < Ch<R>::W; ++w) t[w] = cfma(c, r[i].c[w], t[w]);
        }
        add_y<R>(y, t);
#pragma unroll
        for (int i = 0; i < j; ++i) defer_r(sc.na[j], r, u, i);
        // r_j after its own update: rb_j, formed again where u_{j+1} is still what the sweep left
        if (j == L - 1) defer_r(sc.na[j], r, u, j);
        else r[j] = Ch<R>::ld(rb_at<R>(d, j), q, d.V, s);
    }
}
// the MR step's occurrences r_0..r_{L-1}
template <typename R, int L>
__device__ __forceinline__ void acc_mr(const SolverDev& d, int m, const Ch<R> (&r)[L + 1], double2 (&y)[Ch<R>::W]) {
    const size_t cf0 = (size_t)m * nc_slots(L);
    cx<R> t[Ch<R>::W];
#pragma unroll
    for (int w = 0; w < Ch<R>::W; ++w) t[w] = czero<R>();
#pragma unroll
    for (int k = 0; k < L; ++k) {
        const cx<R> c = weight<R>(d.coef, d.coef4, cf0 + slot_mr(L, k));
#pragma unroll
        for (int w = 0; w < Ch<R>::W; ++w) t[w] = cfma(c, r[k].c[w], t[w]);
    }
    add_y<R>(y, t);
}

// ------------------------------------------------------------------ scalar steps
// The scalar steps of the recurrence run inside the vector kernels, in two
// parts.  The seed part (beta, alpha, the MR coefficients gamma, convergence)
// runs in the last block of the reduction kernel whose partials it reads: each
// block stores its partials, fences and takes a ticket, and the block holding
// the last ticket sums all partials in a fixed order (so the result does not
// depend on which block finished last) and runs the step.  The shift part (the
// zeta recurrences and the per-shift scalars of every BiCG sub-step and MR
// step) is not needed by the next seed-vector kernel: in the double-pass forms
// it runs in an extra block 0 of that next kernel, beside its vector blocks, or
// of the sweep after it (k_hop1_split, STEP_SHIFTS).
// Single-pass solves consume the shift scalars at once and run both parts in
// the last block.
//
// FP64 instructions are scarce on this part (one warp instruction occupies a
// sub-partition's FP64 pipe for tens of cycles, a division for hundreds), so
// the steps use fused multiply-adds, one real division per complex inverse,
// and reuse inverses between the per-shift scalars.
//
// The step's code runs once per launch, in whichever block takes the last
// ticket, so its instructions are usually not in that SM's instruction cache:
// on GB300 (16^3 x 32 solve) fetching them from L2 took most of the last
// block's time (a reduction of 2 x 512 partials: 4.6 us with cold code, 1.3 us
// with the same code run once before on other data).  So the blocks that take
// one of the last kWarmTickets tickets, other than the last, run the step as a
// dry run (no partial loads, no stores; `dry` below) before they exit: the
// blocks that share an SM with the last block finish shortly before it, and
// their dry runs bring the code into that SM's instruction cache while the
// last block still works.  Results do not change: a dry run reads state but
// writes nothing outside its own shared memory.  Only in launches of at most
// about one wave (8 blocks per SM): in a longer launch a block that lingers
// for its dry run holds back the blocks still waiting for a slot (the
// 72-system batch, one launch for all systems, measured 3-10 % slower; the
// double-float Gram matrix with its row groups, us with / without: 16^3 x 32,
// l = 8, 5 x 512 blocks 601 / 405, 32^3 x 64, l = 4, 3 x 1216 1002 / 995).
constexpr unsigned kWarmTickets = 1024, kWarmSkip = 32;
enum { LB_NONE = 0, LB_WARM = 1, LB_LAST = 2 };
__device__ __forceinline__ unsigned sm_count_dev() {
    unsigned n;
    asm("mov.u32 %0, %%nsmid;" : "=r"(n));
    return n;
}
__device__ __forceinline__ int last_block(DevState* S, int ntickets) {
    __shared__ int is_last;
    dep_launch();
    __syncthreads();
    if (threadIdx.x == 0) {
        // one or several threads stored the block's partials; the fence is cumulative
        // over what the barrier ordered before it (release), and the one after the
        // last ticket orders the reads that follow (acquire; the other threads
        // read the partials after the barrier, from L2)
        __threadfence();
        const unsigned t = atomicAdd(&S->ticket, 1u);
        // (the last kWarmSkip before the last block run no dry run: they would
        // end after it on an SM whose code is still cold)
        const bool one_wave = (unsigned long long)gridDim.x * gridDim.y * gridDim.z <= 8u * sm_count_dev();
        is_last = t == (unsigned)ntickets - 1u ? LB_LAST
                  : (one_wave && t + kWarmTickets >= (unsigned)ntickets && t + 1u + kWarmSkip < (unsigned)ntickets
                         ? LB_WARM
                         : LB_NONE);
        if (is_last == LB_LAST) {
            S->ticket = 0u;   // every block of this launch has taken its ticket
            __threadfence();
        }
    }
    __syncthreads();
    return is_last;
}

__device__ __forceinline__ dcx zneg(dcx a) { return {-a.r, -a.i}; }   // a sign flip, free on FMA operands
__device__ __forceinline__ dcx zmul(dcx a, dcx b) {
    return {__fma_rn(a.r, b.r, -__dmul_rn(a.i, b.i)), __fma_rn(a.r, b.i, __dmul_rn(a.i, b.r))};
}
__device__ __forceinline__ dcx zfma(dcx a, dcx b, dcx c) {   // a b + c
    return {__fma_rn(a.r, b.r, __fma_rn(-a.i, b.i, c.r)), __fma_rn(a.r, b.i, __fma_rn(a.i, b.r, c.i))};
}
__device__ __forceinline__ dcx zrfma(double a, dcx b, dcx c) { return {__fma_rn(a, b.r, c.r), __fma_rn(a, b.i, c.i)}; }
__device__ __forceinline__ dcx zscale(double a, dcx b) { return {__dmul_rn(a, b.r), __dmul_rn(a, b.i)}; }
__device__ __forceinline__ dcx zsub(dcx a, dcx b) { return {__dsub_rn(a.r, b.r), __dsub_rn(a.i, b.i)}; }
__device__ __forceinline__ double zabs2(dcx a) { return __fma_rn(a.r, a.r, __dmul_rn(a.i, a.i)); }
__device__ __forceinline__ dcx zconj_scale(double a, dcx b) { return {__dmul_rn(a, b.r), -__dmul_rn(a, b.i)}; }
__device__ __forceinline__ dcx zinv(dcx a) { return zconj_scale(1.0 / zabs2(a), a); }
__device__ __forceinline__ bool zfinite(dcx a) { return isfinite(a.r) && isfinite(a.i); }
// 2^-floor(e/2) for x = f 2^e (x > 0, normal): x * result^2 lies in [1, 4).
// Integer work on the exponent bits only.
__device__ __forceinline__ double pow2_rsqrt(double x) {
    const long long bits = __double_as_longlong(x);
    const int e = (int)((bits >> 52) & 0x7ff) - 1023;
    const int h = e >= 0 ? e / 2 : -((1 - e) / 2);     // floor(e / 2)
    return __longlong_as_double((long long)(1023 - h) << 52);
}
// 1/p and 1/q (p, q > 0) from one division while p q stays well inside the
// FP64 range, else from two
__device__ __forceinline__ void recip2(double p, double q, double& ip, double& iq) {
    const double pq = __dmul_rn(p, q);
    if (pq > 1e-280 && pq < 1e280) {
        const double r = 1.0 / pq;
        ip = __dmul_rn(q, r);
        iq = __dmul_rn(p, r);
    } else {
        ip = 1.0 / p;
        iq = 1.0 / q;
    }
}

// Sums of the nblk partials of slots 0..ns-1 into out[0..ns-1], fixed order:
// each slot is split into four quarters, one warp each (consecutive warps sit
// on different sub-partitions), summed by the lanes in strided order and a
// shuffle tree; the quarters are then added in order.  Partials are read from
// L2 (other blocks of the same launch stored them).  DFP: the partials are
// FP32 pairs (float4: re.hi, re.lo, im.hi, im.lo; the FP32 and double-float
// kernels store them so) and are summed in double-float on the FP32 pipe;
// otherwise FP64 values summed in FP64.
template <typename R> constexpr bool dfp_of() { return !std::is_same<R, double>::value; }

// FP64 partials are those of warps (32-site tiles), nblk of them; eight at a
// time are first added in the order of a warp shuffle tree over eight lanes,
// and the sums of those 256-site groups are what is split into quarters.
//
// dry: warp 0 runs the code of one quarter once, every load predicated off
// (the sums are 0); the other warps only meet the barriers.
__device__ __forceinline__ double2 tile_group(const double2* pd, int i, int n) {
    double2 v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = 8 * i + t < n ? __ldcg(pd + 8 * i + t) : make_double2(0.0, 0.0);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int t = 0; t < o; ++t) {
            v[t].x = __dadd_rn(v[t].x, v[t + o].x);
            v[t].y = __dadd_rn(v[t].y, v[t + o].y);
        }
    return v[0];
}
template <int NSMAX, bool DFP>
__device__ __forceinline__ void reduce_slots(const double2* part, int nblk, int ns, dcx* out, bool dry = false) {
    __shared__ double2 qs[4 * NSMAX];
    __shared__ float4 qf[4 * NSMAX];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int npart = DFP ? nblk : (nblk + 7) >> 3;
    const int per = (npart + 3) >> 2;
    const int ntask = dry ? 1 : 4 * ns;
    if (dry && (int)threadIdx.x < 4 * ns) {   // the quarters a dry run leaves out
        qs[threadIdx.x] = make_double2(0.0, 0.0);
        qf[threadIdx.x] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    // Several slots (the Gram matrix) and quarters of at most 256 partials: each
    // warp takes two quarters at a time, u and u + nw, with the sixteen loads in
    // flight together (the loads were the time: six rounds of them for 6 x 1024
    // partials in a 128-thread block).  The additions of each quarter are those
    // of the loop below, in the same order.  A dry run takes this path too (its
    // code is the one to bring into the instruction cache).
    int u_first = warp;
    if constexpr (DFP && NSMAX >= 3) {
        if (per <= 256) {
            for (int u = warp; u < ntask; u += 2 * nw) {
                const int u2 = u + nw;
                const bool two = u2 < ntask;
                const int i0 = (u & 3) * per, i1 = dry ? i0 : min(nblk, i0 + per);
                const int j0 = (u2 & 3) * per, j1 = (two && !dry) ? min(nblk, j0 + per) : j0;
                const float4* pf = reinterpret_cast<const float4*>(part) + (size_t)(u >> 2) * nblk;
                const float4* pg = reinterpret_cast<const float4*>(part) + (size_t)(u2 >> 2) * nblk;
                float4 v[8], x[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int i = i0 + lane + 32 * t, j = j0 + lane + 32 * t;
                    v[t] = i < i1 ? __ldcg(pf + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    x[t] = j < j1 ? __ldcg(pg + j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                }
                df a(0.0f), b(0.0f), c(0.0f), e(0.0f);
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    a = addR(a, df(v[t].x, v[t].y));
                    b = addR(b, df(v[t].z, v[t].w));
                    c = addR(c, df(x[t].x, x[t].y));
                    e = addR(e, df(x[t].z, x[t].w));
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    a = addR(a, shfl_down_df(a, o));
                    b = addR(b, shfl_down_df(b, o));
                    c = addR(c, shfl_down_df(c, o));
                    e = addR(e, shfl_down_df(e, o));
                }
                if (lane == 0) {
                    qf[u] = make_float4(a.hi, a.lo, b.hi, b.lo);
                    if (two) qf[u2] = make_float4(c.hi, c.lo, e.hi, e.lo);
                }
            }
            u_first = ntask;   // every quarter done
        }
    }
    for (int u = u_first; u < ntask; u += nw) {
        const int k = u >> 2;
        const int i0 = (u & 3) * per, i1 = dry ? i0 : min(npart, i0 + per);
        if constexpr (DFP) {
            const int iend = dry ? i0 + 32 : i1;
            const float4* pf = reinterpret_cast<const float4*>(part) + (size_t)k * nblk;
            df a(0.0f), b(0.0f);
            // eight loads in flight per lane before the adds (zero padding
            // leaves the sums unchanged)
            for (int ib = i0 + lane; ib < iend; ib += 32 * 8) {
                float4 v[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int i = ib + 32 * t;
                    v[t] = i < i1 ? __ldcg(pf + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                }
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    a = addR(a, df(v[t].x, v[t].y));
                    b = addR(b, df(v[t].z, v[t].w));
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a = addR(a, shfl_down_df(a, o));
                b = addR(b, shfl_down_df(b, o));
            }
            if (lane == 0) qf[u] = make_float4(a.hi, a.lo, b.hi, b.lo);
        } else {
            const double2* pd = part + (size_t)k * nblk;
            double a = 0.0, b = 0.0;
            for (int i = i0 + lane; i < i1; i += 32) {
                const double2 v = tile_group(pd, i, nblk);
                a = __dadd_rn(a, v.x);
                b = __dadd_rn(b, v.y);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a = __dadd_rn(a, __shfl_down_sync(0xffffffffu, a, o));
                b = __dadd_rn(b, __shfl_down_sync(0xffffffffu, b, o));
            }
            if (lane == 0) qs[u] = make_double2(a, b);
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < ns; k += blockDim.x) {
        if constexpr (DFP) {
            df a(0.0f), b(0.0f);
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {
                const float4 t = qf[4 * k + q];
                a = addR(a, df(t.x, t.y));
                b = addR(b, df(t.z, t.w));
            }
            out[k] = {todbl(a), todbl(b)};
        } else {
            const double2 q0 = qs[4 * k], q1 = qs[4 * k + 1], q2 = qs[4 * k + 2], q3 = qs[4 * k + 3];
            out[k] = {__dadd_rn(__dadd_rn(q0.x, q1.x), __dadd_rn(q2.x, q3.x)),
                      __dadd_rn(__dadd_rn(q0.y, q1.y), __dadd_rn(q2.y, q3.y))};
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void fail(DevState* S, int code) {
    if (S->status == FA_OK) S->status = code;
    S->done = 1;
}

// start of pass 1: partials hold <rt, r0> and |r0|^2 with r0 = rt = b
template <bool DFP>
__device__ __noinline__ void sc_init(const SolverDev& d, int nblk, double tol, double theta) {
    DevState* S = d.st;
    __shared__ dcx red[2];
    reduce_slots<2, DFP>(d.part, nblk, 2, red);
    const dcx rtr = red[0];
    const double bb = red[1].r;
    for (int sh = threadIdx.x; sh < d.ns; sh += blockDim.x) {
        d.zeta[sh] = pk(mk(1.0));
        d.zeta_p[sh] = pk(mk(1.0));
        d.active[sh] = 1;
        d.iters[sh] = 0;
    }
    if (threadIdx.x == 0) {
        S->bnorm2 = bb;
        S->tol2b = tol * tol * bb;
        S->theta2b = theta * theta * bb;
        S->rnorm2 = bb;
        S->m = 0;
        S->done = 0;
        S->status = FA_OK;
        S->n_active = d.ns;
        S->n_outer = 0;
        S->switch_req = 0;
        S->max_outer = d.max_outer;
        S->omega = pk(mk(1.0));
        S->alpha = pk(mk(0.0));
        S->alpha_prev = pk(mk(1.0));
        // first BiCG sub-step: rho0 <- -omega rho0 with rho0 = 1; beta = alpha rho1/rho0 = 0
        S->rho0 = pk(rtr);
        put_scalar(d.rec_beta, d.rec_beta4, 0, mk(0.0));
        if (!(bb > 0.0) || !isfinite(bb)) fail(S, FA_EINVAL);
    }
}

// beta of BiCG sub-step j >= 1 from rho1 = <rt, r_j>, by one thread
__device__ __forceinline__ void seed_beta(const SolverDev& d, int j, int m, dcx rho0, dcx alpha, dcx rho1) {
    DevState* S = d.st;
    if (zabs2(rho0) == 0.0) { fail(S, FA_EBREAKDOWN); return; }
    const dcx beta = zmul(zmul(alpha, rho1), zinv(rho0));
    if (!zfinite(beta)) { fail(S, FA_ENONFINITE); return; }
    S->rho0 = pk(rho1);
    put_scalar(d.rec_beta, d.rec_beta4, m * d.L + j, beta);
}
// alpha of BiCG sub-step j from den = <rt, u_{j+1}>, by one thread
__device__ __forceinline__ void seed_alpha(const SolverDev& d, int j, int m, dcx rho0, dcx den) {
    DevState* S = d.st;
    if (zabs2(den) == 0.0) { fail(S, FA_EBREAKDOWN); return; }
    const dcx alpha = zmul(rho0, zinv(den));
    if (!zfinite(alpha)) { fail(S, FA_ENONFINITE); return; }
    put_scalar(d.rec_alpha, d.rec_alpha4, m * d.L + j, alpha);
    S->alpha = pk(alpha);
    S->alpha_prev = pk(alpha);
}

// beta of BiCG sub-step j >= 1 from partials of <rt, r_j>
template <bool DFP>
__device__ __noinline__ void sc_beta(const SolverDev& d, int j, int nblk, bool dry) {
    DevState* S = d.st;
    // the state loads are issued with the partial loads and consumed after the
    // reduction (one memory round trip; the done flag only matters then)
    const int done = S->done, m = S->m;
    const dcx rho0 = ld(S->rho0), alpha = ld(S->alpha);
    __shared__ dcx red[1];
    reduce_slots<1, DFP>(d.part, nblk, 1, red, dry);
    if (done) return;
    if (threadIdx.x == 0) {
        const dcx rho1 = red[0];
        if (zabs2(rho0) == 0.0) { if (!dry) fail(S, FA_EBREAKDOWN); return; }
        const dcx beta = zmul(zmul(alpha, rho1), zinv(rho0));
        if (!zfinite(beta)) { if (!dry) fail(S, FA_ENONFINITE); return; }
        if (dry) { red[0] = beta; return; }   // (kept, so that the arithmetic stays on the dry path)
        S->rho0 = pk(rho1);
        put_scalar(d.rec_beta, d.rec_beta4, m * d.L + j, beta);
    }
}

// alpha of BiCG sub-step j from partials of <rt, u_{j+1}> (seed part)
template <bool DFP>
__device__ __noinline__ void sc_alpha_seed(const SolverDev& d, int j, int nblk, bool dry) {
    DevState* S = d.st;
    const int done = S->done, m = S->m;
    const dcx rho0 = ld(S->rho0);
    __shared__ dcx red[1];
    reduce_slots<1, DFP>(d.part, nblk, 1, red, dry);
    if (done) return;
    if (threadIdx.x == 0) {
        const dcx den = dry ? mk(1.0) : red[0];
        if (zabs2(den) == 0.0) { fail(S, FA_EBREAKDOWN); return; }
        const dcx alpha = zmul(rho0, zinv(den));
        if (!zfinite(alpha)) { if (!dry) fail(S, FA_ENONFINITE); return; }
        if (dry) { red[0] = alpha; return; }
        put_scalar(d.rec_alpha, d.rec_alpha4, m * d.L + j, alpha);
        S->alpha = pk(alpha);
        S->alpha_prev = pk(alpha);
    }
}

// Shift part of BiCG sub-step j of the current outer iteration, from the
// recorded alpha, beta and the previous sub-step's alpha:
//   zeta_new = (1 + sigma alpha) zeta + (alpha beta / alpha_prev)(zeta' - zeta)
//   alpha_s = alpha zeta / zeta_new,  beta_s = beta (zeta' / zeta)^2
// and the weights 1/zeta, 1/(alpha_s zeta) = zeta_new / (alpha zeta^2),
// 1/(alpha_s zeta_new) = 1/(alpha zeta) that the sweep and the single-pass
// shift updates use.  One division per shift (recip2).
__device__ __noinline__ void sc_alpha_shifts(const SolverDev& d, int j) {
    DevState* S = d.st;
    if (S->done) return;
    const int m = S->m;
    const int t = m * d.L + j;
    const dcx alpha = ld(d.rec_alpha[t]);
    const dcx beta = ld(d.rec_beta[t]);
    const dcx aprev = t > 0 ? ld(d.rec_alpha[t - 1]) : mk(1.0);
    // 1/alpha and 1/alpha_prev from one division
    double ina, inp;
    recip2(zabs2(alpha), zabs2(aprev), ina, inp);
    const dcx inv_a = zconj_scale(ina, alpha);
    const dcx inv_p = zconj_scale(inp, aprev);
    const dcx c1 = zmul(zmul(alpha, beta), inv_p);
    for (int sh = threadIdx.x; sh < d.ns; sh += blockDim.x) {
        if (!d.active[sh]) continue;
        const double sg = d.sigma[sh];
        const dcx z = ld(d.zeta[sh]), zp = ld(d.zeta_p[sh]);
        const dcx zs = zrfma(sg, zmul(alpha, z), z);            // (1 + sigma alpha) zeta
        const dcx zn = zfma(c1, zsub(zp, z), zs);
        const double nzn = zabs2(zn);
        double izn, iz;
        recip2(nzn, zabs2(z), izn, iz);
        const dcx inv_zn = zconj_scale(izn, zn);
        const dcx inv_z = zconj_scale(iz, z);
        const dcx as = zmul(zmul(alpha, z), inv_zn);
        const dcx r = zmul(zp, inv_z);
        const dcx bs = zmul(beta, zmul(r, r));
        const dcx iaz = zmul(inv_a, inv_z);                       // 1/(alpha zeta)
        double2* P = d.prec + ((size_t)sh * d.max_outer + m) * ps_stride(d.L) + 5 * j;
        P[0] = pk(as);
        P[1] = pk(bs);
        P[2] = pk(inv_z);
        P[3] = pk(zmul(zn, zmul(iaz, inv_z)));
        P[4] = pk(iaz);
        if (!(nzn > 0.0) || !isfinite(izn) || !zfinite(as) || !zfinite(zn)) fail(S, FA_ENONFINITE);
        d.zeta_p[sh] = pk(z);
        d.zeta[sh] = pk(zn);
    }
}

// MR coefficients gamma (seed part) from the Gram partials: diagonally scaled
// normal equations, Gaussian elimination with partial pivoting.
template <int L, bool DFP>
__device__ __noinline__ void sc_mr_seed(const SolverDev& d, int nblk, bool dry) {
    DevState* S = d.st;
    const int done = S->done, m = S->m;
    constexpr int NG = n_gram(L);
    __shared__ dcx G[NG];
    reduce_slots<NG, DFP>(d.part, nblk, NG, G, dry);
    if (done || threadIdx.x != 0) return;
    int bad = 0;
    // slot of (i, k), i <= k, in the row-major upper triangle
    auto slot = [](int i, int k) { return i * (L + 1) - i * (i - 1) / 2 + (k - i); };
    if (dry)   // a regular Gram matrix, so that the dry run takes the solving path
        for (int i = 0; i <= L; ++i) G[slot(i, i)] = mk(1.0);
    dcx gam[L + 1];
    gam[0] = mk(-1.0);
    for (int i = 1; i <= L; ++i) {
        const double gii = G[slot(i, i)].r;
        if (!(gii > 0.0) || !isfinite(gii)) bad = FA_EBREAKDOWN;
    }
    if constexpr (L == 1) {
        // gamma_1 = <r_1, r_0> / <r_1, r_1>
        if (!bad) gam[1] = zscale(1.0 / G[slot(1, 1)].r, conjd(G[slot(0, 1)]));
    } else if constexpr (L == 2) {
        // Cramer's rule on the Hermitian 2 x 2 normal equations (no scaling:
        // the rule is covariant under it)
        const double g11 = G[slot(1, 1)].r, g22 = G[slot(2, 2)].r;
        const dcx g12 = G[slot(1, 2)];
        const dcx b1 = conjd(G[slot(0, 1)]), b2 = conjd(G[slot(0, 2)]);   // <r_i, r_0>
        const double det = __fma_rn(g11, g22, -zabs2(g12));
        if (bad || !(det != 0.0) || !isfinite(det)) {
            bad = bad ? bad : FA_EBREAKDOWN;
        } else {
            const double idet = 1.0 / det;
            gam[1] = zscale(idet, zsub(zscale(g22, b1), zmul(g12, b2)));
            gam[2] = zscale(idet, zsub(zscale(g11, b2), zmul(conjd(g12), b1)));
        }
    } else {
        // Diagonal scaling by powers of two (exact; integer work only), so that
        // the scaled diagonal lies in [1, 4).
        double dsc[L];
        for (int i = 1; i <= L; ++i) dsc[i - 1] = pow2_rsqrt(G[slot(i, i)].r);
        dcx Ab[L][L + 1];
        for (int i = 1; i <= L; ++i) {
            for (int k = 1; k <= L; ++k) {
                const dcx gik = (i <= k) ? G[slot(i, k)] : conjd(G[slot(k, i)]);
                Ab[i - 1][k - 1] = zscale(__dmul_rn(dsc[i - 1], dsc[k - 1]), gik);
            }
            Ab[i - 1][L] = zscale(dsc[i - 1], conjd(G[slot(0, i)]));   // <r_i, r_0>
        }
        dcx z[L];
        {
            // elimination with partial pivoting (the power basis r_1..r_l can
            // make the normal equations numerically indefinite for large l; any
            // solution is a valid MR polynomial); one inverse per pivot
            dcx ipiv[L];
            for (int k = 0; k < L && !bad; ++k) {
                int pr = k;
                double best = zabs2(Ab[k][k]);
                for (int i = k + 1; i < L; ++i)
                    if (zabs2(Ab[i][k]) > best) { best = zabs2(Ab[i][k]); pr = i; }
                if (!(best > 0.0)) { bad = FA_EBREAKDOWN; break; }
                if (pr != k)
                    for (int q = k; q <= L; ++q) { dcx tq = Ab[k][q]; Ab[k][q] = Ab[pr][q]; Ab[pr][q] = tq; }
                ipiv[k] = zinv(Ab[k][k]);
                for (int i = k + 1; i < L; ++i) {
                    const dcx f = zmul(Ab[i][k], ipiv[k]);
                    for (int q = k + 1; q <= L; ++q) Ab[i][q] = zsub(Ab[i][q], zmul(f, Ab[k][q]));
                }
            }
            if (!bad) {
                for (int i = L - 1; i >= 0; --i) {
                    dcx v = Ab[i][L];
                    for (int q = i + 1; q < L; ++q) v = zsub(v, zmul(Ab[i][q], z[q]));
                    z[i] = zmul(v, ipiv[i]);
                }
            }
        }
        if (!bad)
            for (int j = 1; j <= L; ++j) gam[j] = zscale(dsc[j - 1], z[j - 1]);
    }
    if (!bad)
        for (int j = 1; j <= L; ++j)
            if (!zfinite(gam[j])) bad = FA_ENONFINITE;
    if (dry) {
        if (!bad) G[0] = gam[L];
        return;
    }
    if (bad) { fail(S, bad); return; }
    for (int j = 0; j <= L; ++j) put_scalar(d.rec_gamma, d.rec_gamma4, m * (L + 1) + j, gam[j]);
    S->omega = pk(gam[L]);
}

// Shift part of the MR step: p_s = 1 - sum_j gamma_j (-sigma)^j, zeta <- zeta p_s,
// zeta' <- zeta' p_s, and the weights 1/p_s and c_k/(zeta p_s) with c_k = sum_{j>k}
// gamma_j (-sigma)^{j-1-k}.  The powers of -sigma are real.  A thread per shift
// (kMaxShifts <= blockDim.x).
// `between` runs once the new zeta are written, by every thread of the block
// (the ticket and, if it is the last, the convergence step, which waits for
// nothing else of this block): the weights' divisions are then off the kernel's
// longest path.
template <int L, typename F>
__device__ __forceinline__ void mr_shifts(const SolverDev& d, F between) {
    DevState* S = d.st;
    const int sh = threadIdx.x, m = S->m;
    const bool act = !S->done && sh < d.ns && d.active[sh];
    dcx gam[L + 1], ps = mk(1.0), zps = mk(1.0);
    double pw[L + 1], nps = 1.0, nz = 1.0, ips, izps;
    if (act) {
        const double ms = -d.sigma[sh];
        pw[0] = 1.0;
#pragma unroll
        for (int j = 1; j <= L; ++j) {
            gam[j] = ld(d.rec_gamma[m * (L + 1) + j]);
            pw[j] = __dmul_rn(pw[j - 1], ms);
        }
#pragma unroll
        for (int j = 1; j <= L; ++j) ps = zrfma(-pw[j], gam[j], ps);
        zps = zmul(ld(d.zeta[sh]), ps);
        d.zeta[sh] = pk(zps);
        d.zeta_p[sh] = pk(zmul(ld(d.zeta_p[sh]), ps));
        // a failure has to be on record before the convergence step: within these
        // bounds the divisions cannot give one
        nps = zabs2(ps);
        nz = zabs2(zps);
        if (!(nps > 1e-120 && nps < 1e120 && nz > 1e-120 && nz < 1e120)) {
            recip2(nps, nz, ips, izps);
            if (!(nps > 0.0) || !isfinite(ips) || !isfinite(izps) || !zfinite(ps)) fail(S, FA_ENONFINITE);
        }
    }
    between();
    if (!act) return;
    recip2(nps, nz, ips, izps);
    const dcx inv_ps = zconj_scale(ips, ps);
    const dcx inv_zps = zconj_scale(izps, zps);
    double2* P = d.prec + ((size_t)sh * d.max_outer + m) * ps_stride(L) + 5 * L;
    P[0] = pk(inv_ps);
#pragma unroll
    for (int k = 0; k < L; ++k) {
        dcx c = mk(0.0);
#pragma unroll
        for (int j = k + 1; j <= L; ++j) c = zrfma(pw[j - 1 - k], gam[j], c);
        P[1 + k] = pk(zmul(c, inv_zps));
    }
}
template <int L> __device__ __noinline__ void sc_mr_shifts(const SolverDev& d) { mr_shifts<L>(d, [] {}); }

// end of an outer iteration: convergence and freezing of shifts, next beta
template <bool DFP>
__device__ __noinline__ void sc_conv(const SolverDev& d, int nblk, int head, bool dry) {
    DevState* S = d.st;
    // every load the step needs is issued with the partial loads and consumed
    // after the reduction (one memory round trip)
    const int done = S->done, m = S->m;
    const double tol2b = S->tol2b, theta2b = S->theta2b;
    const dcx omega = ld(S->omega), rho_old = ld(S->rho0), alpha = ld(S->alpha);
    const int sh = threadIdx.x;     // one thread per shift (kMaxShifts <= blockDim.x)
    const int act = sh < d.ns ? d.active[sh] : 0;
    const double2 zv = sh < d.ns ? d.zeta[sh] : make_double2(0.0, 0.0);
    __shared__ dcx red[2];
    reduce_slots<2, DFP>(d.part, nblk, 2, red, dry);
    if (done) return;
    const dcx rtr = dry ? mk(1.0) : red[0];
    const double rn2 = dry ? 1.0 : red[1].r;
    __shared__ int n_act, all_small;
    if (threadIdx.x == 0) { n_act = 0; all_small = 1; }
    __syncthreads();
    const bool last = d.fixed_iters && m + 1 >= d.max_outer;
    if (act) {
        const double z2 = zabs2(ld(zv));
        if (last || rn2 <= tol2b * z2) {
            if (!dry) {
                d.active[sh] = 0;
                d.iters[sh] = m + 1;
            }
        } else {
            atomicAdd(&n_act, 1);
            if (rn2 > theta2b * z2) atomicAnd(&all_small, 0);
        }
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (!dry) {
        S->rnorm2 = rn2;
        S->m = m + 1;
        S->n_active = n_act;
    }
    if (!isfinite(rn2) || !zfinite(rtr)) {
        if (!dry) { fail(S, FA_ENONFINITE); S->n_outer = m + 1; }
        return;
    }
    if (head && all_small && !dry) S->switch_req = 1;
    if (n_act == 0) {
        if (!dry) { S->done = 1; S->n_outer = m + 1; }
        return;
    }
    if (m + 1 >= d.max_outer) {
        if (!dry) { fail(S, FA_ENOCONV); S->n_outer = m + 1; }
        return;
    }
    const dcx rho0 = zneg(zmul(omega, rho_old));
    if (zabs2(rho0) == 0.0) {
        if (!dry) { fail(S, FA_EBREAKDOWN); S->n_outer = m + 1; }
        return;
    }
    const dcx beta = zmul(zmul(alpha, rtr), zinv(rho0));
    if (dry) { red[0] = beta; return; }
    S->rho0 = pk(rtr);
    put_scalar(d.rec_beta, d.rec_beta4, (m + 1) * d.L, beta);
}

// Step run by the last block of a reduction over the pass-1 seed vectors.
enum StepKind : int {
    STEP_NONE = 0,
    STEP_BETA = 1,          // beta of sub-step arg
    STEP_ALPHA = 2,         // alpha of sub-step arg (seed part)
    STEP_ALPHA_ALL = 3,     // alpha of sub-step arg, seed and shift parts (single pass)
    STEP_CONV = 4,          // convergence; arg = head flag
    STEP_SHIFTS = 5         // k_hop1_split without inner product: block 0 runs the shift part of sub-step arg
};
struct ScalarStep {
    int kind;
    int arg;
};

// the step itself, by the block that holds the last ticket (or dry)
template <bool DFP>
__device__ __forceinline__ void do_step(const SolverDev& d, ScalarStep e, int nblk, bool dry) {
    if (e.kind == STEP_BETA) {
        sc_beta<DFP>(d, e.arg, nblk, dry);
    } else if (e.kind == STEP_ALPHA || e.kind == STEP_ALPHA_ALL) {
        sc_alpha_seed<DFP>(d, e.arg, nblk, dry);
        if (e.kind == STEP_ALPHA_ALL && !dry) {
            __syncthreads();
            sc_alpha_shifts(d, e.arg);
        }
    } else {
        sc_conv<DFP>(d, nblk, e.arg, dry);
    }
}

// nblk: partials of the reduction; ntickets: blocks of the system in this launch;
// warm: a late block that is not the last may run the step dry (last_block)
template <bool DFP>
__device__ __forceinline__ void run_step(const SolverDev& d, ScalarStep e, int nblk, int ntickets, bool warm = true) {
    if (e.kind == STEP_NONE) return;
    const int lb = last_block(d.st, ntickets);
    // (FP64 kernels run no dry runs: their sweeps are bound by the FP64 pipe,
    // which the dry step would share)
    if (lb == LB_NONE || (lb == LB_WARM && (!warm || !DFP))) return;
    do_step<DFP>(d, e, nblk, lb == LB_WARM);
}

// Resident blocks per SM of the balanced vector kernels (register budget <= 64).
constexpr int kVecBlocks = 4;

// Contiguous site range [s0, s1) of block bx of nbx (V/nbx sites, +-1).  The
// vector kernels run at most one wave (kVecBlocks per SM, which their register
// budget guarantees); larger lattices loop over their range.
__device__ __forceinline__ void site_range(int V, unsigned bx, unsigned nbx, int& s0, int& s1) {
    s0 = (int)(((long long)V * bx) / nbx);
    s1 = (int)(((long long)V * (bx + 1)) / nbx);
}

// Partials of a kThreads-block reduction: one per block, FP64 one per warp
// (the order that reduce_slots takes them in), K slots of n_partials(nbx) each.
template <typename R> __host__ __device__ constexpr int n_partials(int nbx) {
    return std::is_same<R, double>::value ? nbx * (kThreads / 32) : nbx;
}
template <int K, typename R>
__device__ __forceinline__ void reduce_store(cx<R> (&v)[K], double2* out, int nbx, int bx) {
    if constexpr (std::is_same<R, double>::value) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            double a = v[k].r, b = v[k].i;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a = __dadd_rn(a, __shfl_down_sync(0xffffffffu, a, o));
                b = __dadd_rn(b, __shfl_down_sync(0xffffffffu, b, o));
            }
            if ((threadIdx.x & 31) == 0)
                out[(size_t)k * n_partials<R>(nbx) + n_partials<R>(bx) + (threadIdx.x >> 5)] = make_double2(a, b);
        }
    } else {
        block_reduce_store<K, R>(v, out, nbx, bx);
    }
}

// ------------------------------------------------------------------ MR part
// Gram matrix <r_i, r_k>, 0 <= i <= k <= L (FP32: batches, l = 8; one system with
// l <= 4 forms it in its last sweep.  Double-float always; FP64: k_gram_tile),
// grid-stride, per-block partials.  Last block: the MR coefficients (sc_mr_seed).
// DEFER (FP32): the deferred updates of r in registers first.
//
// Double-float: the rows of the triangle are shared out to gridDim.z blocks, so
// that a thread holds at most 3 (l = 2), 5 (l = 4) or 9 (l = 8) products: all 15
// of l = 4 took 250 registers, one block per SM, and 3.1 ms on 32^3 x 64 where
// the arithmetic is 0.95 ms.  The component loop is not unrolled whole: its code
// (85 KB for l = 2) did not stay in the instruction cache.
template <typename R, int L> constexpr int gram_groups() { return std::is_same<R, float>::value || L == 1 ? 1 : (L + 2) / 2; }
// l = 2: groups while their blocks are one wave of 3 per SM, else all products in a thread
// (12^3 x 24: 34 -> 19 us; 16^3 x 32: 43 us, 54 in groups)
// rows of group z: l even {0}, {1, l}, {2, l - 1}, ...; l odd {0, l}, {1, l - 1}, ...
template <int L> constexpr int gram_row_a(int z) { return z; }
template <int L> constexpr int gram_row_b(int z) { return L % 2 ? L - z : (z == 0 ? -1 : L + 1 - z); }
template <typename R, int L, bool GROUPS> constexpr int gram_min_blocks() {
    return !GROUPS ? (L <= 2 ? 4 : 1) : (L <= 4 ? 3 : 2);
}
template <int L> constexpr int gram_row_slot(int i) { return i * (L + 1) - i * (i - 1) / 2; }

template <typename R, int L, int Z>
__device__ __forceinline__ void gram_rows(const SolverDev& d, const Where& w) {
    constexpr int A = gram_row_a<L>(Z), B = gram_row_b<L>(Z);
    constexpr int NA = L + 1 - A, NB = B >= 0 && B != A ? L + 1 - B : 0;
    const typename Ch<R>::T* r = Vec<R>::r(d);
    const size_t vs = vstride<R>(d);
    const int V = d.V;
    cx<R> a[NA], b[NB > 0 ? NB : 1];
#pragma unroll
    for (int k = 0; k < NA; ++k) a[k] = czero<R>();
#pragma unroll
    for (int k = 0; k < NB; ++k) b[k] = czero<R>();
    int s0, s1;
    site_range(V, w.bx, w.nbx, s0, s1);
    for (int s = s0 + threadIdx.x; s < s1; s += kThreads) {
#pragma unroll 2
        for (int q = 0; q < Ch<R>::N; ++q) {
            Ch<R> v[NA];
#pragma unroll
            for (int k = 0; k < NA; ++k) v[k] = Ch<R>::ld(r + (A + k) * vs, q, V, s);
#pragma unroll
            for (int c = 0; c < Ch<R>::W; ++c) {
#pragma unroll
                for (int k = 0; k < NA; ++k) a[k] = cjfma(v[0].c[c], v[k].c[c], a[k]);
#pragma unroll
                for (int k = 0; k < NB; ++k) b[k] = cjfma(v[L + 1 - NB - A].c[c], v[L + 1 - NB - A + k].c[c], b[k]);
            }
        }
    }
    block_reduce_store<NA, R>(a, d.part + (size_t)gram_row_slot<L>(A) * w.nbx, w.nbx, w.bx);
    if constexpr (NB > 0) block_reduce_store<NB, R>(b, d.part + (size_t)gram_row_slot<L>(B) * w.nbx, w.nbx, w.bx);
}

template <typename R, int L, bool DEFER, bool GROUPS>
__global__ void __launch_bounds__(kThreads, gram_min_blocks<R, L, GROUPS>())
k_gram(const SolverDev* __restrict__ ds, const int4* tab) {
    dep_wait();
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, 0)) return;
    const TraceScope trace_(trace_kind<R>(FA_TK_GRAM));
    constexpr int NZ = GROUPS ? gram_groups<R, L>() : 1;
    if constexpr (NZ > 1) {
        if (blockIdx.z == 0) gram_rows<R, L, 0>(d, w);
        else if (blockIdx.z == 1) gram_rows<R, L, 1>(d, w);
        else if (NZ > 2 && blockIdx.z == 2) gram_rows<R, L, (NZ > 2 ? 2 : 0)>(d, w);
        else if (NZ > 3 && blockIdx.z == 3) gram_rows<R, L, (NZ > 3 ? 3 : 0)>(d, w);
        else if (NZ > 4) gram_rows<R, L, (NZ > 4 ? 4 : 0)>(d, w);
    } else {
        const typename Ch<R>::T *r = Vec<R>::r(d), *ub = Vec<R>::u(d);
        const size_t vs = vstride<R>(d);
        constexpr int NG = n_gram(L);
        const StepScalars<R, DEFER ? L : 1> sc(d, d.st->m);
        cx<R> acc[NG];
#pragma unroll
        for (int k = 0; k < NG; ++k) acc[k] = czero<R>();
        int s0, s1;
        site_range(d.V, w.bx, w.nbx, s0, s1);
        auto chunk = [&](int q, int s) {
            Ch<R> v[L + 1];
#pragma unroll
            for (int i = 0; i <= L; ++i) v[i] = Ch<R>::ld(r + i * vs, q, d.V, s);
            if constexpr (DEFER) {
                Ch<R> u[L];
#pragma unroll
                for (int i = 1; i < L; ++i) u[i] = Ch<R>::ld(ub + i * vs, q, d.V, s);
                deferred_r<R, L>(sc, v, u);
            }
            int g = 0;
#pragma unroll
            for (int i = 0; i <= L; ++i)
#pragma unroll
                for (int k = i; k <= L; ++k) {
#pragma unroll
                    for (int w = 0; w < Ch<R>::W; ++w) acc[g] = cjfma(v[i].c[w], v[k].c[w], acc[g]);
                    ++g;
                }
        };
        for (int s = s0 + threadIdx.x; s < s1; s += kThreads) {
            if constexpr (std::is_same<R, float>::value) {
#pragma unroll
                for (int q = 0; q < Ch<R>::N; ++q) chunk(q, s);
            } else {
#pragma unroll 2
                for (int q = 0; q < Ch<R>::N; ++q) chunk(q, s);
            }
        }
        block_reduce_store<NG, R>(acc, d.part, w.nbx, w.bx);
    }
    const int lb = last_block(d.st, w.ntk * NZ);
    if (lb != LB_NONE) sc_mr_seed<L, true>(d, w.nbx, lb == LB_WARM);
}

// MR update of pass 1 (FP32, double-float; FP64: k_mr_tile): r_0 -= sum gamma_j
// r_j, u_0 -= sum gamma_j u_j, the per-block partials of <rt, r_0> (slot 0) and
// |r_0|^2 (slot 1), grid-stride, then `step` (convergence) in the last block.
// DEFER (FP32): the deferred updates first.  Block 0 runs the shift part of the
// MR step (mr_shifts) and takes a ticket too, so that the convergence step
// sees the new zeta; blocks 1.. are the vector blocks.
// l <= 3: registers capped for 4 blocks/SM (64; some bytes spilled), so that a
// 16^3 x 32 lattice (512 blocks) runs in one wave instead of 1.12 (left alone,
// the compiler takes up to 167 registers here).  Double-float: the component
// loop is not unrolled whole (see k_gram).
template <int L> constexpr int mr_min_blocks() { return L <= 3 ? 4 : 1; }
// G: components whose loads are issued together.  The stores of one component
// keep the compiler from moving the next one's loads up, so with a block or two
// per SM a thread waits for one round trip per component; mr_ahead of them at a
// time, in the registers that two blocks per SM leave, while the grid is no more
// than that.  12^3 x 24, l = 2 (162 blocks): FP32 16.0 -> 11.5 us, double-float
// 34.3 -> 23.0 us.
template <int L> constexpr int mr_ahead() { return L <= 2 ? 3 : 2; }
template <typename R, int L, bool DEFER, int G = 1>
__global__ void __launch_bounds__(kThreads, G > 1 ? (mr_min_blocks<L>() < 2 ? 1 : 2) : mr_min_blocks<L>())
k_mr(const SolverDev* __restrict__ ds, ScalarStep step, const int4* tab) {
    dep_wait();
    const Where w = where<true>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, 0)) return;
    const TraceScope trace_(trace_kind<R>(FA_TK_MR, true));
    const int bx = w.bx, nbx = w.nbx;
    if (bx < 0) {
        mr_shifts<L>(d, [&] {
            __threadfence();   // the new zeta of every thread before the ticket
            run_step<true>(d, step, nbx, w.ntk);
        });
        return;
    }
    const int m = d.st->m, V = d.V;
    using T = typename Ch<R>::T;
    T *r = Vec<R>::r(d), *u = Vec<R>::u(d);
    const T* rt = Vec<R>::rt(d);
    const size_t vs = vstride<R>(d);
    T* store = store_at<R>(d, m);
    const StepScalars<R, DEFER ? L : 1> sc(d, m);
    cx<R> ng[L + 1];
    ng[0] = czero<R>();
#pragma unroll
    for (int j = 1; j <= L; ++j) ng[j] = nweight<R>(d.rec_gamma, d.rec_gamma4, m * (L + 1) + j);
    cx<R> dots[2] = {czero<R>(), czero<R>()};
    auto chunk = [&](int q, int s, Ch<R> (&rv)[L + 1], Ch<R> (&uv)[L + 1], const Ch<R>& tv) {
        if constexpr (DEFER) deferred<R, L>(d, m, sc, rv, uv, store, q, s);
        if (store != nullptr) {
#pragma unroll
            for (int k = 0; k < L; ++k) rv[k].stv_cs(store + slot_mr(L, k) * vs, q, V, s);
        }
        if (d.x64 != nullptr) {
#pragma unroll
            for (int j = 1; j <= L; ++j) acc_x<R>(d.x64, q, V, s, d.rec_gamma[m * (L + 1) + j], rv[j - 1]);
        }
        Ch<R> r0 = rv[0], u0 = uv[0];
#pragma unroll
        for (int j = 1; j <= L; ++j) {
#pragma unroll
            for (int w = 0; w < Ch<R>::W; ++w) {
                r0.c[w] = cfma(ng[j], rv[j].c[w], r0.c[w]);
                u0.c[w] = cfma(ng[j], uv[j].c[w], u0.c[w]);
            }
        }
        r0.stv(r, q, V, s);
        u0.stv(u, q, V, s);
#pragma unroll
        for (int w = 0; w < Ch<R>::W; ++w) {
            dots[0] = cjfma(tv.c[w], r0.c[w], dots[0]);
            dots[1].r = fmaR(r0.c[w].r, r0.c[w].r, dots[1].r);
            dots[1].r = fmaR(r0.c[w].i, r0.c[w].i, dots[1].r);
        }
    };
    auto chunks = [&](int q0, int s) {
        Ch<R> rv[G][L + 1], uv[G][L + 1], tv[G];
#pragma unroll
        for (int k = 0; k < G; ++k) {
#pragma unroll
            for (int i = 0; i <= L; ++i) rv[k][i] = Ch<R>::ld(r + i * vs, q0 + k, V, s);
#pragma unroll
            for (int i = 0; i <= L; ++i) uv[k][i] = Ch<R>::ld(u + i * vs, q0 + k, V, s);
            tv[k] = Ch<R>::ld(rt, q0 + k, V, s);
        }
#pragma unroll
        for (int k = 0; k < G; ++k) chunk(q0 + k, s, rv[k], uv[k], tv[k]);
    };
    static_assert(Ch<R>::N % G == 0, "whole groups of components");
    int s0, s1;
    site_range(V, bx, nbx, s0, s1);
    for (int s = s0 + threadIdx.x; s < s1; s += kThreads) {
        if constexpr (std::is_same<R, float>::value) {
#pragma unroll
            for (int q = 0; q < Ch<R>::N; q += G) chunks(q, s);
        } else if constexpr (G > 1) {
#pragma unroll 1
            for (int q = 0; q < Ch<R>::N; q += G) chunks(q, s);
        } else {
#pragma unroll 2
            for (int q = 0; q < Ch<R>::N; ++q) chunks(q, s);
        }
    }
    block_reduce_store<2, R>(dots, d.part, nbx, bx);
    run_step<true>(d, step, nbx, w.ntk);
}

// <rt, r0> (slot 0) and |r0|^2 (slot 1), grid-stride (start of a solve)
template <typename R>
__device__ __forceinline__ void k_dot2_body(int V, const typename Ch<R>::T* rt, const typename Ch<R>::T* r0,
                                            double2* partials, int bx, int nbx) {
    cx<R> dots[2] = {czero<R>(), czero<R>()};
    int s0, s1;
    site_range(V, bx, nbx, s0, s1);
    for (int s = s0 + threadIdx.x; s < s1; s += kThreads) {
#pragma unroll
        for (int q = 0; q < Ch<R>::N; ++q) {
            Ch<R> a = Ch<R>::ld(rt, q, V, s), b = Ch<R>::ld(r0, q, V, s);
#pragma unroll
            for (int w = 0; w < Ch<R>::W; ++w) {
                dots[0] = cjfma(a.c[w], b.c[w], dots[0]);
                dots[1].r = fmaR(b.c[w].r, b.c[w].r, dots[1].r);
                dots[1].r = fmaR(b.c[w].i, b.c[w].i, dots[1].r);
            }
        }
    }
    reduce_store<2, R>(dots, partials, nbx, bx);
}

template <typename R>
__global__ void __launch_bounds__(kThreads)
k_dot2(int V, const typename Ch<R>::T* rt, const typename Ch<R>::T* r0, double2* partials) {
    k_dot2_body<R>(V, rt, r0, partials, blockIdx.x, gridDim.x);
}

// start of pass 1: <rt, r0>, |r0|^2 and, in the last block, the initial state
template <typename R>
__global__ void __launch_bounds__(kThreads, kVecBlocks)
k_dot2_sys(const SolverDev* __restrict__ ds, double tol, double theta, const int4* tab) {
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    k_dot2_body<R>(d.V, Vec<R>::rt(d), Vec<R>::r(d), d.part, w.bx, w.nbx);
    if (last_block(d.st, w.ntk) == LB_LAST) sc_init<dfp_of<R>()>(d, n_partials<R>(w.nbx), tol, theta);
}

// A application inside the solver: out = scale * g5 D in on the system's own
// links, mu and scale (scale = 1 for the first hop of A, c for the second).
// Vector selectors: 0 = u family, 1 = r family, 2 = scratch, 3 = rb family.  DOT: per-block
// partials of <rt, out> into the system's partial buffer.
template <typename R>
__device__ __forceinline__ typename Ch<R>::T* select_vec(const SolverDev& d, int sel, int j) {
    typename Ch<R>::T* base = sel == 0 ? Vec<R>::u(d) : sel == 1 ? Vec<R>::r(d) : sel == 2 ? Vec<R>::tmp(d) : Vec<R>::rb(d);
    return base + (size_t)j * vstride<R>(d);
}

// A block of the FP64 sweep with a thread per site; DOT: the site's term of <dotv, out>
template <bool DOT>
__device__ __forceinline__ cx<double> hop64_site_body(const Geom& g, const LinkView<double>& U,
                                                      const SpinorView<double>& in, const SpinorView<double>& out,
                                                      const Op64& op, const SpinorView<double>& dotv, int bx) {
    const int s = bx * kSite64 + (int)threadIdx.x;
    cx<double> a = czero<double>();
    if (s < g.V) {
        cx<double> p[12];
        hop_site<double, false, true>(g, U, in, s, op.cdiag, op.chop, op.ef, op.eb, op.bc, p);
        out.store(s, p);
        if (DOT) {
#pragma unroll
            for (int k = 0; k < 12; ++k) a = cjfma(dotv.ld1(s, k), p[k], a);
        }
    }
    return a;
}
// the partials of the block's 32-site tiles, as dot64_tile leaves them
__device__ __forceinline__ void store_tile_dot(cx<double> v, double2* part, int V, int bx) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.r = __dadd_rn(v.r, __shfl_down_sync(0xffffffffu, v.r, o));
        v.i = __dadd_rn(v.i, __shfl_down_sync(0xffffffffu, v.i, o));
    }
    const int tile = bx * (kSite64 / 32) + (int)(threadIdx.x >> 5);
    if ((threadIdx.x & 31) == 0 && tile < tiles64(V)) part[tile] = make_double2(v.r, v.i);
}

// FP64, one system, pointers as kernel parameters: C blocks per tile (hop64.cuh)
template <int C, bool DOT>
__global__ void __launch_bounds__(hop64_threads<C>(), hop64_min_blocks<C>())
k_hop64(Geom g, const double2* __restrict__ U, const double2* in, double2* out, Op64 op, const double2* dotv,
        double2* partials, const int* done, const SolverDev* __restrict__ ds, ScalarStep step) {
    dep_wait();
    if (done != nullptr && *done) return;
    const TraceScope trace_(trace_kind<double>(FA_TK_HOP1, DOT));
    __shared__ Smem64<C> sm;
    const int tile = blockIdx.x / C, rank = blockIdx.x % C;
    hop64_tile<C, true, DOT>(g, U, internal64(in, g.V), internal64(out, g.V), op, tile, rank, sm);
    if (DOT && rank == 0) {
        dep_launch();
        const double2 v = dot64_tile<C>(internal64(dotv, g.V), g.V, tile, sm);
        if (threadIdx.x == 0) partials[tile] = v;
        run_step<false>(ds[0], step, gridDim.x / C, gridDim.x / C);
    }
}

// FP64, a batch: one tile of one system per block
template <bool DOT>
__global__ void __launch_bounds__(hop64_threads<1>(), hop64_min_blocks<1>())
k_hop64_sys(const SolverDev* __restrict__ ds, int in_sel, int in_j, int out_sel, int out_j, int second, int pass2,
            ScalarStep step, const int4* tab) {
    dep_wait();
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, pass2)) return;
    const TraceScope trace_(trace_kind<double>(FA_TK_HOP_SYS, DOT));
    __shared__ Smem64<1> sm;
    const double sc = second ? d.scale : 1.0;
    const Op64 op{sc * d.diag, -0.5 * sc, d.ef, d.eb, d.bc, 0, 1};
    hop64_tile<1, true, DOT>(d.g, d.links64, internal64(select_vec<double>(d, in_sel, in_j), d.V),
                             internal64(select_vec<double>(d, out_sel, out_j), d.V), op, w.bx, 0, sm);
    if (DOT) {
        dep_launch();
        const double2 v = dot64_tile<1>(internal64(d.rt64, d.V), d.V, w.bx, sm);
        if (threadIdx.x == 0) d.part[w.bx] = v;
        run_step<false>(d, step, w.nbx, w.ntk);
    }
}

// FP64, a thread per site (launch rule: hop64_by_site), one system
template <bool DOT>
__global__ void __launch_bounds__(kSite64, kSite64Blocks)
k_hop64_site(Geom g, LinkView<double> U, SpinorView<double> in, SpinorView<double> out, Op64 op,
             SpinorView<double> dotv, double2* partials, const int* done, const SolverDev* __restrict__ ds,
             ScalarStep step) {
    dep_wait();
    if (done != nullptr && *done) return;
    const TraceScope trace_(trace_kind<double>(FA_TK_HOP1, DOT));
    const cx<double> v = hop64_site_body<DOT>(g, U, in, out, op, dotv, blockIdx.x);
    if (DOT) {
        store_tile_dot(v, partials, g.V, blockIdx.x);
        run_step<false>(ds[0], step, tiles64(g.V), gridDim.x);
    }
}
// and a batch
template <bool DOT>
__global__ void __launch_bounds__(kSite64, kSite64Blocks)
k_hop64_site_sys(const SolverDev* __restrict__ ds, int in_sel, int in_j, int out_sel, int out_j, int second, int pass2,
                 ScalarStep step, const int4* tab) {
    dep_wait();
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, pass2)) return;
    const TraceScope trace_(trace_kind<double>(FA_TK_HOP_SYS, DOT));
    const double sc = second ? d.scale : 1.0;
    const Op64 op{sc * d.diag, -0.5 * sc, d.ef, d.eb, d.bc, 0, 1};
    const cx<double> v = hop64_site_body<DOT>(d.g, LinkView<double>{d.links64, d.V},
                                              SpinorView<double>{select_vec<double>(d, in_sel, in_j), d.V},
                                              SpinorView<double>{select_vec<double>(d, out_sel, out_j), d.V}, op,
                                              SpinorView<double>{d.rt64, d.V}, w.bx);
    if (DOT) {
        store_tile_dot(v, d.part, d.V, w.bx);
        run_step<false>(d, step, tiles64(d.V), w.ntk);
    }
}

// Systems that share one gauge field and lattice (the sources of one lattice in
// a batch): the multi-RHS sweep applies D_w to all of them tile by tile.
constexpr int kMaxRhs = 16;
struct GroupDev {
    int nsys;
    int ntile;             // tiles of kHopNarrowThreads sites
    int sys[kMaxRhs];      // descriptor index of each system
};

// The seed steps (beta or alpha) of the systems whose last ticket this block
// holds: it often is the last for all right-hand sides of its run, so their
// partials are summed side by side and a thread per system runs the step
// (reduce_slots, sc_beta and sc_alpha_seed, the same operations in the same
// order).
__device__ __noinline__ void mrhs_steps(const SolverDev* __restrict__ ds, const GroupDev& G, int first, int nr,
                                        const int* lasts, ScalarStep e) {
    __shared__ float4 qf[4 * kMaxRhs];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nblk = G.ntile, per = (nblk + 3) >> 2;
    for (int u = warp; u < 4 * nr; u += nw) {
        if (!lasts[u >> 2]) continue;
        const float4* pf = reinterpret_cast<const float4*>(ds[G.sys[first + (u >> 2)]].part);
        const int i0 = (u & 3) * per, i1 = min(nblk, i0 + per);
        df a(0.0f), b(0.0f);
        for (int ib = i0 + lane; ib < i1; ib += 32 * 8) {
            float4 v[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int i = ib + 32 * t;
                v[t] = i < i1 ? __ldcg(pf + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                a = addR(a, df(v[t].x, v[t].y));
                b = addR(b, df(v[t].z, v[t].w));
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a = addR(a, shfl_down_df(a, o));
            b = addR(b, shfl_down_df(b, o));
        }
        if (lane == 0) qf[u] = make_float4(a.hi, a.lo, b.hi, b.lo);
    }
    __syncthreads();
    const int r = threadIdx.x;
    if (r >= nr || !lasts[r]) return;
    const SolverDev& d = ds[G.sys[first + r]];
    DevState* S = d.st;
    df a(0.0f), b(0.0f);
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
        const float4 t = qf[4 * r + q];
        a = addR(a, df(t.x, t.y));
        b = addR(b, df(t.z, t.w));
    }
    if (S->done) return;
    const dcx red = {todbl(a), todbl(b)};
    if (e.kind == STEP_BETA) seed_beta(d, e.arg, S->m, ld(S->rho0), ld(S->alpha), red);
    else seed_alpha(d, e.arg, S->m, ld(S->rho0), red);
}

// FP32 sweep of a batch, several right-hand sides per block.  items[blockIdx.x]
// = (group, tile, first, end): the block applies the sweep to the systems
// first..end-1 of the group on the tile's sites, one after the other, so the
// tile's links (and the neighbours' backward links) come from HBM once and
// from L1 for the other right-hand sides.  Each system's arithmetic, its
// per-tile partials of <rt, out> and its scalar step are those of the
// one-system sweep of the same launch shape (128-thread blocks), so a batched
// solve equals the one-at-a-time solve bit for bit.
//
// The inner products of a block's right-hand sides are finished together: one
// fence and one ticket round for all of them instead of a barrier, a fence and
// an atomic after each sweep (12 sources on 12^3 x 24 and 8^3 x 16, us per
// sweep: 55.8 with a round per right-hand side, 31.8 for the sweep without
// inner products).
template <bool DOT, int MB>
__global__ void __launch_bounds__(kHopNarrowThreads, MB)
k_hop_mrhs(const SolverDev* __restrict__ ds, const GroupDev* __restrict__ groups, const int4* __restrict__ items,
           int in_sel, int in_j, int out_sel, int out_j, int second, int pass2, ScalarStep step) {
    constexpr int NT = kHopNarrowThreads, NW = NT / 32;
    dep_wait();
    const int4 it = items[blockIdx.x];
    const GroupDev& G = groups[it.x];
    // no record of a block that finds all its systems finished (looked up while tracing only:
    // a flag kept through the loop below cost 20 bytes of spills and 0.8 % of a batch)
    if (trace_on()) {
        bool idle = true;
        for (int r = it.z; r < it.w; ++r) idle = idle && sys_idle(ds[G.sys[r]], pass2);
        if (idle) return;
    }
    const TraceScope trace_(trace_kind<float>(FA_TK_HOP_MRHS, DOT));
    const int tile = it.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ float2 sums[DOT ? kMaxRhs : 1][NW];
    __shared__ int lasts[DOT ? kMaxRhs : 1];
    for (int r = it.z; r < it.w; ++r) {
        const SolverDev& d = ds[G.sys[r]];
        if (sys_idle(d, pass2)) continue;   // the same for every thread of the block
        const int s = tile * NT + (int)threadIdx.x;
        cx<float> dres = czero<float>();
        if (s < d.V) {
            const SpinorView<float> in{select_vec<float>(d, in_sel, in_j), d.V};
            const SpinorView<float> out{select_vec<float>(d, out_sel, out_j), d.V};
            cx<float> p[12];
            hop_site<float, false, true>(d.g, LinkView<float>{d.links32, d.V}, in, s, second ? d.fdiag2 : d.fdiag1,
                                         second ? d.fhop2 : d.fhop1, d.fef, d.feb, d.fbc, p);
            out.store(s, p);
            if (DOT) {
                const SpinorView<float> rt{d.rt32, d.V};
                cx<float> q[12];
                rt.load(s, q);
#pragma unroll
                for (int k = 0; k < 12; ++k) dres = cjfma(q[k], p[k], dres);
            }
        }
        if (DOT) {   // the warp's sum, as in block_reduce_store
            float a = dres.r, b = dres.i;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a += __shfl_down_sync(0xffffffffu, a, o);
                b += __shfl_down_sync(0xffffffffu, b, o);
            }
            if (lane == 0) sums[r - it.z][warp] = make_float2(a, b);
        }
    }
    if constexpr (DOT) {
        dep_launch();
        const int nr = it.w - it.z;
        __syncthreads();
        // a thread per right-hand side: the warps' sums in the order of the block's shuffle
        // tree, the partial, and the system's ticket
        if ((int)threadIdx.x < nr) {
            const SolverDev& d = ds[G.sys[it.z + threadIdx.x]];
            int last = 0;
            if (!sys_idle(d, pass2)) {
                df a[NW], b[NW];
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    a[w] = df(sums[threadIdx.x][w].x);
                    b[w] = df(sums[threadIdx.x][w].y);
                }
#pragma unroll
                for (int o = NW / 2; o > 0; o >>= 1)
#pragma unroll
                    for (int w = 0; w < o; ++w) {
                        a[w] = addR(a[w], a[w + o]);
                        b[w] = addR(b[w], b[w + o]);
                    }
                reinterpret_cast<float4*>(d.part)[tile] = make_float4(a[0].hi, a[0].lo, b[0].hi, b[0].lo);
                if (step.kind != STEP_NONE) {
                    __threadfence();
                    last = atomicAdd(&d.st->ticket, 1u) == (unsigned)G.ntile - 1u;
                    if (last) {
                        d.st->ticket = 0u;
                        __threadfence();
                    }
                }
            }
            lasts[threadIdx.x] = last;
        }
        __syncthreads();
        int any = 0;
        for (int r = 0; r < nr; ++r) any |= lasts[r];
        if (any) mrhs_steps(ds, G, it.z, nr, lasts, step);
    }
}

// double-float batches: the row-split sweep (kRowThreads per block)
template <typename R, bool DOT>
__global__ void __launch_bounds__(kRowThreads, rows_sys_min_blocks<DOT>())
k_hop_sys_rows(const SolverDev* __restrict__ ds, int in_sel, int in_j, int out_sel, int out_j, int second, int pass2,
               ScalarStep step, const int4* tab) {
    dep_wait();
    const Where w = where<false>(tab);
    const SolverDev& d = ds[w.sys];
    if (sys_idle(d, pass2)) return;
    const TraceScope trace_(trace_kind<R>(FA_TK_HOP_SYS_ROWS, DOT));
    const double sc = second ? d.scale : 1.0;
    const Geom g = d.g;
    const SpinorView<R> in{select_vec<R>(d, in_sel, in_j), d.V}, out{select_vec<R>(d, out_sel, out_j), d.V};
    const SpinorView<R> rt{Vec<R>::rt(d), d.V};
    cx<R> dres[1] = {hop_rows_body<R, false, true, DOT>(g, Vec<R>::links(d), in, out,
                                                        fromdbl<R>(sc * d.diag), fromdbl<R>(-0.5 * sc),
                                                        fromdbl<R>(d.ef), fromdbl<R>(d.eb), fromdbl<R>(d.bc), rt,
                                                        w.bx)};
    if (DOT) {
        block_reduce_store<1, R, kRowThreads>(dres, d.part, 0, w.bx);
        run_step<dfp_of<R>()>(d, step, w.nbx, w.ntk, false);   // ALU-bound sweep: no dry runs
    }
}

// The hop of a single solve with its pointers as kernel parameters (the
// descriptor is read only by the scalar step of the last block).  DOT:
// partials of <dotv, out>, then `step`.  Double-float uses the row-split
// sweep (kRowThreads per block, one partial per block).
template <typename R, bool DOT>
__global__ void __launch_bounds__(kRowThreads, rows_min_blocks<DOT>())
k_hop1_rows(Geom g, LinkView<R> U, SpinorView<R> in, SpinorView<R> out, R cdiag, R chop, R ef, R eb, R bc,
            SpinorView<R> dotv, double2* partials, const int* done, const SolverDev* __restrict__ ds,
            ScalarStep step) {
    dep_wait();
    if (done != nullptr && *done) return;
    const TraceScope trace_(trace_kind<R>(FA_TK_HOP1_ROWS, DOT));
    cx<R> dres[1] = {hop_rows_body<R, false, true, DOT>(g, U, in, out, cdiag, chop, ef, eb, bc, dotv, blockIdx.x)};
    if (DOT) {
        block_reduce_store<1, R, kRowThreads>(dres, partials, 0, blockIdx.x);
        run_step<dfp_of<R>()>(ds[0], step, gridDim.x, gridDim.x, false);   // ALU-bound sweep: no dry runs
    }
}

template <typename R, bool DOT, int NT = kThreads, int MB = FA_HOP_MINB>
__global__ void __launch_bounds__(NT, MB)
k_hop1(Geom g, LinkView<R> U, SpinorView<R> in, SpinorView<R> out, R cdiag, R chop, R ef, R eb, R bc,
       SpinorView<R> dotv, double2* partials, const int* done, const SolverDev* __restrict__ ds, ScalarStep step) {
    dep_wait();
    if (done != nullptr && *done) return;
    const TraceScope trace_(trace_kind<R>(FA_TK_HOP1, DOT));
    const int s = blockIdx.x * NT + threadIdx.x;
    cx<R> dres[1] = {czero<R>()};
    if (s < g.V) {
        cx<R> p[12];
        hop_site<R, false, true>(g, U, in, s, cdiag, chop, ef, eb, bc, p);
        out.store(s, p);
        if (DOT) {
            cx<R> q[12];
            dotv.load(s, q);
            cx<R> a = czero<R>();
#pragma unroll
            for (int k = 0; k < 12; ++k) a = cjfma(q[k], p[k], a);
            dres[0] = a;
        }
    }
    if (DOT) {
        block_reduce_store<1, R, NT>(dres, partials, 0, blockIdx.x);
        run_step<dfp_of<R>()>(ds[0], step, gridDim.x, gridDim.x);
    }
}

// the FP32 sweep with two threads per site (hop_site_split), 128 sites per block.
// The sweep of r_j carries the shift part of sub-step j (STEP_SHIFTS), 4 us of FP64
// in one warp that nothing before the next sub-step needs: beside the update of
// r_j, which takes 1-2 us on such lattices, it was what that kernel waited for.
// (12^3 x 24 mixed_df: 7.54 -> 7.47 ms together with mr_shifts' early ticket; the
// ticket alone, 16^3 x 32: 14.43 -> 14.35 ms.)
template <bool DOT>
__global__ void __launch_bounds__(2 * kSplitSites, kSplitBlocks)
k_hop1_split(Geom g, LinkView<float> U, SpinorView<float> in, SpinorView<float> out, float cdiag, float chop, float ef,
             float eb, float bc, SpinorView<float> dotv, double2* partials, const int* done,
             const SolverDev* __restrict__ ds, ScalarStep step) {
    dep_wait();
    if (done != nullptr && *done) return;
    const TraceScope trace_(trace_kind<float>(FA_TK_HOP1, DOT));
    int bx = blockIdx.x;
    if (!DOT && step.kind == STEP_SHIFTS) {
        if (bx == 0) {
            sc_alpha_shifts(ds[0], step.arg);
            return;
        }
        --bx;
    }
    const int s = bx * kSplitSites + (threadIdx.x & (kSplitSites - 1));
    cx<float> dres[1] = {czero<float>()};
    cx<float> p[12];
    hop_site_split<false, true>(g, U, in, s, cdiag, chop, ef, eb, bc, p);
    if (threadIdx.x < kSplitSites && s < g.V) {
        out.store(s, p);
        if (DOT) {
            cx<float> q[12];
            dotv.load(s, q);
            cx<float> a = czero<float>();
#pragma unroll
            for (int k = 0; k < 12; ++k) a = cjfma(q[k], p[k], a);
            dres[0] = a;
        }
    }
    if (DOT) {
        block_reduce_store<1, float, kSplitSites>(dres, partials, 0, blockIdx.x);
        run_step<true>(ds[0], step, gridDim.x, gridDim.x);
    }
}

// ------------------------------------------------------------------ reliable update
// r_0 <- b - A x with A x (FP64) already in ax; the new r_0 is rounded to R.
// Rewrites the partials of <rt, r_0> (slot 0) and |r_0|^2 (slot 1) that the
// convergence step reads, grid-stride like k_mr.
template <typename R>
__global__ void __launch_bounds__(kThreads, kVecBlocks)
k_reliable(const SolverDev* __restrict__ ds, const double2* ax, int pass2, ScalarStep step) {
    const SolverDev& d = ds[blockIdx.y];   // one system (reliable updates are not batched)
    if (sys_idle(d, pass2)) return;
    const TraceScope trace_(trace_kind<R>(FA_TK_RELIABLE));
    typename Ch<R>::T* r0 = Vec<R>::r(d);
    const typename Ch<R>::T* rt = Vec<R>::rt(d);
    cx<R> dots[2] = {czero<R>(), czero<R>()};
    int s0, s1;
    site_range(d.V, blockIdx.x, gridDim.x, s0, s1);
    for (int s = s0 + threadIdx.x; s < s1; s += kThreads) {
#pragma unroll
        for (int q = 0; q < Ch<R>::N; ++q) {
            Ch<R> v;
#pragma unroll
            for (int w = 0; w < Ch<R>::W; ++w) {
                const size_t k = (size_t)(q * Ch<R>::W + w) * d.V + s;
                const double2 bb = d.b64[k], aa = ax[k];
                v.c[w] = {fromdbl<R>(__dsub_rn(bb.x, aa.x)), fromdbl<R>(__dsub_rn(bb.y, aa.y))};
            }
            v.stv(r0, q, d.V, s);
            Ch<R> tv = Ch<R>::ld(rt, q, d.V, s);
#pragma unroll
            for (int w = 0; w < Ch<R>::W; ++w) {
                dots[0] = cjfma(tv.c[w], v.c[w], dots[0]);
                dots[1].r = fmaR(v.c[w].r, v.c[w].r, dots[1].r);
                dots[1].r = fmaR(v.c[w].i, v.c[w].i, dots[1].r);
            }
        }
    }
    reduce_store<2, R>(dots, d.part, gridDim.x, blockIdx.x);
    run_step<dfp_of<R>()>(d, step, n_partials<R>(gridDim.x), gridDim.x);
}

// ------------------------------------------------------------------ pseudo-double-pass gather
// y += sum_{m in [m_begin, m_end)} sum_k coef[m][k] v(m, k), the stored seed-vector
// occurrences of pass 1 (store slot (m - m0) * NC + k).  One thread per site and
// chunk (grid.x = chunks x site blocks), so a thread holds a few accumulators and
// many loads stay in flight.  Terms are summed in R in groups of four; each group
// enters a compensated FP32-pair accumulator (FP64 for an FP64 store), which is
// added to y in FP64 once.
template <typename R> struct GatherAcc {        // FP32 and double-float stores
    df a[2 * Ch<R>::W];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int k = 0; k < 2 * Ch<R>::W; ++k) a[k] = df(0.0f);
    }
    __device__ __forceinline__ static df widen(float x) { return df(x); }
    __device__ __forceinline__ static df widen(df x) { return x; }
    __device__ __forceinline__ void add(const cx<R> (&t)[Ch<R>::W]) {
#pragma unroll
        for (int w = 0; w < Ch<R>::W; ++w) {
            a[2 * w] = addR(a[2 * w], widen(t[w].r));
            a[2 * w + 1] = addR(a[2 * w + 1], widen(t[w].i));
        }
    }
    __device__ __forceinline__ double get(int k) const { return todbl(a[k]); }
};
template <> struct GatherAcc<double> {
    double a[2];
    __device__ __forceinline__ void zero() { a[0] = a[1] = 0.0; }
    __device__ __forceinline__ void add(const cx<double> (&t)[1]) {
        a[0] = __dadd_rn(a[0], t[0].r);
        a[1] = __dadd_rn(a[1], t[0].i);
    }
    __device__ __forceinline__ double get(int k) const { return a[k]; }
};

template <typename R>
__global__ void __launch_bounds__(kThreads)
k_gather(const SolverDev* __restrict__ ds) {
    const TraceScope trace_(trace_kind<R>(FA_TK_GATHER));
    const SolverDev& d = ds[blockIdx.y];
    const int nsb = (d.V + kThreads - 1) / kThreads;
    const int q = blockIdx.x / nsb;
    const int s = (blockIdx.x - q * nsb) * kThreads + threadIdx.x;
    if (q >= Ch<R>::N || s >= d.V) return;
    const int M = d.st->n_outer;
    int m_begin, m_end, m0;
    const typename Ch<R>::T* store;
    if (sizeof(R) == 8) {
        m_begin = 0;
        m_end = min(M, d.cap64);
        if (d.m0_32 >= 0) m_end = min(m_end, d.m0_32);
        m0 = 0;
        store = reinterpret_cast<const typename Ch<R>::T*>(d.store64);
    } else {
        if (d.m0_32 < 0) return;
        m_begin = d.m0_32;
        m_end = min(M, d.m0_32 + d.cap32);
        m0 = d.m0_32;
        store = reinterpret_cast<const typename Ch<R>::T*>(d.store32);
    }
    if (m_end <= m_begin) return;
    const size_t vs = vstride<R>(d);
    const int NC = nc_slots(d.L);
    const int n = (m_end - m_begin) * NC;
    const size_t cf0 = (size_t)m_begin * NC;
    const typename Ch<R>::T* base = store + (size_t)(m_begin - m0) * NC * vs;
    constexpr int W = Ch<R>::W;
    GatherAcc<R> acc;
    acc.zero();
    int k0 = 0;
    for (; k0 + 4 <= n; k0 += 4) {
        Ch<R> v[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) v[g] = Ch<R>::ld_cs(base + (size_t)(k0 + g) * vs, q, d.V, s);
        cx<R> t[W];
#pragma unroll
        for (int w = 0; w < W; ++w) t[w] = czero<R>();
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const cx<R> c = weight<R>(d.coef, d.coef4, cf0 + k0 + g);
#pragma unroll
            for (int w = 0; w < W; ++w) t[w] = cfma(c, v[g].c[w], t[w]);
        }
        acc.add(t);
    }
    if (k0 < n) {
        cx<R> t[W];
#pragma unroll
        for (int w = 0; w < W; ++w) t[w] = czero<R>();
        for (int k = k0; k < n; ++k) {
            const Ch<R> v = Ch<R>::ld_cs(base + (size_t)k * vs, q, d.V, s);
            const cx<R> c = weight<R>(d.coef, d.coef4, cf0 + k);
#pragma unroll
            for (int w = 0; w < W; ++w) t[w] = cfma(c, v.c[w], t[w]);
        }
        acc.add(t);
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
        double2* p = d.y + (size_t)(q * W + w) * d.V + s;
        double2 a = *p;
        a.x = __dadd_rn(a.x, acc.get(2 * w));
        a.y = __dadd_rn(a.y, acc.get(2 * w + 1));
        *p = a;
    }
}

// pass 2: advance the outer-iteration counter
__global__ void k_advance(const SolverDev* __restrict__ ds) {
    dep_wait();
    const TraceScope trace_(FA_TK_ADVANCE);
    DevState* S = ds[blockIdx.x].st;
    if (S->m < S->n_outer) S->m += 1;
}
// pass 2 starts at outer iteration min(m, M) of each system
__global__ void k_set_m(const SolverDev* __restrict__ ds, int m) {
    DevState* S = ds[blockIdx.x].st;
    S->m = m < S->n_outer ? m : S->n_outer;
    S->done = 0;
}
// done flag of every system (polled by the host)
__global__ void k_flags(const SolverDev* __restrict__ ds, int n, int* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = ds[i].st->done;
}

// ------------------------------------------------------------------ backward sweep
// One thread per shift walks its recorded linear operations backwards
// (adjoint of "dst <- sum a src + sum c v_occ"), starting from the adjoint
// lambda_X = 1 of its final solution; the adjoint of each seed-vector
// occurrence is that occurrence's weight in x_s.
//
// The walk is a serial chain of FP64 instructions in one warp (64 cycles each),
// so it carries only the adjoints lambda_U of the shift directions and leaves
// those that the weights need; k_coef_reduce forms the weights from them in
// parallel over outer iterations, slots and shifts.  The record of the next
// (earlier) iteration is fetched ahead.  With the weights formed in the walk it
// took 161 us on the 16^3 x 32 workload (52 outer iterations, l = 2).
// cs[shift][m]: slot_mr(j) = lambda_U[j+1] before sub-step j, slot_old(j, i) =
// lambda_U[i] in sub-step j before its scaling by -beta_s.
template <int L> struct SweepRec {
    double2 ips, as[L], bs[L], gam[L];
    __device__ __forceinline__ void load(const SolverDev& d, int sh, int m) {
        const double2* P = d.prec + ((size_t)sh * d.max_outer + m) * ps_stride(L);
        const double2* G = d.rec_gamma + m * (L + 1);
        ips = __ldg(P + 5 * L);
#pragma unroll
        for (int j = 0; j < L; ++j) {
            as[j] = __ldg(P + 5 * j);
            bs[j] = __ldg(P + 5 * j + 1);
            gam[j] = __ldg(G + j + 1);
        }
    }
};
template <int L>
__global__ void k_sweep(const SolverDev* __restrict__ ds) {
    const TraceScope trace_(FA_TK_SWEEP);
    const SolverDev& d = ds[blockIdx.y];
    const int sh = blockIdx.x * blockDim.x + threadIdx.x;
    if (sh >= d.ns) return;
    constexpr int NC = nc_slots(L);
    const int Ms = d.iters[sh];
    const double nsg = -d.sigma[sh];
    dcx lU[L + 1];
#pragma unroll
    for (int i = 0; i <= L; ++i) lU[i] = mk(0.0);
    SweepRec<L> next;
    if (Ms > 0) next.load(d, sh, Ms - 1);
    for (int m = Ms - 1; m >= 0; --m) {
        const SweepRec<L> R = next;
        if (m > 0) next.load(d, sh, m - 1);
        double2* out = d.cs + ((size_t)sh * d.max_outer + m) * NC;
        // MR, reversed: u0 <- (u0 - sum gamma_j u_j)/p_s
        const dcx t = zmul(lU[0], ld(R.ips));
#pragma unroll
        for (int jj = 1; jj <= L; ++jj) lU[jj] = zfma(zneg(ld(R.gam[jj - 1])), t, lU[jj]);
        lU[0] = t;
#pragma unroll
        for (int j = L - 1; j >= 0; --j) {
            // x += alpha_s u_0 with lambda_X = 1
            lU[0] = {__dadd_rn(R.as[j].x, lU[0].r), __dadd_rn(R.as[j].y, lU[0].i)};
            // u_{j+1} <- r_old_j/(alpha_s zeta) - r_j/(alpha_s zeta_new) - sigma u_j
            const dcx lu = lU[j + 1];
            out[slot_mr(L, j)] = pk(lu);
            lU[j] = zrfma(nsg, lu, lU[j]);
            lU[j + 1] = mk(0.0);
            // u_i <- r_old_i/zeta - beta_s u_i
            const dcx nbs = zneg(ld(R.bs[j]));
#pragma unroll
            for (int i = 0; i <= j; ++i) {
                out[slot_old(j, i)] = pk(lU[i]);
                lU[i] = zmul(nbs, lU[i]);
            }
        }
    }
}

// coef[m][k] = sum_s omega_s c_s[m][k] for m < M (fixed order over s), c_s the
// weight of occurrence k in x_s, from the adjoints that the sweep left and the
// shift's record.  32 (m, k) per block, a warp per eighth of the shifts.
__global__ void __launch_bounds__(256) k_coef_reduce(const SolverDev* __restrict__ ds) {
    const TraceScope trace_(FA_TK_COEF_REDUCE);
    const SolverDev& d = ds[blockIdx.y];
    const int L = d.L, M = d.st->n_outer, NC = nc_slots(L);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int idx = blockIdx.x * 32 + lane;
    const bool valid = idx < M * NC;
    const int m = idx / NC, k = idx - m * NC;
    __shared__ double2 w[kMaxShifts][32];
    // slot k: (j, i) of a sub-step, or the MR step's vector mr
    int j = 0;
    while (j < L && k >= (j + 1) * (j + 2) / 2) ++j;
    const int i = k - j * (j + 1) / 2, mr = j == L ? i : -1;
    for (int sh = warp; sh < d.ns; sh += 8) {
        if (!valid || m >= d.iters[sh]) continue;
        const double2* T = d.cs + ((size_t)sh * d.max_outer + m) * NC;
        const double2* P = d.prec + ((size_t)sh * d.max_outer + m) * ps_stride(L);
        dcx c;
        if (mr >= 0) {
            c = ld(P[5 * L + 1 + mr]);
            if (mr == L - 1) c = zfma(ld(T[slot_mr(L, mr)]), zneg(ld(P[5 * mr + 4])), c);
        } else if (i == j) {
            c = zfma(ld(T[slot_mr(L, j)]), ld(P[5 * j + 3]), mk(0.0));
            c = zfma(ld(T[k]), ld(P[5 * j + 2]), c);
        } else {
            c = zfma(ld(T[k]), ld(P[5 * j + 2]), mk(0.0));
            if (i == j - 1) c = zfma(ld(T[slot_mr(L, i)]), zneg(ld(P[5 * i + 4])), c);
        }
        w[sh][lane] = pk(d.omega[sh] * c);
    }
    __syncthreads();
    if (warp != 0 || !valid) return;
    dcx a = mk(0.0);
    for (int sh = 0; sh < d.ns; ++sh) {
        if (m >= d.iters[sh]) continue;
        a = a + ld(w[sh][lane]);
    }
    // and as an FP32 pair per part (hi = FP32 rounding, lo = rest)
    put_scalar(d.coef, d.coef4, (size_t)m * NC + k, a);
}

// single-pass result y = sum_s omega_s x_s (FP64 [12][V]) of each system
__global__ void k_combine_sys(const SolverDev* __restrict__ ds) {
    const SolverDev& d = ds[blockIdx.y];
    const int idx = blockIdx.x * kThreads + threadIdx.x;
    if (idx >= 12 * d.V) return;
    const size_t svs = (size_t)12 * d.V;
    double a = 0.0, b = 0.0;
    for (int sh = 0; sh < d.ns; ++sh) {
        const double2 v = d.xs[sh * svs + idx];
        a = __fma_rn(d.omega[sh], v.x, a);
        b = __fma_rn(d.omega[sh], v.y, b);
    }
    d.y[idx] = make_double2(a, b);
}

// single-pass result y = sum_s omega_s x_s (FP64 [12][V]); accumulate: y += that sum
__global__ void k_combine(int V, int ns, const double* omega, const double2* xs, size_t svs, double2* y,
                          int accumulate = 0) {
    const int idx = blockIdx.x * kThreads + threadIdx.x;
    if (idx >= 12 * V) return;
    double a = 0.0, b = 0.0;
    if (accumulate) {
        a = y[idx].x;
        b = y[idx].y;
    }
    for (int sh = 0; sh < ns; ++sh) {
        const double2 v = xs[sh * svs + idx];
        a = __fma_rn(omega[sh], v.x, a);
        b = __fma_rn(omega[sh], v.y, b);
    }
    y[idx] = make_double2(a, b);
}

}  // namespace fa
