// Wilson-Dirac hop kernels D_w(mu) for sm_103a, FP64 (18-real links) and
// FP32 (12-real links), plus layout conversions.
//
// D_w(mu) is named in Sec. 1 (the kernel of the overlap operator at nonzero
// chemical potential); the definition implemented is the standard mass form
//   (D psi)(x) = (4+m) psi(x) - 1/2 sum_nu [ f+ (1 - g_nu) U_nu(x) psi(x+nu)
//                                          + f- (1 + g_nu) U_nu(x-nu)^H psi(x-nu) ]
// with f+- = e^{+-mu} on time hops and the time-boundary sign on hops that
// cross t = T-1 <-> 0.  Each hop projects the neighbour spinor to a half
// spinor with the DeGrand-Rossi projector (1 -+ g_nu), multiplies the two
// colour vectors by the link and rebuilds the lower spin components.
//
// FP32: one thread per site; double-float: three, one per colour row; FP64: 32-site
// tiles, a warp per hop, or one thread per site (hop64.cuh).  The nearest-neighbour reuse of spinors and links is
// left to L1/L2 (the 126 MB L2 holds several time slices of every field even
// on 32^3 x 64).  Memory traffic floor per site and sweep: one spinor in, one
// out, four links (FP32: 96 + 96 + 4 * 48 = 384 B).
#include "hop64.cuh"
#include "hop_device.cuh"

namespace fa {

// FP32.  CANON: the result is written to the canonical field `canon` instead of
// `out`: each thread stores its record of 192 bytes itself, 32 bytes at a time
// where the field is 32-byte aligned, else 16.
template <bool G5IN, bool G5OUT, bool CANON, int NT, int MB>
__global__ void __launch_bounds__(NT, MB)
hop_kernel(Geom g, LinkView<float> U, SpinorView<float> in, SpinorView<float> out, double2* canon, float cdiag,
           float chop, float ef, float eb, float bc) {
    dep_wait();
    if (g.V <= kEarlySites) dep_launch();
    const int s = blockIdx.x * NT + threadIdx.x;
    cx<float> p[12];
    if (s < g.V) {
        hop_site<float, G5IN, G5OUT>(g, U, in, s, cdiag, chop, ef, eb, bc, p);
        if (!CANON) out.store(s, p);
    }
    if constexpr (CANON) {
        if (s >= g.V) return;
        double2* o = canon + (size_t)s * 12;
        if ((reinterpret_cast<uintptr_t>(canon) & 31u) == 0) {
#pragma unroll
            for (int k = 0; k < 12; k += 2) {
                double v[4] = {f2d_int(p[k].r), f2d_int(p[k].i), f2d_int(p[k + 1].r), f2d_int(p[k + 1].i)};
                asm volatile("st.global.cs.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(o + k), "d"(v[0]), "d"(v[1]), "d"(v[2]),
                             "d"(v[3]) : "memory");
            }
        } else {
#pragma unroll
            for (int k = 0; k < 12; ++k) o[k] = make_double2(f2d_int(p[k].r), f2d_int(p[k].i));
        }
    }
}

// Number of SMs of the current device (cached per device).
int sm_count() {
    static int cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (cache[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        cache[dev] = n;
    }
    return cache[dev];
}

bool hop_narrow(int V) {
    const int n = sm_count();
    return n > 0 && kHopNarrowBlocks > 0 && (V + kHopNarrowThreads - 1) / kHopNarrowThreads <= kHopNarrowBlocks * n;
}

// the same sweep split by colour row (double-float)
template <bool G5IN, bool G5OUT, bool CANON>
__global__ void __launch_bounds__(kRowThreads, rows_min_blocks<false>())
hop_rows_kernel(Geom g, LinkView<df> U, SpinorView<df> in, SpinorView<df> out, double2* canon, df cdiag, df chop, df ef,
                df eb, df bc) {
    dep_wait();
    if (g.V <= kEarlySites) dep_launch();
    const int a = row_of_thread(), s = site_of_thread(blockIdx.x);
    cx<df> o[4];
    hop_site_row_sh<G5IN, G5OUT>(g, U, in, s, a, s < g.V, cdiag, chop, ef, eb, bc, o);
    if (!CANON) {
        if (s < g.V) {
#pragma unroll
            for (int sp = 0; sp < 4; ++sp) out.st1(s, sp * 3 + a, o[sp]);
        }
    } else {
        __shared__ float4 turn[12][kRowSites + 1];
        const int i = (int)(threadIdx.x & (kRowSites - 1));
        if (s < g.V) {
#pragma unroll
            for (int sp = 0; sp < 4; ++sp) turn[sp * 3 + a][i] = make_float4(o[sp].r.hi, o[sp].r.lo, o[sp].i.hi, o[sp].i.lo);
        }
        __syncthreads();
        const int s0 = blockIdx.x * kRowSites, n = min(kRowSites, g.V - s0) * 12;
        for (int e = threadIdx.x; e < n; e += kRowThreads) {
            const float4 v = turn[e % 12][e / 12];
            __stcs(canon + (size_t)s0 * 12 + e, make_double2(__dadd_rn(f2d_int(v.x), f2d_int(v.y)),
                                                             __dadd_rn(f2d_int(v.z), f2d_int(v.w))));
        }
    }
}

// FP64: a tile of 32 sites per block or cluster (hop64.cuh).  CANON: canonical
// output, staged in shared memory (a thread of phase 2 holds one real number of
// every 192-byte record, so direct stores would write 8 bytes per 32-byte sector).
template <int C, bool CANON>
__global__ void __launch_bounds__(hop64_threads<C>(), hop64_min_blocks<C>())
hop64_kernel(Geom g, const double2* __restrict__ U, View64 in, View64 out, Op64 op, const int* done, int early) {
    dep_wait();
    if (early) dep_launch();
    if (done != nullptr && *done) return;
    __shared__ Smem64<C> sm;
    const int tile = blockIdx.x / C, rank = blockIdx.x % C;
    hop64_tile<C, !CANON, CANON>(g, U, in, out, op, tile, rank, sm);
    if (CANON && rank == 0) store_canonical<C>(out.p, g.V, tile, sm);
}

// FP64 between internal fields, a thread per site (rule: hop64_by_site)
template <bool G5OUT>
__global__ void __launch_bounds__(kSite64, kSite64Blocks)
hop64_site_kernel(Geom g, LinkView<double> U, SpinorView<double> in, SpinorView<double> out, Op64 op, const int* done) {
    dep_wait();
    if (done != nullptr && *done) return;
    const int s = blockIdx.x * kSite64 + threadIdx.x;
    if (s >= g.V) return;
    cx<double> p[12];
    hop_site<double, false, G5OUT>(g, U, in, s, op.cdiag, op.chop, op.ef, op.eb, op.bc, p);
    out.store(s, p);
}

template <int C>
static int launch_hop64(const Geom& g, const double2* links, const View64& in, const View64& out, const Op64& op,
                        const int* done, cudaStream_t st, bool after) {
    const dim3 grid(tiles64(g.V) * C);
    // (the successor's blocks must find SMs of their own: they share an SM's FP64 pipe)
    const int early = 2 * (int)grid.x <= sm_count() ? 1 : 0;
    if (out.ks == 1) launch_ex(after, C, hop64_kernel<C, true>, grid, hop64_threads<C>(), st, g, links, in, out, op, done, early);
    else launch_ex(after, C, hop64_kernel<C, false>, grid, hop64_threads<C>(), st, g, links, in, out, op, done, early);
    return launch_status("FP64 hop kernel");
}

int launch_hop_f64(const Geom& g, const double2* links, const View64& in, const View64& out, double diag, double ef,
                   double eb, double t_bc, double scale, bool g5in, bool g5out, const int* done, cudaStream_t st,
                   bool after) {
    const Op64 op{scale * diag, -0.5 * scale, ef, eb, t_bc, g5in ? 1 : 0, g5out ? 1 : 0};
    const int nb = site64_blocks(g.V);
    if (in.ss == 1 && out.ss == 1 && !g5in && hop64_by_site(nb, sm_count())) {
        const SpinorView<double> vi{in.p, g.V}, vo{out.p, g.V};
        const LinkView<double> U{links, g.V};
        if (g5out) launch_ex(after, 1, hop64_site_kernel<true>, dim3(nb), kSite64, st, g, U, vi, vo, op, done);
        else launch_ex(after, 1, hop64_site_kernel<false>, dim3(nb), kSite64, st, g, U, vi, vo, op, done);
        return launch_status("FP64 hop kernel");
    }
    switch (hop64_split(g.V, sm_count())) {
        case 1: return launch_hop64<1>(g, links, in, out, op, done, st, after);
        case 2: return launch_hop64<2>(g, links, in, out, op, done, st, after);
        default: return launch_hop64<4>(g, links, in, out, op, done, st, after);
    }
}

int launch_hop_df(const Geom& g, const float4* links, const float4* in, float4* out, double* canon, double diag,
                  double ef, double eb, double t_bc, double scale, bool g5in, bool g5out, cudaStream_t st, bool after) {
    LinkView<df> U{links, g.V};
    SpinorView<df> vin{const_cast<float4*>(in), g.V};
    SpinorView<df> vout{out, g.V};
    double2* cn = reinterpret_cast<double2*>(canon);
    const df cdiag = host_cvt<df>(scale * diag), chop = host_cvt<df>(-0.5 * scale);
    const df ref = host_cvt<df>(ef), reb = host_cvt<df>(eb), rbc = host_cvt<df>(t_bc);
    const int nb = row_blocks(g.V);
    auto go = [&](auto kernel) {
        launch_ex(after, 1, kernel, dim3(nb), kRowThreads, st, g, U, vin, vout, cn, cdiag, chop, ref, reb, rbc);
    };
    if (!g5in && !g5out) canon ? go(hop_rows_kernel<false, false, true>) : go(hop_rows_kernel<false, false, false>);
    else if (!g5in && g5out) canon ? go(hop_rows_kernel<false, true, true>) : go(hop_rows_kernel<false, true, false>);
    else if (g5in && g5out) canon ? go(hop_rows_kernel<true, true, true>) : go(hop_rows_kernel<true, true, false>);
    else return FA_EINVAL;
    return launch_status("hop kernel");
}

template <bool G5IN, bool G5OUT, typename... A>
static void launch_hop32(bool after, bool narrow, bool canon, int nb, cudaStream_t st, A... args) {
    constexpr int NT = kHopNarrowThreads, MB = kHopNarrowBlocks, WT = kThreads, WB = FA_HOP_MINB;
    if (narrow && canon) launch_ex(after, 1, hop_kernel<G5IN, G5OUT, true, NT, MB>, dim3(nb), NT, st, args...);
    else if (narrow) launch_ex(after, 1, hop_kernel<G5IN, G5OUT, false, NT, MB>, dim3(nb), NT, st, args...);
    else if (canon) launch_ex(after, 1, hop_kernel<G5IN, G5OUT, true, WT, WB>, dim3(nb), WT, st, args...);
    else launch_ex(after, 1, hop_kernel<G5IN, G5OUT, false, WT, WB>, dim3(nb), WT, st, args...);
}

int launch_hop_f32(const Geom& g, const float4* links, const float4* in, float4* out, double* canon, double diag,
                   double ef, double eb, double t_bc, double scale, bool g5in, bool g5out, cudaStream_t st, int shape,
                   bool after) {
    LinkView<float> U{links, g.V};
    SpinorView<float> vin{const_cast<float4*>(in), g.V};
    SpinorView<float> vout{out, g.V};
    double2* cn = reinterpret_cast<double2*>(canon);
    const float cdiag = (float)(scale * diag), chop = (float)(-0.5 * scale);
    const float ref = (float)ef, reb = (float)eb, rbc = (float)t_bc;
    const bool narrow = hop_use_narrow(shape, g.V);
    const int nt = narrow ? kHopNarrowThreads : kThreads;
    const int nb = (g.V + nt - 1) / nt;
    if (!g5in && !g5out)
        launch_hop32<false, false>(after, narrow, canon != nullptr, nb, st, g, U, vin, vout, cn, cdiag, chop, ref, reb, rbc);
    else if (!g5in && g5out)
        launch_hop32<false, true>(after, narrow, canon != nullptr, nb, st, g, U, vin, vout, cn, cdiag, chop, ref, reb, rbc);
    else if (g5in && g5out)
        launch_hop32<true, true>(after, narrow, canon != nullptr, nb, st, g, U, vin, vout, cn, cdiag, chop, ref, reb, rbc);
    else return FA_EINVAL;
    return launch_status("hop kernel");
}

// ------------------------------------------------------------------ link force (adjoint)
// For the bilinears B_p = <a_p, D_w(mu) b_p> (p = 1, 2) the variation under a
// link change dU_nu(x) is sum_ij [dU_ij M_ij + conj(dU_ji) K_ij] with
//   M_ij = -1/2 f+ sum_s conj(a_si(x))      ((1 - g_nu) b(x+nu))_sj   (forward hop at x)
//   K_ij = -1/2 f- sum_s conj(a_si(x+nu))   ((1 + g_nu) b(x))_sj      (backward hop at x+nu)
// so Re dB = Re tr(G^H dU) with G = conj(M) + K^T.  The kernel adds
// w * (G_1 + G_2) to the canonical gradient array and writes per-block partials
// of w * (dB_1/dmu + dB_2/dmu), dB/dmu = sum M_ij U_ij - sum K_ij conj(U_ji) on
// time links.  a_1 enters as gamma_5 a_1 when G5A1 is set.
template <int MU>
__device__ __forceinline__ void force_dir(int s, int nb, double fp, double fm, const LinkView<double>& U,
                                          const SpinorView<double> a[2], const SpinorView<double> b[2],
                                          double w, double2* Gout, cx<double>& dmu) {
    cx<double> Gm[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) Gm[i][j] = czero<double>();
    cx<double> Uc[3][3];
    if (MU == 3) U.load(3, s, Uc);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        cx<double> ax[12], an[12], bx[12], bn[12], Pb[12], Qb[12], h[6];
        a[p].load(s, ax);
        a[p].load(nb, an);
        b[p].load(s, bx);
        b[p].load(nb, bn);
        if (p == 0) {
#pragma unroll
            for (int k = 6; k < 12; ++k) { ax[k] = {-ax[k].r, -ax[k].i}; an[k] = {-an[k].r, -an[k].i}; }
        }
#pragma unroll
        for (int k = 0; k < 12; ++k) { Pb[k] = czero<double>(); Qb[k] = czero<double>(); }
        project<MU, +1>(bn, h);
        recon_add<MU, +1>(Pb, h);
        project<MU, -1>(bx, h);
        recon_add<MU, -1>(Qb, h);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                cx<double> m = czero<double>(), k = czero<double>();
#pragma unroll
                for (int sp = 0; sp < 4; ++sp) {
                    m = cjfma(ax[3 * sp + i], Pb[3 * sp + j], m);
                    k = cjfma(an[3 * sp + i], Qb[3 * sp + j], k);
                }
                m = cscale(-0.5 * fp, m);
                k = cscale(-0.5 * fm, k);
                // G_ij += conj(M_ij); G_ji += K_ij
                Gm[i][j] = cadd(Gm[i][j], cx<double>{m.r, -m.i});
                Gm[j][i] = cadd(Gm[j][i], k);
                if (MU == 3) {
                    dmu = cfma(m, Uc[i][j], dmu);                                     // + M_ij U_ij
                    dmu = cfma(cx<double>{-k.r, -k.i}, cx<double>{Uc[j][i].r, -Uc[j][i].i}, dmu);  // - K_ij conj(U_ji)
                }
            }
    }
    double2* g = Gout + ((size_t)s * 4 + MU) * 9;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        double2 v = g[e];
        v.x = __fma_rn(w, Gm[e / 3][e % 3].r, v.x);
        v.y = __fma_rn(w, Gm[e / 3][e % 3].i, v.y);
        g[e] = v;
    }
}

__global__ void __launch_bounds__(kThreads)
k_force(Geom g, LinkView<double> U, SpinorView<double> a1, SpinorView<double> b1, SpinorView<double> a2,
        SpinorView<double> b2, double2* G, double w, double ef, double eb, double bc, double2* partials) {
    const int s = blockIdx.x * kThreads + threadIdx.x;
    cx<double> dm[1] = {czero<double>()};
    if (s < g.V) {
        const int X = g.X, Y = g.Y, Z = g.Z, T = g.T;
        const int x = s % X, r1 = s / X, y = r1 % Y, r2 = r1 / Y, z = r2 % Z, t = r2 / Z;
        const int sY = X, sZ = X * Y, sT = X * Y * Z;
        const SpinorView<double> a[2] = {a1, a2};
        const SpinorView<double> b[2] = {b1, b2};
        force_dir<0>(s, (x == X - 1) ? s - (X - 1) : s + 1, 1.0, 1.0, U, a, b, w, G, dm[0]);
        force_dir<1>(s, (y == Y - 1) ? s - (Y - 1) * sY : s + sY, 1.0, 1.0, U, a, b, w, G, dm[0]);
        force_dir<2>(s, (z == Z - 1) ? s - (Z - 1) * sZ : s + sZ, 1.0, 1.0, U, a, b, w, G, dm[0]);
        // forward hop at x crosses the boundary from t = T-1; so does the backward hop at x + t_hat
        const double fp = (t == T - 1) ? ef * bc : ef;
        const double fm = (t == T - 1) ? eb * bc : eb;
        force_dir<3>(s, (t == T - 1) ? s - (T - 1) * sT : s + sT, fp, fm, U, a, b, w, G, dm[0]);
        dm[0] = cscale(w, dm[0]);
    }
    block_reduce_store<1, double>(dm, partials, 0);
}

int launch_force(const Geom& g, const double2* links, const double2* a1, const double2* b1, const double2* a2,
                 const double2* b2, double* G_canon, double w, double ef, double eb, double t_bc,
                 double2* partials, cudaStream_t st) {
    LinkView<double> U{links, g.V};
    SpinorView<double> va1{const_cast<double2*>(a1), g.V}, vb1{const_cast<double2*>(b1), g.V};
    SpinorView<double> va2{const_cast<double2*>(a2), g.V}, vb2{const_cast<double2*>(b2), g.V};
    k_force<<<nblocks(g.V), kThreads, 0, st>>>(g, U, va1, vb1, va2, vb2, (double2*)G_canon, w, ef, eb, t_bc,
                                                partials);
    return launch_status("hop kernel");
}

// ------------------------------------------------------------------ layout conversions
// canonical spinor: double [V][12][2]; element (s, k) at 2*(12 s + k).
//
// A block turns a tile of 64 sites round in shared memory, so that the 12 KB of
// canonical records and the rows of 64 internal elements both move in whole
// lines (one thread per internal element read 16 bytes of every 192: each
// 32-byte sector was fetched twice and on lattices beyond L2 every record six
// times).  Measured on GB300, 32^3 x 64, before -> after: double-float pack
// 502 -> 137 us, FP64 unpack 268 -> 135 us (786 MB: 118 us at the copy rate).
constexpr int kPackSites = 64;
template <typename R> struct PackOut;   // element q of a site from its 12 complex numbers
template <> struct PackOut<double> {
    using T = double2;
    static constexpr int N = 12;
    __device__ static T get(const double2* c, int q) { return c[q]; }
};
template <> struct PackOut<float> {
    using T = float4;
    static constexpr int N = 6;
    __device__ static T get(const double2* c, int q) {
        const double2 a = c[2 * q], b = c[2 * q + 1];
        return make_float4(d2f_int(a.x), d2f_int(a.y), d2f_int(b.x), d2f_int(b.y));
    }
};
template <> struct PackOut<df> {
    using T = float4;
    static constexpr int N = 12;
    __device__ static T get(const double2* c, int q) {
        const float2 r = d2df_int(c[q].x), i = d2df_int(c[q].y);
        return make_float4(r.x, r.y, i.x, i.y);
    }
};

template <typename R>
__global__ void __launch_bounds__(kThreads)
pack_kernel(int V, const double2* __restrict__ canon, typename PackOut<R>::T* __restrict__ out) {
    __shared__ double2 rec[kPackSites][13];   // odd stride in 16-byte units: no bank conflicts across sites
    if (V <= kEarlySites) dep_launch();
    const int s0 = blockIdx.x * kPackSites, ns = min(kPackSites, V - s0);
#pragma unroll
    for (int r = 0; r < 12 * kPackSites / kThreads; ++r) {
        const int e = r * kThreads + threadIdx.x;
        if (e < 12 * ns) rec[e / 12][e % 12] = __ldcs(canon + (size_t)s0 * 12 + e);
    }
    __syncthreads();
    const int i = threadIdx.x % kPackSites;
    if (i >= ns) return;
    for (int q = threadIdx.x / kPackSites; q < PackOut<R>::N; q += kThreads / kPackSites)
        out[(size_t)q * V + s0 + i] = PackOut<R>::get(rec[i], q);
}

__global__ void __launch_bounds__(kThreads)
unpack_f64_kernel(int V, const double2* __restrict__ in, double2* __restrict__ canon) {
    __shared__ double2 rec[kPackSites][13];
    const int s0 = blockIdx.x * kPackSites, ns = min(kPackSites, V - s0);
    const int i = threadIdx.x % kPackSites;
    if (i < ns) {
#pragma unroll
        for (int q = 0; q < 12; q += kThreads / kPackSites) {
            const int k = q + threadIdx.x / kPackSites;
            rec[i][k] = in[(size_t)k * V + s0 + i];
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 12 * kPackSites / kThreads; ++r) {
        const int e = r * kThreads + threadIdx.x;
        if (e < 12 * ns) canon[(size_t)s0 * 12 + e] = rec[e / 12][e % 12];
    }
}

__global__ void convert_f64_f32_kernel(int V, const double2* __restrict__ in, float4* __restrict__ out) {
    const int idx = blockIdx.x * kThreads + threadIdx.x;   // idx = q*V + s
    if (idx >= 6 * V) return;
    const int q = idx / V, s = idx - q * V;
    const double2 a = in[(size_t)(2 * q) * V + s], b = in[(size_t)(2 * q + 1) * V + s];
    out[idx] = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
}

// canonical links: double [V][4][3][3][2]
__device__ __forceinline__ float4 to_df4(double2 v) {
    const float rh = __double2float_rn(v.x), ih = __double2float_rn(v.y);
    return make_float4(rh, __double2float_rn(__dsub_rn(v.x, (double)rh)), ih,
                       __double2float_rn(__dsub_rn(v.y, (double)ih)));
}

__global__ void pack_links_kernel(int V, const double2* __restrict__ canon, double2* __restrict__ l64,
                                  float4* __restrict__ l32, float4* __restrict__ ldf) {
    const int idx = blockIdx.x * kThreads + threadIdx.x;   // idx = mu*V + s
    if (idx >= 4 * V) return;
    const int mu = idx / V, s = idx - mu * V;
    const double2* src = canon + ((size_t)s * 4 + mu) * 9;
    double2 e[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) e[k] = src[k];
#pragma unroll
    for (int k = 0; k < 9; ++k) l64[((size_t)mu * 9 + k) * V + s] = e[k];
    if (ldf != nullptr) {
#pragma unroll
        for (int k = 0; k < 9; ++k) ldf[((size_t)mu * 9 + k) * V + s] = to_df4(e[k]);
    }
    if (l32 != nullptr) {
#pragma unroll
        for (int q = 0; q < 3; ++q)
            l32[((size_t)mu * 3 + q) * V + s] =
                make_float4((float)e[2 * q].x, (float)e[2 * q].y, (float)e[2 * q + 1].x, (float)e[2 * q + 1].y);
    }
}

static int grid_for(size_t n) { return (int)((n + kThreads - 1) / kThreads); }

static int pack_blocks(int V) { return (V + kPackSites - 1) / kPackSites; }

int launch_pack_spinor_f64(const Geom& g, const double* canon, double2* out, cudaStream_t st) {
    pack_kernel<double><<<pack_blocks(g.V), kThreads, 0, st>>>(g.V, (const double2*)canon, out);
    return launch_status("layout conversion kernel");
}
int launch_unpack_spinor_f64(const Geom& g, const double2* in, double* canon, cudaStream_t st) {
    unpack_f64_kernel<<<pack_blocks(g.V), kThreads, 0, st>>>(g.V, in, (double2*)canon);
    return launch_status("layout conversion kernel");
}
int launch_pack_spinor_f32(const Geom& g, const double* canon, float4* out, cudaStream_t st) {
    pack_kernel<float><<<pack_blocks(g.V), kThreads, 0, st>>>(g.V, (const double2*)canon, out);
    return launch_status("layout conversion kernel");
}
int launch_pack_spinor_df(const Geom& g, const double* canon, float4* out, cudaStream_t st) {
    pack_kernel<df><<<pack_blocks(g.V), kThreads, 0, st>>>(g.V, (const double2*)canon, out);
    return launch_status("layout conversion kernel");
}
int launch_pack_links(const Geom& g, const double* canon, double2* l64, float4* l32, float4* ldf, cudaStream_t st) {
    pack_links_kernel<<<grid_for((size_t)4 * g.V), kThreads, 0, st>>>(g.V, (const double2*)canon, l64, l32, ldf);
    return launch_status("layout conversion kernel");
}

// double-float -> FP32 ([12][V] float4 -> [6][V] float4): hi + lo rounded once
__global__ void convert_df_f32_kernel(int V, const float4* __restrict__ in, float4* __restrict__ out) {
    const int idx = blockIdx.x * kThreads + threadIdx.x;   // idx = q*V + s
    if (idx >= 6 * V) return;
    const int q = idx / V, s = idx - q * V;
    const float4 a = in[(size_t)(2 * q) * V + s], b = in[(size_t)(2 * q + 1) * V + s];
    out[idx] = make_float4(__fadd_rn(a.x, a.y), __fadd_rn(a.z, a.w), __fadd_rn(b.x, b.y), __fadd_rn(b.z, b.w));
}

int launch_convert_df_to_f32(const Geom& g, const float4* in, float4* out, cudaStream_t st) {
    convert_df_f32_kernel<<<grid_for((size_t)6 * g.V), kThreads, 0, st>>>(g.V, in, out);
    return launch_status("layout conversion kernel");
}
int launch_convert_f64_to_f32(const Geom& g, const double2* in, float4* out, cudaStream_t st) {
    convert_f64_f32_kernel<<<grid_for((size_t)6 * g.V), kThreads, 0, st>>>(g.V, in, out);
    return launch_status("layout conversion kernel");
}

}  // namespace fa
