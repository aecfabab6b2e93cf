// The FP64 Wilson-Dirac sweep, split over the eight hops of a site.
//
// What bounds it: the FP64 pipe.  A GB300 SM takes one FP64 warp instruction every 19
// cycles while its four sub-partitions all ask (add, multiply or FMA, dependent or not:
// 76 cycles per sub-partition, 0.53 T thread instructions/s at 2.06 GHz); a
// sub-partition alone gets one every 64.  A sweep takes 992 FP64 warp instructions
// per 32 sites here (ncu; 914 with a thread per site), so it takes 230 us on 16^3 x 32
// (17.6 cycles each) whatever the memory does (126 MB
// there: 19 us), and one warp that walks a whole site takes 28 us even on an idle
// chip.  One thread per site in 256-thread blocks put a 4^3 x 8 lattice on 2 of 152
// SMs (50-60 us per sweep) and left 3.4 waves of one block per SM on 16^3 x 32
// (270 us).
//
// So a tile is 32 consecutive sites and its work is spread over the warps of a
// block, and for small lattices over the blocks of a cluster:
//   phase 1: 16 units (hop, projected spin row); a warp projects the row of the
//            neighbour, multiplies it by the link and leaves three complex
//            numbers per site in shared memory;
//   phase 2: 24 real output components per tile; a thread adds the eight hops'
//            contributions to its component in the fixed order x+, x-, ... t-,
//            then the diagonal term.
// Every number is formed by the same operations in the same order whatever the
// split, so results do not depend on it.  C blocks of a cluster share a tile
// (hops 8/C each; phase 2 reads the other blocks' products through
// distributed shared memory): C = 1 is the least work per SM, larger C the
// shortest time when there are fewer tiles than SMs (rule in hop64_split).
//
// The hop is a runtime index (neighbour, partner spin, sign bits), not a
// template parameter: eight copies of the code would be fetched cold by every
// short launch, and the integer work hides under the FP64 pipe.
#pragma once

#include <cmath>

#include "fa_internal.cuh"

namespace fa {

constexpr int kTile64 = 32;   // sites of a tile: one warp, and one reduction partial
template <int C> constexpr int hop64_threads() { return C == 4 ? 128 : 256; }
// 3 blocks of 256 threads per SM: 24 warps cover the loads and the barriers
template <int C> constexpr int hop64_min_blocks() { return C == 4 ? 6 : 3; }
inline __host__ __device__ int tiles64(int V) { return (V + kTile64 - 1) / kTile64; }

// A spinor field with strides (in complex numbers) of site and component:
// internal layout (1, V), canonical layout (12, 1).
struct View64 {
    double2* p;
    int ss, ks;
    __device__ __forceinline__ double2 ld(int s, int k) const { return __ldg(p + (size_t)s * ss + (size_t)k * ks); }
};
__host__ __device__ inline View64 internal64(const double2* p, int V) { return {const_cast<double2*>(p), 1, V}; }
__host__ __device__ inline View64 canonical64(const double* p) { return {reinterpret_cast<double2*>(const_cast<double*>(p)), 12, 1}; }

// Operator scalars of one sweep: out = g5out? ((cdiag in' + chop sum of hops)), in' = g5in? g5 in : in
struct Op64 {
    double cdiag, chop, ef, eb, bc;
    int g5in, g5out;
};

template <int C> struct Smem64 {
    double2 hs[8 / C][6][kTile64];   // this block's hops: [hop][3 row + colour][site]
    double2 out[12][kTile64];        // sweep output (inner product, canonical store); rank 0's copy is read
};

__device__ __forceinline__ double flip(double x, unsigned neg) {   // x or -x
    return __hiloint2double(__double2hiint(x) ^ (int)(neg << 31), __double2loint(x));
}

// shared-memory address of `p` in block `rank` of the cluster, and accesses to it
__device__ __forceinline__ unsigned cluster_addr(const void* p, int rank) {
    unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ double ld_cluster(unsigned a) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
template <int C> __device__ __forceinline__ void tile_sync() {
    if constexpr (C == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// One sweep of tile `tile` by block `rank` of its cluster; every thread of the
// block calls it.  DIRECT: the output is stored to `out`; STAGE: it is left in
// rank 0's sm.out.
template <int C, bool DIRECT, bool STAGE>
__device__ __forceinline__ void hop64_tile(const Geom& g, const double2* __restrict__ U, const View64& in,
                                           const View64& out, const Op64& op, int tile, int rank, Smem64<C>& sm) {
    constexpr int NW = hop64_threads<C>() / 32;   // warps of the block
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int V = g.V;
    const int s = tile * kTile64 + lane;
    const bool valid = s < V;
    const int sv = valid ? s : V - 1;
    {
        const int X = g.X, Y = g.Y, Z = g.Z, T = g.T;
        const int x = sv % X, r1 = sv / X, y = r1 % Y, r2 = r1 / Y, z = r2 % Z, t = r2 / Z;
        constexpr int NU = 16 / C;                // units of the block
#pragma unroll 1
        for (int u = warp; u < NU; u += NW) {
            // C = 1: a warp takes both rows of one hop (u, u + 8), else consecutive units
            const int hl = C == 1 ? (u & 7) : (u >> 1);
            const int sp = C == 1 ? (u >> 3) : (u & 1);
            const int hop = rank * (8 / C) + hl;
            const int mu = hop >> 1;
            const unsigned bwd = hop & 1;
            // neighbour s +- mu_hat
            const int pos = mu == 0 ? x : mu == 1 ? y : mu == 2 ? z : t;
            const int ext = mu == 0 ? X : mu == 1 ? Y : mu == 2 ? Z : T;
            const int str = mu == 0 ? 1 : mu == 1 ? X : mu == 2 ? X * Y : X * Y * Z;
            const int nb = bwd ? (pos == 0 ? sv + (ext - 1) * str : sv - str)
                               : (pos == ext - 1 ? sv - (ext - 1) * str : sv + str);
            // row sp of (1 -+ g_mu) psi: psi_sp + phase psi_q, phase = +-1 (mu = 1, 3) or +-i (mu = 0, 2)
            const int q = mu < 2 ? 3 - sp : 2 + sp;
            const bool im = (mu & 1) == 0;
            // the phase's sign for the forward hop: - for mu 0 and 3, + - for mu 1, - + for mu 2
            unsigned neg = mu == 1 ? (unsigned)sp : (mu == 2 ? (unsigned)(1 - sp) : 1u);
            neg ^= bwd ^ (unsigned)(op.g5in != 0);
            double2 h[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double2 a = in.ld(nb, 3 * sp + c), b = in.ld(nb, 3 * q + c);
                h[c].x = __dadd_rn(a.x, flip(im ? b.y : b.x, im ? neg ^ 1u : neg));
                h[c].y = __dadd_rn(a.y, flip(im ? b.x : b.y, neg));
            }
            // U_mu(s) forward, U_mu(nb)^H backward
            const double2* L = U + (size_t)mu * 9 * V + (bwd ? nb : sv);
            const int ea = bwd ? 1 : 3, ec = bwd ? 3 : 1;   // element (a, c) at a ea + c ec
            const bool wt = mu == 3;
            const double w = bwd ? (t == 0 ? __dmul_rn(op.eb, op.bc) : op.eb)
                                 : (t == T - 1 ? __dmul_rn(op.ef, op.bc) : op.ef);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                double2 l = __ldg(L + (size_t)(a * ea) * V);
                double li = flip(l.y, bwd);
                double tr = __fma_rn(-li, h[0].y, __dmul_rn(l.x, h[0].x));
                double ti = __fma_rn(li, h[0].x, __dmul_rn(l.x, h[0].y));
#pragma unroll
                for (int c = 1; c < 3; ++c) {
                    l = __ldg(L + (size_t)(a * ea + c * ec) * V);
                    li = flip(l.y, bwd);
                    tr = __fma_rn(l.x, h[c].x, tr);
                    tr = __fma_rn(-li, h[c].y, tr);
                    ti = __fma_rn(l.x, h[c].y, ti);
                    ti = __fma_rn(li, h[c].x, ti);
                }
                if (wt) {
                    tr = __dmul_rn(w, tr);
                    ti = __dmul_rn(w, ti);
                }
                sm.hs[hl][3 * sp + a][lane] = make_double2(tr, ti);
            }
        }
    }
    tile_sync<C>();
    // real component ch = 2 (3 spin + colour) + part
    constexpr int NCH = 24 / C;
#pragma unroll 1
    for (int cl = warp; cl < NCH; cl += NW) {
        const int ch = rank * NCH + cl;
        const int k = ch >> 1, part = ch & 1;
        const int spin = k / 3, col = k - 3 * spin;
        const bool up = spin < 2;
        double acc = 0.0;
#pragma unroll
        for (int hop = 0; hop < 8; ++hop) {
            constexpr int HB = 8 / C;
            const int mu = hop >> 1;
            const unsigned bwd = hop & 1;
            // spins 0, 1: the row itself.  Spins 2, 3: the partner row times +-1 or +-i
            const bool im = (mu & 1) == 0;
            const int row = up ? spin : (mu < 2 ? 3 - spin : spin - 2);
            const int pt = (up || !im) ? part : 1 - part;
            // forward hop: mu 0: (-, +) for the (real, imaginary) part; mu 1: -, + for spins 2, 3;
            // mu 2: (-, +) and (+, -) for spins 2, 3; mu 3: -
            unsigned neg = mu == 0 ? (unsigned)(1 - part)
                         : mu == 1 ? (unsigned)(3 - spin)
                         : mu == 2 ? (unsigned)(part == 0 ? 3 - spin : spin - 2)
                                   : 1u;
            neg = up ? 0u : ((neg ^ bwd) & 1u);
            const double2* e = &sm.hs[hop % HB][3 * row + col][lane];
            double v;
            if constexpr (C == 1) v = pt ? e->y : e->x;
            else v = ld_cluster(cluster_addr(e, hop / HB) + 8u * (unsigned)pt);
            v = flip(v, neg);
            acc = hop == 0 ? v : __dadd_rn(acc, v);
        }
        const unsigned gin = (!up && op.g5in) ? 1u : 0u, gout = (!up && op.g5out) ? 1u : 0u;
        const double2 pv = in.ld(sv, k);
        const double p = flip(part ? pv.y : pv.x, gin ^ gout);
        const double o = __fma_rn(flip(op.chop, gout), acc, __dmul_rn(op.cdiag, p));
        if constexpr (DIRECT)
            if (valid) (&out.p[(size_t)s * out.ss + (size_t)k * out.ks].x)[part] = o;
        if constexpr (STAGE) {
            double* d = &sm.out[k][lane].x + part;
            if constexpr (C == 1) *d = valid ? o : 0.0;
            else st_cluster(cluster_addr(d, 0), valid ? o : 0.0);
        }
    }
    // distributed shared memory: no block leaves before the others have read it
    if constexpr (C > 1 || STAGE) tile_sync<C>();
}

// <dotv, out> over the tile from sm.out: warp 0 forms the real part, warp 1 the
// imaginary part, a site's 12 components in order, then a shuffle tree; the
// result is in thread 0 (call from every thread of the block that holds sm.out)
template <int C>
__device__ __forceinline__ double2 dot64_tile(const View64& dotv, int V, int tile, const Smem64<C>& sm) {
    __shared__ double im;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int s = tile * kTile64 + lane;
    double a = 0.0;
    if (warp < 2 && s < V) {
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const double2 q = dotv.ld(s, k), p = sm.out[k][lane];
            a = __fma_rn(q.x, warp ? p.y : p.x, a);
            a = __fma_rn(warp ? -q.y : q.y, warp ? p.x : p.y, a);
        }
    }
    if (warp < 2) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a = __dadd_rn(a, __shfl_down_sync(0xffffffffu, a, o));
    }
    if (threadIdx.x == 32) im = a;
    __syncthreads();
    return make_double2(a, im);
}

// sm.out to a canonical field, coalesced (a tile is 6 KB in a row there)
template <int C>
__device__ __forceinline__ void store_canonical(double2* out, int V, int tile, const Smem64<C>& sm) {
    const int n = min(kTile64, V - tile * kTile64) * 12;
    double2* o = out + (size_t)tile * kTile64 * 12;
    for (int e = threadIdx.x; e < n; e += hop64_threads<C>()) o[e] = sm.out[e % 12][e / 12];
}

// Blocks per tile.  A tile is 912 FP64 warp instructions, 228 per sub-partition
// with one block on an SM; the busiest SM takes ceil(tiles C / SMs) / C of that,
// which C = 2 or 4 lowers for few tiles and evens out for a few per SM; 8 % per
// doubling is charged for the cluster's barriers and remote reads.  Measured on
// GB300, 16 outer iterations of FP64 double pass from graphs, ms with C = 1 / 2 /
// 4: 512 sites 4.5 / 3.7 / 3.3, 2160 sites 4.6 / 3.7 / 3.8, 3456 sites 4.7 / 4.9 /
// 4.4, 4096 sites 4.6 / 4.9 / 4.9, 6144 sites 6.9 / 6.3 / 6.3, 16000 sites 12.1 /
// 11.7 / 11.7, 41472 sites 25.2 / 26.4 / 26.2; one sweep on 16^3 x 32 234 / 239 /
// 246 us.
inline int hop64_split(int V, int nsm) {
    if (nsm < 1) nsm = 152;
    const long long t = tiles64(V);
    int best = 1;
    double cost = 1e30;
    for (int C = 1; C <= 4; C *= 2) {
        const double f = (double)((t * C + nsm - 1) / nsm) / C * (C == 1 ? 1.0 : C == 2 ? 1.08 : 1.16);
        if (f < cost) {
            cost = f;
            best = C;
        }
    }
    return best;
}

// A thread per site instead (hop_site in hop_device.cuh; the same bits), in blocks of
// 128 threads at 255 registers: 914 FP64 warp instructions per 32 sites against the
// tile form's 992 (ncu), both at about 17.5 cycles of the SM's pipe (a probe: 19.0
// when all four sub-partitions ask in step, 16 would be its best); but a wave of
// one block per SM (19,456 sites) takes 31.2 us however few
// of its blocks there are, where the tile form takes 1.75 ns per site.  So it is
// used where the last wave is full enough (the busiest SM's blocks against the
// mean).  Measured on GB300, us per sweep, tiles / a thread per site: 32^3 x 64
// 3649 / 3348, 16^3 x 32 230 / 219, 155,648 sites (8.0 waves) 273 / 251, 98,304 (5.05)
// 179 / 187, 41,472 (2.1) 77 / 94, 16,384 33 / 32; with the inner product 32^3 x 64
// 4045 / 3643.
constexpr int kSite64 = 128, kSite64Blocks = 2;
inline int site64_blocks(int V) { return (V + kSite64 - 1) / kSite64; }
inline bool full_waves(double blocks, int nsm) {
    const double x = blocks / (nsm > 0 ? nsm : 152);
    return 0.93 * std::ceil(x) <= x;
}
inline bool hop64_by_site(long long blocks, int nsm) { return full_waves((double)blocks, nsm); }

// out = scale g5out (diag in' - 1/2 sum hops(in')), in' = g5in ? g5 in : in, one
// FP64 D_w sweep between fields of either layout.  A block returns at once
// when *done is set (done may be null).  after: launched programmatically behind
// the kernel before it in the stream (see launch_hop_f32).
int launch_hop_f64(const Geom& g, const double2* links, const View64& in, const View64& out, double diag, double ef,
                   double eb, double t_bc, double scale, bool g5in, bool g5out, const int* done, cudaStream_t st,
                   bool after = false);

// Kernel launch with programmatic stream serialization when `pdl` is set (see
// dep_wait) and in clusters of `cluster` blocks.
template <typename... KArgs, typename... Args>
inline void launch_ex(bool pdl, int cluster, void (*k)(KArgs...), dim3 grid, int block, cudaStream_t st, Args... args) {
    cudaLaunchAttribute at[2];
    int n = 0;
    if (pdl) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster;
        at[n].val.clusterDim.y = 1;
        at[n++].val.clusterDim.z = 1;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = n;
    (void)cudaLaunchKernelEx(&cfg, k, args...);   // errors surface through cudaGetLastError
}

}  // namespace fa
