/*
 * fapath — f(A) b by multi-shift BiCGstab(l), single-pass and double-pass,
 * on one NVIDIA GB300 (sm_103a).
 *
 * What is computed (Heybrock, "Double-pass variants for multi-shift
 * BiCGstab(l)", Lattice 2010):
 *
 *     y = f(A) b ~= sum_{s=1}^{Ns} omega_s (A + sigma_s)^{-1} b      (Eq. 1)
 *     A = c (gamma_5 D_w(mu))^2                                      (Sec. 1)
 *
 * D_w(mu) is the Wilson-Dirac operator with chemical potential (named in
 * Sec. 1, Eq. for D_ov; the definition used here is the standard mass form)
 *
 *   (D psi)(x) = (4+m) psi(x) - 1/2 sum_nu [ f+ (1-g_nu) U_nu(x) psi(x+nu)
 *                                          + f- (1+g_nu) U_nu(x-nu)^H psi(x-nu) ]
 *
 * with f+- = e^{+-mu} on time hops, 1 on spatial hops, times t_bc on hops that
 * cross the time boundary; gamma matrices in the DeGrand-Rossi basis,
 * gamma_5 = diag(1, 1, -1, -1).
 *
 * Canonical layouts (the only layouts that cross this boundary), C order,
 * interleaved complex128 (re, im):
 *   spinor  [T][Z][Y][X][spin 4][colour 3]             24 doubles per site
 *   gauge   [T][Z][Y][X][mu 4][row 3][col 3]           72 doubles per site
 *           mu = 0,1,2,3 <-> x,y,z,t; U_mu(x) links x to x + mu_hat.
 * Spinor arguments are DEVICE pointers unless the name says host.  The caller
 * owns them; the context owns its packed copies of the gauge field and all
 * work space.  Vectors must not alias unless stated.
 *
 * Errors: every call returns an fa_status (0 = FA_OK).  No call aborts or
 * throws.  A failed CUDA call returns FA_ECUDA and leaves a message for
 * fa_last_error().  Calls on one context are stream-ordered on the stream
 * given to fa_create(); they are not thread-safe on a shared context.
 */
#ifndef FAPATH_H
#define FAPATH_H

#ifdef __cplusplus
extern "C" {
#endif

typedef struct fa_ctx fa_ctx;

typedef enum {
    FA_OK = 0,
    FA_EINVAL = -1,       /* bad argument (null pointer, size, range)          */
    FA_ENOMEM = -2,       /* device or host allocation failed                  */
    FA_ECUDA = -3,        /* a CUDA runtime call failed; see fa_last_error()   */
    FA_EBREAKDOWN = -4,   /* a Krylov denominator vanished                      */
    FA_ENOCONV = -5,      /* not all shifts converged within max_outer         */
    FA_ENONFINITE = -6,   /* a recurrence scalar became NaN or Inf             */
    FA_ETIMEOUT = -7,     /* a bounded device wait expired                      */
    FA_ESTATE = -8        /* call out of order (no gauge field, no poles, ...) */
} fa_status;

/* FA_SINGLE: shift vectors updated alongside the seed (Sec. 3 "1-pass").
 * FA_DOUBLE: Sec. 2 option 1, pass 2 regenerates the seed vectors.  Pass 2 takes
 *            no memory that pass 1 does not hold; with FA_F32 and l > 2 a solve
 *            holds l - 2 spinors (l - 1 with reliable updates) besides its 2 l + 4.
 * FA_PSEUDO: Sec. 2 option 2, pass 1 stores the seed-vector occurrences of as
 *            many outer iterations as store_gb allows (a contiguous prefix);
 *            the rest, if any, is regenerated by a pass 2 from a snapshot. */
typedef enum { FA_SINGLE = 0, FA_DOUBLE = 1, FA_PSEUDO = 2 } fa_mode;

typedef enum {
    FA_F64 = 0,           /* FP64 spinors, FP64 18-real links, FP64 scalars          */
    FA_F32 = 1,           /* FP32 spinors, FP32 12-real links, FP64 scalars/reductions */
    FA_MIXED = 2,         /* FP64 head until every live shift residual is below
                             switch_resid |b|, then FP32 bulk (double-pass only)     */
    FA_DF = 3,            /* double-float: each real an unevaluated pair of FP32
                             numbers (about 44 bits), computed on the FP32 pipes;
                             operator entry points only                           */
    FA_MIXED_DF = 4       /* like FA_MIXED with a double-float head instead of FP64 */
} fa_precision;

typedef struct {
    int ell;              /* BiCGstab(l) degree, 1..8                                  */
    double tol;           /* per shift: stop when |r_0| / |zeta_s| <= tol |b|          */
    int max_outer;        /* outer-iteration cap (also sizes the scalar record)        */
    int mode;             /* fa_mode                                                   */
    int precision;        /* fa_precision                                              */
    double switch_resid;  /* FA_MIXED: head/tail switch threshold; <= 0:
                             min(0.04/l^2, 0.4/l^6)                                  */
    int flags;            /* bit 0: time the passes with CUDA events; bit 1: time the
                             hop kernels (see fa_hop_timing); bit 2: replay each outer
                             iteration from a captured CUDA graph (needs a non-default
                             stream; hop timing is off while replaying); bit 3: fixed
                             cost: run exactly max_outer outer iterations unless every
                             shift converges first, then freeze the remaining shifts and
                             finish normally (no FA_ENOCONV; the fixed-M l runs of
                             Sec. 3, Fig. 2); bit 4: plain stream order between the
                             kernels of an outer iteration (by default each kernel is
                             launched with programmatic stream serialization, so its
                             launch overlaps the end of the previous one; results are
                             the same bit for bit either way); bit 5: FP32 stretches
                             of a one-system double-pass solve (l <= 4) with the MR
                             Gram matrix in a kernel of its own (by default the last
                             D_w sweep of each outer iteration forms it in its
                             epilogue; the results differ only in the summation
                             order of the Gram entries)                             */
    double store_gb;      /* FA_PSEUDO: device memory for stored occurrences, GB;
                             <= 0: min(16, a quarter of the free memory)                */
    int reliable_every;   /* > 0: accumulate the seed solution x in FP64 and, after every
                             reliable_every-th outer iteration, replace r_0 by the FP64
                             true residual b - A x (replayed identically in pass 2);
                             one system per call.  0: off                               */
    int shift_chunk;      /* fa_grad: solve for at most this many poles at a time, so
                             that device memory holds 2 shift_chunk (l + 2) FP64 shift
                             spinors instead of 2 N_s (l + 2); <= 0 or >= N_s: all at
                             once.  Other calls ignore it.                            */
} fa_solver_params;

typedef struct {
    int status;               /* fa_status of the solve                              */
    int outer_iters;          /* M: outer iterations of pass 1                        */
    int switch_outer;         /* FA_MIXED: first FP32 outer iteration, else -1        */
    int ns;                   /* number of shifts                                     */
    int iters_per_shift[64];  /* M_s: outer iterations until shift s froze            */
    double resid_recurrence;  /* |r_0| / |b| of the seed at the end of pass 1         */
    long long n_mv;           /* matrix-vector products A v (both passes)             */
    long long n_dot;          /* global inner products                                */
    long long n_launch;       /* kernel launches by the context so far                */
    int stored_outer;         /* FA_PSEUDO: outer iterations whose occurrences were stored */
    double t_pass1_ms, t_sweep_ms, t_pass2_ms;   /* with flags bit 0, else 0          */
} fa_solver_stats;

/* Create a context for an X*Y*Z*T lattice (each extent >= 2, V = XYZT <=
 * 2^26 sites) whose work runs on `cuda_stream` (a cudaStream_t; NULL = the
 * legacy default stream) of the current device.  *out receives the handle. */
int fa_create(fa_ctx** out, const int dims[4], void* cuda_stream);

/* Release all device memory of the context.  NULL is accepted. */
int fa_destroy(fa_ctx* ctx);

/* Load the gauge field (canonical complex128 layout above) from host memory
 * (on_device = 0) or device memory (on_device = 1).  Packs FP64 18-real links
 * and FP32 12-real links (rows 1-2; row 3 = conj(row1 x row2) is rebuilt in
 * registers, exact for SU(3)).  The boundary sign and e^{+-mu} are kept as
 * separate scalars, never folded into the links. */
int fa_set_gauge(fa_ctx* ctx, const double* U, int on_device);

/* Use the packed gauge field of `owner` (same lattice shape and device)
 * instead of a copy: systems on one gauge field, such as the 12 spin-colour
 * sources of a propagator, then read one set of links.  The owner must keep
 * its gauge field and outlive ctx; a later fa_set_gauge(ctx, ...) gives ctx
 * its own copy again. */
int fa_share_gauge(fa_ctx* ctx, const fa_ctx* owner);

/* Wilson mass m (diagonal 4+m), chemical potential mu, time-boundary sign
 * t_bc (+1 periodic, -1 antiperiodic) and the scale c of A = c (g5 D)^2. */
int fa_set_params(fa_ctx* ctx, double wilson_mass, double mu, int t_bc, double scale_c);

/* Power iteration for the scale (workload recipe): v = v0/|v0|, then `iters`
 * times v <- A1 v/|A1 v| with A1 = (g5 D)^2 (c = 1), lambda = |A1 v|;
 * *scale_out = 1/lambda.  v0 is a device spinor (canonical), not modified.
 * FP64 throughout.  Does not change the context's c. */
int fa_estimate_scale(fa_ctx* ctx, const double* v0, int iters, double* scale_out);

/* Poles {omega_s, sigma_s} of Eq. (1), 1 <= ns <= 64, sigma_s > 0 (host arrays). */
int fa_set_poles(fa_ctx* ctx, int ns, const double* omega, const double* sigma);

/* Neuberger's poles (captions of Figs. 1, 3): theta_s = pi (s - 1/2)/(2 ns),
 * omega_s = (1/ns)/cos^2 theta_s, sigma_s = tan^2 theta_s (host arrays). */
int fa_neuberger_poles(int ns, double* omega, double* sigma);

/* Zolotarev's poles (the expansion the caption of Fig. 3 names for small mu):
 * the best uniform approximation x sum_s omega_s / (x^2 + sigma_s) of sign(x)
 * on eps <= |x| <= 1, i.e. of z^{-1/2} on [eps^2, 1] in the relative sense, with
 * ns poles (1 <= ns <= 64, 0 < eps < 1); sigma_s = eps^2 sn^2 / cn^2 at
 * (2s - 1) K' / (2 ns) with modulus sqrt(1 - eps^2).  delta, if not NULL,
 * receives the maximum relative error on that interval.  For f(A) = A^{-1/2}
 * pick eps^2 at or below the smallest |eigenvalue| of the scaled A (host arrays).
 * The elliptic functions of modulus sqrt(1 - eps^2) are evaluated through
 * Jacobi's imaginary transformation and theta series, accurate to rounding for
 * any eps; the result checks itself (positive residues, the error equal in size
 * with alternating signs at the 2 ns + 1 alternation points) and the call returns
 * FA_EINVAL, with fa_last_error saying so, if that check fails. */
int fa_zolotarev_poles(int ns, double eps, double* omega, double* sigma, double* delta);

/* out = D_w(mu) in (dagger = 0) or D_w(mu)^H in (dagger = 1), canonical
 * complex128 device spinors, computed in `precision` (FA_F64, FA_F32 or FA_DF;
 * FP32 and FA_DF round in and out through their packed layouts).  in != out. */
int fa_apply_dw(fa_ctx* ctx, const double* in, double* out, int dagger, int precision);

/* out = A in (dagger = 0) or A^H in = A(-mu) in (dagger = 1). */
int fa_apply_A(fa_ctx* ctx, const double* in, double* out, int dagger, int precision);

/* out = A in (dagger = 0) or A^H in (dagger = 1) in FP64, like fa_apply_A
 * with precision FA_F64, but without allocating any device memory: for
 * callers that cannot let the library call cudaMalloc, such as code recording
 * a CUDA graph under global stream-capture mode (where cudaMalloc is refused)
 * or code whose device memory is owned by a framework allocator or a fixed
 * budget.  The paper has no counterpart; this is a library convenience.
 * The working spinor lives in one static device array sized for at most
 * 8192 sites (1.5 MiB, resident on every GPU that loads the library until the
 * process exits); larger lattices return FA_EINVAL.  The first call on a
 * device looks up that array's device address (make it before any stream
 * capture); the context's device must be current.  All calls share the array,
 * so calls that overlap on one GPU race and must be serialised by the caller.
 * Stream-ordered on the context's stream; in and out are canonical device
 * spinors, in != out. */
int fa_apply_A_noalloc(fa_ctx* ctx, const double* in, double* out, int dagger);

/* Single-pass multi-shift solve (FP64): x_s = (A + sigma_s)^{-1} b for every
 * pole; x_s is an array of ns device spinors (canonical). */
int fa_solve_multishift(fa_ctx* ctx, const double* b, double* const* x_s,
                        const fa_solver_params* params, fa_solver_stats* stats);

/* y = sum_s omega_s (A + sigma_s)^{-1} b by the single-pass (params->mode =
 * FA_SINGLE, FP64) or the double-pass form (FA_DOUBLE; any precision).
 * b, y: device spinors (canonical).  Returns after the result is in y. */
int fa_apply_f(fa_ctx* ctx, const double* b, double* y,
               const fa_solver_params* params, fa_solver_stats* stats);

/* Batched f(A) b (the batched configuration of Sec. 3's setting: many sources
 * and lattices): system i is context ctxs[i] (its own gauge field, mu, mass,
 * scale and poles) with source b[i] and result y[i] (device spinors).  All
 * systems are solved together, whatever their lattice shapes: every kernel
 * launch of the solve serves all of them through work tables (one entry per
 * thread block: system, block within the system), each system with its own
 * scalars, shifts and convergence.  Contexts that share a packed gauge field
 * (fa_share_gauge: the sources of one lattice) form a group, at most 16
 * systems; the FP32 D_w sweep applies a group's operators tile by tile, the
 * right-hand sides of a tile one after the other in one thread block, so each
 * link is read from HBM once per tile for all of them.  The per-system
 * arithmetic and reduction order are those of a one-system solve with 128-
 * thread FP32 sweeps, so each y[i] equals fa_apply_f's for that system bit for
 * bit.  FA_MIXED / FA_MIXED_DF: the batch runs its head until every system
 * asks for the switch, then all switch at that outer iteration.  All contexts
 * must be on the same device; the work runs on ctxs[0]'s stream.  params is
 * shared (store_gb, if > 0, is the budget of the whole call, split so that
 * every system stores the same number of outer iterations; reliable_every
 * needs n = 1); stats, if not NULL, receives n entries.  Returns the first
 * non-OK status. */
int fa_apply_f_batched(fa_ctx* const* ctxs, int n, const double* const* b, double* const* y,
                       const fa_solver_params* params, fa_solver_stats* stats);

/* The k eigenpairs of H = gamma_5 D_w(mu) smallest in magnitude, with right
 * and left eigenvectors: the deflation subspace of the benchmarks of Sec. 3
 * (Figs. 3, 4), input of fa_apply_sign_deflated.  Krylov-Schur iteration
 * (restarted Arnoldi keeping a Schur basis of the wanted Ritz vectors) on
 * H^{-1} = c H A^{-1}, whose largest eigenvalues are the inverses of the
 * wanted ones; every application is one solve with A (the solver of
 * fa_apply_f, `params` for its form, precision and tolerance, with the single
 * pole omega = 1, sigma = 0; the context's own poles are kept) and one FP64
 * D_w sweep.  Left eigenvectors: the same iteration for H^H = H(-mu) (the
 * eigenvalues conj(lambda)), paired with the right ones and scaled so that
 * l_i^H r_j = delta_ij.
 *   k: wanted pairs (>= 1); m: Krylov dimension, k + 2 <= m <= 512 (2k + 8 is
 *      a reasonable choice); tol: convergence of a Ritz pair of H^{-1},
 *      |H^{-1} x - theta x| <= tol |theta| |x|; max_restarts: cap of restarts;
 *   seed: the counter-based start vector's seed (mu uses seed, -mu seed + 1);
 *   lambda: 2k host doubles (re, im); R, Lv: device arrays of k canonical
 *   spinors each (caller-owned, distinct), the right and left eigenvectors;
 *   *n_converged: pairs converged (both sides); *n_solves: solves used.
 * The context needs its gauge field and parameters (poles are not used).
 * Errors: FA_EINVAL for bad sizes; FA_ESTATE; FA_ENOCONV if fewer than k
 * pairs converge within max_restarts (the outputs then hold the current Ritz
 * pairs, or are incomplete if no left partner matched); FA_EBREAKDOWN when the
 * Krylov space is exhausted (k + 2 > the dimension of an invariant subspace
 * reached from the start vector); solver errors as for fa_apply_f. */
int fa_eigs_smallest(fa_ctx* ctx, int k, int m, double tol, int max_restarts, const fa_solver_params* params,
                     unsigned long long seed, double* lambda, double* R, double* Lv, int* n_converged,
                     int* n_solves);

/* Autotuner of the batched FP32 D_w sweep (the paper has no counterpart: a
 * choice of launch shape).  Times chains of the multi-RHS sweep over the
 * batch ctxs[0..n-1] (set up as for fa_apply_f_batched: gauge fields,
 * parameters, poles) for each number of right-hand sides per thread block in
 * {1, 2, 3, 4, 6, 12, 16} and each residency in {7, 4} blocks per SM, `reps`
 * launches between two CUDA events, the best of three rounds, and keeps the
 * fastest in ctxs[0], which fa_apply_f_batched uses when ctxs[0] leads a
 * batch.  Results do not depend on the choice.  The chosen values are written
 * to *rhs_per_block and *min_blocks; times_ms (may be NULL) receives up to
 * ntimes mean launch times in the order of the two lists (rhs outer).
 * Errors: FA_EINVAL for bad arguments, FA_ESTATE if a context lacks its gauge
 * field, parameters or poles. */
int fa_autotune_batched(fa_ctx* const* ctxs, int n, int reps, int* rhs_per_block, int* min_blocks,
                        double* times_ms, int ntimes);

/* sign(H) b with H = gamma_5 D_w(mu) (Sec. 1: sign z = z / sqrt(z^2), through
 * the partial-fraction expansion of Eq. 1).  With A = c H^2 (c = the context's
 * scale), sign(H) b = sqrt(c) H f(A) b: the solve of fa_apply_f with the same
 * params (any form and precision), then one FP64 D_w sweep.  The poles must
 * approximate z^{-1/2} (fa_neuberger_poles, or fa_zolotarev_poles with eps^2
 * below the spectrum of A); the accuracy is that of the pole expansion on the
 * spectrum of A.  b, out: device spinors (canonical),
 * b != out; stats as for fa_apply_f.  Returns after the result is in out. */
int fa_apply_sign(fa_ctx* ctx, const double* b, double* out,
                  const fa_solver_params* params, fa_solver_stats* stats);

/* The overlap operator at chemical potential mu (Sec. 1):
 * D_ov(mu) b = b + gamma_5 sign(gamma_5 D_w(mu)) b = b + sqrt(c) D_w(mu) f(A) b.
 * Arguments, poles and errors as for fa_apply_sign. */
int fa_apply_overlap(fa_ctx* ctx, const double* b, double* out,
                     const fa_solver_params* params, fa_solver_stats* stats);

/* sign(H) b (overlap = 0) or D_ov(mu) b (overlap != 0) with k eigenpairs of
 * H = gamma_5 D_w(mu) treated exactly, the deflation of the benchmarks of
 * Sec. 3 (Figs. 3, 4): with right eigenvectors r_i, left eigenvectors l_i
 * (l_i^H r_j = delta_ij) and eigenvalues lambda_i, a_i = l_i^H b and
 *   sign(H) b = sum_i sign(Re lambda_i) a_i r_i + sign(H) (b - sum_i a_i r_i),
 * the last term as in fa_apply_sign (poles chosen for the deflated spectrum).
 * R, Lv: k device spinors each, contiguous (k x 12 V complex128, canonical
 * order); lambda: 2 k host doubles (re, im).  k = 0 is fa_apply_sign /
 * fa_apply_overlap.  FA_EINVAL for k outside 0..1024, aliasing of out with
 * b, R or Lv, or an eigenvalue with zero real part.  The k inner products are
 * summed on the host in a fixed order. */
int fa_apply_sign_deflated(fa_ctx* ctx, const double* b, double* out, int k, const double* lambda,
                           const double* R, const double* Lv, int overlap,
                           const fa_solver_params* params, fa_solver_stats* stats);

/* The same as fa_apply_f with b and y in HOST memory: the host<->device
 * copies are part of the call. */
int fa_apply_f_host(fa_ctx* ctx, const double* b_host, double* y_host,
                    const fa_solver_params* params, fa_solver_stats* stats);

/* Adjoint gradient of L = Re <eta, y>, y = sum_s omega_s (A + sigma_s)^{-1} b
 * (Eq. 1; the paper computes no derivatives, this is its adjoint):
 *   dL = -Re sum_s omega_s <lambda_s, dA x_s>,  lambda_s = (A^H + sigma_s)^{-1} eta,
 *   A^H = A(-mu),  dA = c (g5 dD g5 D + g5 D g5 dD)  with the scale c held fixed.
 * Both multi-shift solves are single-pass FP64 (params->ell, tol, max_outer).
 * With params->shift_chunk = k (0 < k < N_s) the poles are taken k at a time:
 * per chunk the two solves run with that chunk's poles only and its link
 * forces are added, so the shift vectors held on the device are those of one
 * chunk (the seed recurrence is rerun per chunk; each x_s and lambda_s, and so
 * every output, is the same as with all poles at once).
 * Outputs: dLdU (device, canonical gauge layout) with dL = Re sum tr(dLdU^H dU)
 * over all links; *dLdmu and *L (host doubles); dLdb (device spinor, may be
 * NULL) = sum_s omega_s lambda_s, the gradient of L with respect to b.
 * b and eta: device spinors (canonical).  Returns after all outputs are written. */
int fa_grad(fa_ctx* ctx, const double* b, const double* eta, double* dLdU, double* dLdmu, double* L,
            double* dLdb, const fa_solver_params* params, fa_solver_stats* stats);

/* Wait for all work of the context; returns a deferred device error, if any. */
int fa_sync(fa_ctx* ctx);

/* Kernel launches issued by this context since creation (instrumentation). */
long long fa_launch_count(const fa_ctx* ctx);

/* Measured FP32 instruction issue rate of the current device (instrumentation,
 * no counterpart in the paper: the denominator of the double-float sweep's
 * roofline, which is bound by FP32 issue).  A probe kernel with eight
 * independent FP32 fused multiply-add chains per thread, 2048 threads per SM,
 * timed with CUDA events on a stream of its own after one warm-up launch; best
 * of `reps` launches (>= 1).  *thread_instr_per_s: FP32 instructions executed
 * per second, counted per thread (a warp instruction counts 32); *ms: the
 * launch's device time.  FA_EINVAL for a null output or reps < 1, FA_ECUDA. */
int fa_fp32_issue_rate(int reps, double* thread_instr_per_s, double* ms);

/* Device memory owned by the context (instrumentation for the memory claim of
 * Sec. 2: the double-pass forms keep no per-shift vectors).  field_bytes: the
 * lattice-sized buffers (links, seed and work spinors, y, the single-pass shift
 * vectors, pseudo-double-pass stores, staging, reduction partials); scalar_bytes:
 * solver state, shift scalars, scalar records and pass-2 weights.  Buffers grow
 * on demand and are kept for later calls.  FA_EINVAL for a null argument. */
int fa_device_bytes(const fa_ctx* ctx, unsigned long long* field_bytes, unsigned long long* scalar_bytes);

/* Mean device time (ms) of the hop kernels (one D_w sweep) issued by solves
 * with params->flags bit 1 set since the last reset, and how many were timed.
 * Reset with fa_hop_timing_reset(). */
int fa_hop_timing(const fa_ctx* ctx, int precision, double* mean_ms, long long* count);
/* The same, split by kernel (instrumentation, no counterpart in the paper):
 * with_dot = 0 for the plain sweeps, 1 for the sweeps
 * that also form <dot_with, out> (in a solve: the inner product after the second
 * hop of A and the scalar step in the last block), 2 for the FP32 sweep that
 * forms the MR Gram matrix in its epilogue (the last sweep of an outer
 * iteration; precision FA_F32 only), -1 for all (= fa_hop_timing).
 * FA_EINVAL for another with_dot or precision. */
int fa_hop_timing_split(const fa_ctx* ctx, int precision, int with_dot, double* mean_ms, long long* count);
int fa_hop_timing_reset(fa_ctx* ctx);

/* Kernel timeline tracing of the solver's kernels (the D_w sweeps of the
 * solves, the BiCG vector updates, the Gram and MR kernels, the pass-2 gathers
 * and the backward sweep), for every context on the current device.  While
 * tracing is on, thread 0 of every block of those kernels reads the GPU's global
 * nanosecond timer when the block enters the kernel and again when it leaves,
 * and appends one record to a ring of its SM (none for a block that finds its
 * system finished).  A launch spans from the earliest
 * entry to the latest exit of its blocks; the latest exit includes the scalar
 * step that the last block of a reduction runs.  No work is inserted between
 * launches, so replayed CUDA graphs are timed as they run.  Cost: one atomic
 * increment of a per-SM counter and one 32-byte store per block while on.
 *
 * kernel = FA_TK_* | (working precision << 8: 0 FP64, 1 FP32, 2 double-float)
 *          | (variant << 10: 1 for the sweep that also forms an inner product,
 *          and for the vector kernels' shift block launches). */
typedef struct {
    unsigned long long t_start_ns, t_end_ns;   /* %globaltimer at block entry / exit */
    int kernel;
    int block;                                 /* blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z) */
    int sm;
    int grid;                                  /* blocks of the launch */
} fa_trace_record;
enum {
    FA_TK_UPDATE_U = 1, FA_TK_UPDATE_R = 2, FA_TK_GRAM = 3, FA_TK_MR = 4, FA_TK_HOP_SYS = 5,
    FA_TK_HOP_MRHS = 6, FA_TK_HOP_SYS_ROWS = 7, FA_TK_HOP1_ROWS = 8, FA_TK_HOP1 = 9, FA_TK_HOP_GRAM = 10,
    FA_TK_RELIABLE = 11, FA_TK_GATHER = 12, FA_TK_SWEEP = 13, FA_TK_COEF_REDUCE = 14, FA_TK_ADVANCE = 15
};
/* Turn tracing on with room for `capacity` records on the current device
 * (split evenly over its SMs), cleared.  Starting again restarts.  Returns
 * FA_OK, FA_EINVAL (capacity < 1), FA_ENOMEM, FA_ECUDA.  Synchronises the device. */
int fa_trace_start(long long capacity);
/* Wait for the device, turn tracing off and copy up to `capacity` records to
 * host memory `records` (grouped by SM, each group in arrival order); *n gets
 * the number copied and *dropped the number lost (a full SM ring, or beyond
 * `capacity`).  Returns FA_OK, FA_EINVAL (null records, n or dropped, or
 * capacity < 0), FA_ESTATE (tracing not on), FA_ECUDA. */
int fa_trace_stop(fa_trace_record* records, long long capacity, long long* n, long long* dropped);

/* Launch shapes of the FP32 D_w sweep (the paper has no counterpart: a choice of
 * thread-block size and residency for the stencil kernel).
 *   FA_SHAPE_WIDE    256-thread blocks, 3 per SM (80 registers)
 *   FA_SHAPE_NARROW  128-thread blocks, 7 per SM (72 registers)
 *   FA_SHAPE_AUTO    narrow when the lattice fits one wave of it (the default)
 * One-system solves on lattices of up to three 128-site blocks per SM run the sweep
 * with two threads per site (256-thread blocks of 128 sites, 3 per SM) unless the
 * shape is WIDE; fa_apply_dw and fa_apply_A take the shapes as listed. */
typedef enum { FA_SHAPE_AUTO = 0, FA_SHAPE_WIDE = 1, FA_SHAPE_NARROW = 2 } fa_hop_shape;

/* Set / read the FP32 sweep launch shape of ctx; it applies to fa_apply_dw,
 * fa_apply_A and the single-system solves.  Results do not depend on the shape
 * (every site runs the same arithmetic).  Errors: FA_EINVAL for a null ctx or
 * an unknown shape (fa_get_hop_shape returns the shape or FA_EINVAL). */
int fa_set_hop_shape(fa_ctx* ctx, int shape);
int fa_get_hop_shape(const fa_ctx* ctx);

/* Autotuner: time every FP32 sweep launch shape on ctx's lattice, as a one-system
 * solve with that shape runs it (chains of `reps` sweeps, each reading the previous one's output, on scratch spinors
 * owned by ctx, between CUDA events on ctx's stream; replayed from a CUDA graph,
 * as the solver replays its outer iterations, unless ctx's stream is the legacy
 * or per-thread default stream, where they are launched directly; three
 * interleaved rounds, the best per shape), write the ms per launch of shape k to times_ms[k - 1]
 * (times_ms holds FA_SHAPE_NARROW doubles, host memory), and set the automatic
 * shape unless the other one is faster by more than 3 %.  Returns the chosen shape (> 0) or a
 * negative fa_status: FA_EINVAL (null ctx or times_ms, reps < 1), FA_ESTATE
 * (gauge field or parameters not set), FA_ECUDA.  Synchronises ctx's stream.
 * The Python binding caches the choice in a JSON file keyed by lattice and GPU. */
int fa_autotune(fa_ctx* ctx, int reps, double* times_ms);

const char* fa_status_string(int status);
const char* fa_last_error(void);
const char* fa_version(void);

#ifdef __cplusplus
}
#endif
#endif /* FAPATH_H */
