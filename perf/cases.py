"""The work that users of this library have it do, as timed cases: operator
applications, the set-up of a new gauge field, multi-shift solves, f(A) b in
its forms and precisions, batches of sources, the overlap operator and the
adjoint gradient, all through the Python binding's public calls.

Gauge fields and sources follow the recipe of `inputs` (U = exp(i eps H) with
H Gaussian, traceless and Hermitian; complex Gaussian or point sources), made
on the GPU from the seed.  Mass -1.8, antiperiodic time boundary, lattice
shapes and solver settings as in this repository's workloads and tests.
"""
import math

import numpy as np
import torch

import paper_1010_2592_gb300 as fa

MASS, T_BC = -1.8, -1
C128 = torch.complex128


# ------------------------------------------------------------------ the cases
def _case(name, kind, dims, **kw):
    X, Y, Z, T = dims
    c = dict(name=name, kind=kind, X=X, Y=Y, Z=Z, T=T, mu=0.05, eps=0.4, op="A", dagger=False, precision="f64",
             mode="double", ell=2, ns=16, tol=1e-10, graph=False, theta=0.0, store_gb=0.0, nrhs=1)
    c.update(kw)
    return c


def listed():
    return [
        # one FP64 application of A on the paper's 4^3 x 8 lattice: the smallest call, what a
        # user's own Krylov method does in its inner loop
        _case("A_f64_4x4x4x8", "operator", (4, 4, 4, 8), eps=0.5),
        # D_w^H in double-float on the lattice of the paper's Fig. 4
        _case("dw_df_12x12x12x24", "operator", (12, 12, 12, 24), op="dw", dagger=True, precision="df", mu=0.1),
        # one FP32 sweep on the largest lattice of the workloads
        _case("dw_f32_32x32x32x64", "operator", (32, 32, 32, 64), op="dw", precision="f32", eps=0.35),
        # a new configuration of an ensemble: load the links, estimate the scale c with
        # the recipe's 100 power iterations, apply the scaled operator once
        _case("setup_16x16x16x32", "setup", (16, 16, 16, 32), mu=0.1),
        # every shifted solution on the paper's lattice, single pass
        _case("multishift_f64_4x4x4x8", "multishift", (4, 4, 4, 8), mode="single", eps=0.5, ns=10, tol=1e-12),
        # f(A) b in the form that apply_f defaults to (double pass, FP64, direct launches), at the
        # tolerance of a reference solve
        _case("f_f64_8x8x8x16", "f", (8, 8, 8, 16), eps=0.5, ns=12, tol=1e-12),
        # the benchmark's workload: pseudo-double-pass, double-float head, FP32 tail, graph replay
        _case("f_mixed_df_16x16x16x32", "f", (16, 16, 16, 32), mu=0.1, mode="pseudo", precision="mixed_df", ns=20,
              tol=1e-9, graph=True, theta=0.02, store_gb=16.0),
        # the largest workload, in the form that stores nothing (option 1 of Sec. 2)
        _case("f_mixed_df_32x32x32x64", "f", (32, 32, 32, 64), eps=0.35, precision="mixed_df", ell=4, ns=32,
              tol=3e-9, graph=True, theta=0.0025),
        # the overlap operator on the lattice of Fig. 4 with its 16 poles
        _case("overlap_12x12x12x24", "overlap", (12, 12, 12, 24), mode="pseudo", precision="mixed_df", tol=1e-9,
              graph=True, store_gb=8.0),
        # propagators: 12 spin-colour point sources on each of two lattices, FP32 bulk
        _case("batch_f32_12x2", "batch", (12, 12, 12, 24), mode="pseudo", precision="f32", graph=True, store_gb=16.0,
              nrhs=12, mu=0.1),
        # the adjoint gradient with respect to links, mu and source
        _case("grad_8x8x8x16", "grad", (8, 8, 8, 16), mode="single", eps=0.5, ns=12, tol=1e-12),
        # host buffers in and out on a ragged lattice, FP64 head and FP32 tail, l = 3
        _case("host_mixed_6x4x6x10", "host", (6, 4, 6, 10), precision="mixed", ell=3, ns=10, tol=1e-9, eps=0.5),
    ]


# most sites of a drawn lattice, per kind (FP64 solves cost the most per site)
_MOST = dict(operator=1 << 21, setup=1 << 17, multishift=1 << 13, f=1 << 17, overlap=1 << 17, batch=41472, grad=1 << 13,
             host=1 << 15)


def _draw_dims(rng, most):
    """Extents of a lattice of 108 to `most` sites, the volume spread over its
    logarithm, time about twice the spatial extents, odd ones among them."""
    while True:
        v = math.exp(rng.uniform(math.log(108.0), math.log(float(most))))
        s = (v / 2.0) ** 0.25
        d = [max(2, round(s * math.exp(rng.uniform(-0.3, 0.3)))) for _ in range(3)]
        d.append(max(2, round(v / (d[0] * d[1] * d[2]))))
        if 64 <= d[0] * d[1] * d[2] * d[3] <= most:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["operator", "operator", "f", "f", "f", "host", "overlap", "batch", "multishift", "grad", "setup"])
    dims = _draw_dims(rng, _MOST[kind])
    V = dims[0] * dims[1] * dims[2] * dims[3]
    c = _case("", kind, dims, mu=round(rng.uniform(0.0, 0.2), 4), eps=rng.choice([0.35, 0.4, 0.5]),
              ns=rng.randint(4, 24))
    del c["name"]
    if kind == "operator":
        c.update(op=rng.choice(["A", "dw"]), dagger=rng.random() < 0.3, precision=rng.choice(["f64", "f32", "df"]))
    elif kind in ("f", "host", "overlap"):
        c.update(precision=rng.choice(["f64", "f32", "mixed", "mixed_df", "mixed_df"]), mode=rng.choice(["double", "pseudo"]),
                 ell=rng.choice([1, 2, 2, 4]), graph=kind != "host" and rng.random() < 0.6, store_gb=16.0)
        c["tol"] = 1e-12 if c["precision"] == "f64" else 1e-9
    elif kind == "batch":
        c.update(mode="pseudo", precision=rng.choice(["f32", "mixed_df"]), graph=True, store_gb=16.0,
                 nrhs=rng.randint(2, 12), tol=1e-9)
    elif kind in ("multishift", "grad"):
        c.update(mode="single", ns=rng.randint(4, 12), tol=1e-12)
    return c


def _dims(case):
    return case["X"], case["Y"], case["Z"], case["T"]


def _lattices(case):
    """Lattices of the case: a batch has a second one of two thirds the extents."""
    d = _dims(case)
    return [d, tuple(max(2, 2 * x // 3) for x in d)] if case["kind"] == "batch" else [d]


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _gauss(g, shape):
    """Entries (N(0,1) + i N(0,1)) / sqrt(2)."""
    x = torch.randn(tuple(shape) + (2,), generator=g, dtype=torch.float64, device="cuda")
    return torch.view_as_complex(x) * math.sqrt(0.5)


def _mm(a, b):
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _gauge(g, dims, eps):
    X, Y, Z, T = dims
    U = torch.empty((T, Z, Y, X, 4, 3, 3), dtype=C128, device="cuda")
    eye = torch.eye(3, dtype=C128, device="cuda")
    for mu in range(4):
        H = _gauss(g, (T, Z, Y, X, 3, 3))
        H = 0.5 * (H + H.mH)
        H = H - (H.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3.0)[..., None, None] * eye
        # exp by its series at a quarter of the argument, squared twice
        H = (0.25j * eps) * H
        E = eye + H / 16.0
        for n in range(15, 0, -1):
            E = eye + _mm(H, E) / n
        E = _mm(E, E)
        U[..., mu, :, :] = _mm(E, E)
    return U


def _spinor_shape(dims):
    X, Y, Z, T = dims
    return (T, Z, Y, X, 4, 3)


def _sources(case, g, dims):
    if case["kind"] != "batch":
        return [_gauss(g, _spinor_shape(dims))]
    out = []
    for k in range(case["nrhs"]):     # point sources at the origin, spin k // 3, colour k % 3
        b = torch.zeros(_spinor_shape(dims), dtype=C128, device="cuda")
        b[0, 0, 0, 0, (k // 3) % 4, k % 3] = 1.0
        out.append(b)
    return out


def _inputs(case, seed):
    """Per lattice: links, sources, the scale's start vector; and eta of a gradient."""
    g = _gen(seed)
    lat = []
    for dims in _lattices(case):
        U = _gauge(g, dims, case["eps"])
        lat.append((dims, U, _sources(case, g, dims), _gauss(g, _spinor_shape(dims))))
    eta = _gauss(g, _spinor_shape(_dims(case))) if case["kind"] == "grad" else None
    return lat, eta


# scale of A in a case: 1 / the largest eigenvalue of (g5 D)^2 on such fields, as the power
# iteration estimates it, rounded (a figure that a user keeps with the ensemble)
def _scale(case):
    return {0.35: 0.028, 0.4: 0.0285, 0.5: 0.03}[case["eps"]]


def _solver_kw(case):
    kw = dict(ell=case["ell"], tol=case["tol"], mode=case["mode"], precision=case["precision"])
    if case["graph"]:
        kw["graph"] = True
    if case["theta"] > 0.0:
        kw["switch_resid"] = case["theta"]
    if case["mode"] == "pseudo":
        kw["store_gb"] = case["store_gb"]
    return kw


def prepare(case, seed):
    lat, eta = _inputs(case, seed)
    s = dict(case=case, ctxs=[], srcs=[], eta=eta)
    # a stream of its own where outer iterations are replayed from graphs, else the current one
    s["stream"] = torch.cuda.Stream() if case["graph"] else None
    torch.cuda.synchronize()                  # the inputs, made on the current stream
    for dims, U, srcs, v0 in lat:
        owner = None
        for b in srcs:
            ctx = fa.Context(dims, s["stream"])
            if owner is None:
                owner = ctx
                ctx.set_gauge(U)
            else:
                ctx.share_gauge(owner)
            ctx.set_params(MASS, case["mu"], T_BC, _scale(case))
            ctx.set_poles(*fa.neuberger_poles(case["ns"]))
            s["ctxs"].append(ctx)
            s["srcs"].append(b)
        if case["kind"] == "setup":
            s["U"], s["v0"] = U, v0
    if case["kind"] == "host":
        s["srcs"] = [b.cpu().numpy() for b in s["srcs"]]
    torch.cuda.synchronize()
    return s


def run(s):
    case, ctx, b = s["case"], s["ctxs"][0], s["srcs"][0]
    kind = case["kind"]
    if kind == "operator":
        f = ctx.apply_A if case["op"] == "A" else ctx.apply_dw
        return f(b, dagger=case["dagger"], precision=case["precision"])
    if kind == "setup":
        ctx.set_gauge(s["U"])
        ctx.set_params(MASS, case["mu"], T_BC, 1.0)
        c = ctx.estimate_scale(s["v0"], 100)
        ctx.set_params(MASS, case["mu"], T_BC, c)
        return c, ctx.apply_A(b)
    if kind == "multishift":
        return ctx.solve_multishift(b, ell=case["ell"], tol=case["tol"]).y
    if kind == "f":
        return ctx.apply_f(b, **_solver_kw(case)).y
    if kind == "host":
        return ctx.apply_f_host(b, **_solver_kw(case)).y
    if kind == "overlap":
        return ctx.apply_overlap(b, **_solver_kw(case)).y
    if kind == "batch":
        return fa.apply_f_batched(s["ctxs"], s["srcs"], **_solver_kw(case))[0]
    L, dU, dmu, db, _ = ctx.grad(b, s["eta"], ell=case["ell"], tol=case["tol"])
    return L, dU, dmu, db


# ------------------------------------------------------------------ work
# bytes of one real number of a spinor in the precision of the bulk, and of a link
_REAL = dict(f64=8, df=8, f32=4, mixed=4, mixed_df=4)
_LINK = dict(f64=144, df=144, f32=48, mixed=48, mixed_df=48)


def work(case):
    """Bytes: the caller's fields read and written once, and for an iterative
    method, per application of A (two sweeps), the links, one vector in and one
    out of each sweep in the precision of the bulk, plus the recurrence's own
    vectors once.  Flops: 1464 per site and sweep (8 x 183: projection, colour
    product, sum; 1464 with the diagonal term)."""
    V = sum(d[0] * d[1] * d[2] * d[3] * (case["nrhs"] if case["kind"] == "batch" else 1) for d in _lattices(case))
    p = case["precision"]
    sweep = 2 * 24 * _REAL[p] + 4 * _LINK[p]
    kind = case["kind"]
    if kind == "operator":
        n = 2 if case["op"] == "A" else 1
        return {"bytes": V * (2 * 192 + 4 * _LINK[p]), "flops": n * 1464.0 * V}
    if kind == "setup":
        return {"bytes": V * (576.0 * 2 + 202 * sweep), "flops": 202 * 1464.0 * V}
    decades = -math.log10(case["tol"])
    mv = 20.0 * decades                       # applications of A: about 20 per decade on these fields
    if case["mode"] == "double":
        mv *= 2                               # pass 2 regenerates the vectors
    if kind == "grad":
        mv *= 2                               # forward and adjoint systems
    vec = 24 * _REAL[p]
    per_mv = 2 * sweep + 6 * vec
    if case["mode"] == "single":
        per_mv += 3 * case["ns"] * vec        # the shift vectors
    return {"bytes": V * (2 * 192 + mv * per_mv), "flops": V * mv * (2 * 1464.0 + 300.0)}


# ------------------------------------------------------------------ 64-bit values, plain torch
# gamma_mu psi = phase[s] psi[perm[s]] (DeGrand-Rossi basis)
_GAMMA = [((3, 2, 1, 0), (1j, 1j, -1j, -1j)), ((3, 2, 1, 0), (-1, 1, 1, -1)),
          ((2, 3, 0, 1), (1j, -1j, -1j, 1j)), ((2, 3, 0, 1), (1, 1, 1, 1))]


def _gam(mu, psi):
    perm, ph = _GAMMA[mu]
    return torch.tensor(ph, dtype=C128, device=psi.device)[:, None] * psi[..., list(perm), :]


def _dw(U, psi, mu_chem):
    out = (4.0 + MASS) * psi
    T = psi.shape[0]
    e = mu_chem if isinstance(mu_chem, torch.Tensor) else torch.tensor(mu_chem, dtype=torch.float64, device=psi.device)
    at = torch.arange(T, device=psi.device)
    wf = torch.where(at == T - 1, float(T_BC), 1.0).to(torch.float64) * torch.exp(e)
    wb = torch.where(at == 0, float(T_BC), 1.0).to(torch.float64) * torch.exp(-e)
    for mu, ax in enumerate((3, 2, 1, 0)):
        Um = U[..., mu, :, :]
        f = torch.roll(psi, -1, ax)
        f = f - _gam(mu, f)
        f = sum(Um[..., None, :, k] * f[..., :, k, None] for k in range(3))
        w = psi + _gam(mu, psi)
        w = sum(Um[..., None, k, :].conj() * w[..., :, k, None] for k in range(3))
        w = torch.roll(w, 1, ax)
        if mu == 3:
            f = f * wf[:, None, None, None, None, None]
            w = w * wb[:, None, None, None, None, None]
        out = out - 0.5 * (f + w)
    return out


def _g5(psi):
    return psi * torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device=psi.device)[:, None]


def _A(U, psi, mu, c):
    return c * _g5(_dw(U, _g5(_dw(U, psi, mu)), mu))


def _poles(ns):
    th = [math.pi * (s - 0.5) / (2.0 * ns) for s in range(1, ns + 1)]
    return [1.0 / ns / math.cos(t) ** 2 for t in th], [math.tan(t) ** 2 for t in th]


def _shifted(U, b, mu, c, sigma, weights=None, most=480):
    """(A + sigma_s)^{-1} b for every shift (weights: their weighted sum instead)
    by full orthogonalisation in the Krylov space, to rounding."""
    n = b.numel()
    nb = float(torch.linalg.vector_norm(b))
    Q = torch.empty((most + 1, n), dtype=C128, device=b.device)
    Q[0] = (b / nb).reshape(-1)
    H = np.zeros((most + 1, most), dtype=np.complex128)
    m, old = 0, None
    while m < most:
        w = _A(U, Q[m].view(b.shape), mu, c).reshape(-1)
        for _ in range(2):
            h = Q[:m + 1].conj() @ w
            w = w - h @ Q[:m + 1]
            H[:m + 1, m] += h.cpu().numpy()
        beta = float(torch.linalg.vector_norm(w))
        H[m + 1, m] = beta
        m += 1
        full = beta < 1e-13 or m == min(n, most)
        if m % 20 == 0 or full:
            e1 = np.zeros(m, dtype=np.complex128)
            e1[0] = nb
            z = np.stack([np.linalg.solve(H[:m, :m] + s * np.eye(m), e1) for s in sigma])
            if weights is not None:
                z = (np.asarray(weights)[:, None] * z).sum(0, keepdims=True)
            if old is not None:
                d = z.copy()
                d[:, :old.shape[1]] -= old
                if (np.linalg.norm(d, axis=1) <= 1e-14 * np.linalg.norm(z, axis=1)).all():
                    break
            old = z
        if full:
            break
        Q[m] = w / beta
    out = [(torch.from_numpy(v).to(b.device) @ Q[:m]).view(b.shape) for v in z]
    return out[0] if weights is not None else out


def exact(case, seed):
    kind, mu, c = case["kind"], case["mu"], _scale(case)
    V = math.prod(_dims(case))
    if kind != "operator" and V > 140000:
        return None                           # minutes
    lat, eta = _inputs(case, seed)
    _, U, srcs, v0 = lat[0]
    b = srcs[0]
    om, sg = _poles(case["ns"])
    if kind == "operator":
        # D^H(mu) = g5 D(-mu) g5, A^H(mu) = A(-mu)
        m = -mu if case["dagger"] else mu
        if case["op"] == "A":
            return _A(U, b, m, c)
        return _g5(_dw(U, _g5(b), m)) if case["dagger"] else _dw(U, b, m)
    if kind == "setup":
        v = v0 / torch.linalg.vector_norm(v0)
        for _ in range(100):
            v = _A(U, v, mu, 1.0)
            v = v / torch.linalg.vector_norm(v)
        c = 1.0 / float(torch.linalg.vector_norm(_A(U, v, mu, 1.0)))
        return c, _A(U, b, mu, c)
    if kind == "multishift":
        return _shifted(U, b, mu, c, sg)
    if kind in ("f", "host"):
        y = _shifted(U, b, mu, c, sg, om)
        return y.cpu().numpy() if kind == "host" else y
    if kind == "overlap":
        return b + math.sqrt(c) * _dw(U, _shifted(U, b, mu, c, sg, om), mu)
    if kind == "batch":
        return [_shifted(u, x, mu, c, sg, om) for _, u, xs, _ in lat for x in xs]
    # gradient of Re <eta, y>: dL = -Re sum_s omega_s <lambda_s, dA x_s>, A^H = A(-mu)
    xs = _shifted(U, b, mu, c, sg)
    ls = _shifted(U, eta, -mu, c, sg)
    L = float(torch.vdot(eta.reshape(-1), sum(w * x for w, x in zip(om, xs)).reshape(-1)).real)
    Ug = U.clone().requires_grad_(True)
    mg = torch.tensor(mu, dtype=torch.float64, device="cuda", requires_grad=True)
    for w, x, l in zip(om, xs, ls):
        (-w * torch.vdot(l.reshape(-1), _A(Ug, x, mg, c).reshape(-1)).real).backward()
    return L, Ug.grad, float(mg.grad), sum(w * l for w, l in zip(om, ls))
