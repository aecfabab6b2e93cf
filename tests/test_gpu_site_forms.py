"""FP64 kernels with a thread per site (lattices of many tiles) against the tile
kernels: equal bit for bit.  The forms are chosen by the sites of a launch, so a
batch takes the site kernels where each of its systems alone takes tiles."""
import numpy as np
import pytest

import inputs
import paper_1010_2592_gb300 as fa
from fa_cases import make_context, to_dev, to_host

pytestmark = pytest.mark.gpu


# on a 152-SM part: two systems of 74 blocks of 128 sites (148 of 152 SMs; ragged tile and
# block): the sweep; two of 13,520 (l <= 2) and of 26,364 sites: the Gram matrix and the MR step of
# a double pass, at 26,364 the updates with shifts; four of 37,349 (3.84 waves of 256 sites): the MR step with shifts
@pytest.mark.parametrize("dims,nsys", [((13, 13, 7, 8), 2), ((13, 13, 8, 10), 2), ((13, 13, 13, 12), 2), ((13, 17, 13, 13), 4)])
@pytest.mark.parametrize("mode,ell,ns", [("double", 1, 4), ("double", 2, 4), ("pseudo", 4, 4), ("double", 8, 2),
                                         ("single", 1, 16), ("single", 2, 3), ("single", 2, 17), ("single", 4, 2)])
def test_site_forms_equal_tile_forms(dims, nsys, mode, ell, ns):
    U = to_dev(inputs.unit_gauge(dims) * 1.0)
    U = U * to_dev(np.exp(1j * np.linspace(0.0, 3.0, 4))).reshape(1, 1, 1, 1, 4, 1, 1)   # a phase per direction
    ctxs, srcs = [], []
    for k in range(nsys):
        ctx = fa.Context(dims)
        ctx.set_gauge(U) if k == 0 else ctx.share_gauge(ctxs[0])
        ctx.set_params(-1.8, 0.1, -1, 0.028)
        ctx.set_poles(*fa.neuberger_poles(ns))
        ctxs.append(ctx)
        srcs.append(to_dev(inputs.gaussian_spinor(dims, 751 + k)))
    kw = dict(ell=ell, tol=1e-300, max_outer=3, fixed_iters=True, mode=mode, precision="f64")
    # the same number of stored outer iterations: a batch's budget is for all its systems
    ys, _ = fa.apply_f_batched(ctxs, srcs, store_gb=0.1 * nsys, **kw)
    for ctx, b, y in zip(ctxs, srcs, ys):
        y = to_host(y)
        assert np.all(np.isfinite(y)) and np.array_equal(to_host(ctx.apply_f(b, store_gb=0.1, **kw).y), y)


def test_scale_and_gradient_take_the_site_sweep():
    """19,456 sites: one block of 128 per SM.  The power iteration against the same
    steps through the operator call (tiles: it writes the caller's layout), to the
    rounding of the norms (1e-13); dL/dmu against the central difference of L at
    h = 1e-4 (truncation about h^2, cancellation 1e-12 / h: 1e-6)."""
    import torch
    dims = (16, 16, 4, 19)
    ctx = make_context(dims, inputs.su3_exp_gauge(dims, 0.4, 761), -1.8, 0.1, 1.0)
    v0 = to_dev(inputs.gaussian_spinor(dims, 762))
    v = v0 / torch.linalg.vector_norm(v0)
    for _ in range(3):
        v = ctx.apply_A(v)
        v = v / torch.linalg.vector_norm(v)
    c = 1.0 / float(torch.linalg.vector_norm(ctx.apply_A(v)))
    assert abs(ctx.estimate_scale(v0, 3) - c) < 1e-13 * c

    eta = to_dev(inputs.gaussian_spinor(dims, 763))
    ctx.set_poles(*fa.neuberger_poles(2))
    L = {}
    for h in (-1e-4, 0.0, 1e-4):
        ctx.set_params(-1.8, 0.1 + h, -1, 0.028)
        L[h] = ctx.grad(v0, eta)
    fd = (L[1e-4][0] - L[-1e-4][0]) / 2e-4
    assert abs(L[0.0][2] - fd) < 1e-6 * abs(fd) + 1e-6 * abs(L[0.0][0])
