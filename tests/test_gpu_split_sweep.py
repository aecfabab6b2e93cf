"""The FP32 sweep with two threads per site (one system on a small lattice)
against the one-thread sweep of a batch with the same 128-site partials: equal
bit for bit at the edges of its blocks and of the size up to which it is used,
with the Gram matrix in a kernel of its own and in the sweep's epilogue."""
import numpy as np
import pytest

import inputs
import paper_1010_2592_gb300 as fa
from fa_cases import oracle_double, rel, make_context, to_dev, to_host, workload_case

pytestmark = pytest.mark.gpu


# 16 sites, 128 (one block), 130 (two more), 12 x 16 x 16 x 19 = 456 blocks = 3 per SM, one time slice more
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 4, 2), (13, 5, 2, 2), (12, 16, 16, 19), (12, 16, 16, 20)])
@pytest.mark.parametrize("ell", [1, 2])
def test_split_sweep_equals_batched_sweep(dims, ell):
    # unit links and a Gaussian source: this test is about the sweep's bits, not its operator
    U = to_dev(inputs.unit_gauge(dims))
    ctxs = []
    for k in range(2):
        ctx = fa.Context(dims)
        ctx.set_gauge(U) if k == 0 else ctx.share_gauge(ctxs[0])
        ctx.set_params(-1.8, 0.1, -1, 0.028)
        ctx.set_poles(*fa.neuberger_poles(4))
        ctxs.append(ctx)
    srcs = [to_dev(inputs.gaussian_spinor(dims, 732 + k)) for k in range(2)]
    kw = dict(ell=ell, tol=1e-300, max_outer=4, fixed_iters=True, mode="double", precision="f32")
    ys, _ = fa.apply_f_batched(ctxs, srcs, **kw)
    for ctx, b, y in zip(ctxs, srcs, ys):
        ctx.set_hop_shape("narrow")
        assert np.array_equal(to_host(ctx.apply_f(b, gram_epilogue=False, **kw).y), to_host(y))


@pytest.mark.parametrize("ell", [1, 2, 3, 4])
def test_gram_epilogue_of_the_split_sweep(ell):
    """A ragged lattice (240 sites: two blocks, the second half full) against the oracle."""
    dims = (6, 4, 2, 5)
    w = workload_case("wilson_4x4x4x8", dims)
    y_o, _ = oracle_double("wilson_4x4x4x8", dims, ell, 1e-12)
    ctx = make_context(dims, w["U"], w["mass"], w["mu"], w["c"], w["t_bc"], w["omega"], w["sigma"])
    r = ctx.apply_f(to_dev(w["b"]), ell=ell, tol=1e-10, precision="f32", max_outer=400)
    # the FP32 solver tests' bounds
    assert rel(to_host(r.y), y_o) < (1e-6 if ell <= 3 else 1e-5)
