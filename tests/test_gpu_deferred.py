"""Deferred updates of the double-pass forms: the sub-steps' site-local updates
made up by the MR step (FP32) or by a kernel of their own (double-float) give
the same vectors bit for bit, so a batch that defers them equals its systems
solved one at a time without; and every l and precision that defers meets the
oracle, with reliable updates (the seed solution moves with them) and with a
pass 2 from a partial store."""
import numpy as np
import pytest

import inputs
import paper_1010_2592_gb300 as fa
from fa_cases import make_context, oracle_double, rel, to_dev, to_host, workload_case

pytestmark = pytest.mark.gpu

C1 = "wilson_4x4x4x8"


@pytest.mark.parametrize("mode", ["double", "pseudo"])
def test_batch_beyond_l2_equals_one_at_a_time(mode):
    """l = 2, FP32: two 16^3 x 32 systems together are above the size from which the
    updates are deferred, one alone is below it."""
    dims = (16, 16, 16, 32)
    U = to_dev(inputs.su3_exp_gauge(dims, 0.4, 721))
    om, sg = fa.neuberger_poles(6)
    ctxs = []
    for k in range(2):
        ctx = fa.Context(dims)
        ctx.set_gauge(U) if k == 0 else ctx.share_gauge(ctxs[0])
        ctx.set_params(-1.8, 0.1, -1, 0.028)
        ctx.set_poles(om, sg)
        ctxs.append(ctx)
    srcs = [to_dev(inputs.gaussian_spinor(dims, 722 + k)) for k in range(2)]
    kw = dict(ell=2, tol=1e-4, mode=mode, precision="f32", store_gb=1.0)
    ys, _ = fa.apply_f_batched(ctxs, srcs, **kw)
    for ctx, b, y in zip(ctxs, srcs, ys):
        ctx.set_hop_shape("narrow")
        r = ctx.apply_f(b, gram_epilogue=False, **dict(kw, store_gb=0.5))
        assert np.array_equal(to_host(y), to_host(r.y))


@pytest.mark.parametrize("ell", [3, 4, 8])
@pytest.mark.parametrize("mode,store", [("double", 0.0), ("pseudo", 0.0), ("pseudo", 7.5)])
def test_double_float_head_defers(ell, mode, store):
    """store: outer iterations that the double-float store holds (0: all)."""
    w = workload_case(C1)
    y_o, _ = oracle_double(C1, None, ell, 1e-12)
    ctx = make_context(w["dims"], w["U"], w["mass"], w["mu"], w["c"], w["t_bc"], w["omega"], w["sigma"])
    V = int(np.prod(w["dims"]))
    per = (ell * (ell + 1) // 2 + ell) * 12 * V * 16 / 1e9
    # head to 1e-6 |b|: l = 8 loses too much in an FP32 tail from further up (power basis)
    kw = dict(ell=ell, tol=1e-10, mode=mode, precision="mixed_df", store_gb=2 * store * per, max_outer=400,
              switch_resid=1e-6)
    r = ctx.apply_f(to_dev(w["b"]), **kw)
    assert rel(to_host(r.y), y_o) < 1e-8
    r2 = ctx.apply_f(to_dev(w["b"]), reliable_every=4, **kw)
    assert rel(to_host(r2.y), y_o) < 1e-8


@pytest.mark.parametrize("ell", [1, 2, 3, 4])
@pytest.mark.parametrize("precision", ["mixed_df", "f32"])
@pytest.mark.parametrize("lt", [18, 20])
def test_mr_step_on_both_sides_of_its_grid_rule(lt, precision, ell):
    """288 and 320 blocks of the MR step, a little below and above two per SM of a
    152-SM part: components loaded in groups, and one at a time.  All fixed outer
    iterations, so that both precisions stop at the same polynomial degree and differ
    by rounding alone: 24 sub-steps at most, residuals of order 1, FP32 sums of 12 V
    terms in blocks of 256 and a growth of a few per sub-step stay below 1e-3."""
    dims = (16, 16, 16, lt)
    ctx = fa.Context(dims)
    ctx.set_gauge(to_dev(inputs.su3_exp_gauge(dims, 0.4, 731)))
    ctx.set_params(-1.8, 0.1, -1, 0.028)
    ctx.set_poles(*fa.neuberger_poles(6))
    b = to_dev(inputs.gaussian_spinor(dims, 732))
    kw = dict(ell=ell, tol=1e-30, mode="double", max_outer=3, fixed_iters=True)
    y = to_host(ctx.apply_f(b, precision=precision, **kw).y)
    y64 = to_host(ctx.apply_f(b, precision="f64", **kw).y)
    assert np.all(np.isfinite(y)) and rel(y, y64) < 1e-3
