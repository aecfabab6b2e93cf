"""Closer bounds for the double-float and grouped kernels than the solver tests
have: the head's vectors against FP64 at double-float accuracy, the MR step
with components loaded in groups against one at a time bit for bit, and
double-float conversion outside its integer range."""
import numpy as np
import pytest

import inputs
import paper_1010_2592_gb300 as fa
from fa_cases import make_context, rel, to_dev, to_host

pytestmark = pytest.mark.gpu


def solver_contexts(dims, n):
    U = to_dev(inputs.unit_gauge(dims))
    ctxs = []
    for k in range(n):
        ctx = fa.Context(dims)
        ctx.set_gauge(U) if k == 0 else ctx.share_gauge(ctxs[0])
        ctx.set_params(-1.8, 0.1, -1, 0.028)
        ctx.set_poles(*fa.neuberger_poles(6))
        ctxs.append(ctx)
    return ctxs


@pytest.mark.parametrize("ell", [1, 2, 3, 4])
@pytest.mark.parametrize("lt", [18, 20])
def test_double_float_head_at_its_accuracy(lt, ell):
    """Three outer iterations that never leave the head, on both sides of the MR step's
    grid rule: unit roundoff 2^-44 = 6e-14, at most 12 sub-steps, and a growth of
    the power basis of up to 1e4 between the largest summand and the result: 1e-9."""
    (ctx,) = solver_contexts((16, 16, 16, lt), 1)
    b = to_dev(inputs.gaussian_spinor((16, 16, 16, lt), 801))
    kw = dict(ell=ell, tol=1e-30, mode="double", max_outer=3, fixed_iters=True)
    y = to_host(ctx.apply_f(b, precision="mixed_df", switch_resid=1e-30, **kw).y)
    assert rel(y, to_host(ctx.apply_f(b, precision="f64", **kw).y)) < 1e-9


@pytest.mark.parametrize("ell", [1, 2, 3, 4])
@pytest.mark.parametrize("precision", ["mixed_df", "f32"])
def test_grouped_mr_loads_give_the_same_bits(precision, ell):
    """160 blocks of the MR step alone (groups: at most two per SM of a 152-SM part), 320 in
    a batch of two (one component at a time)."""
    dims = (16, 16, 16, 10)
    ctxs = solver_contexts(dims, 2)
    srcs = [to_dev(inputs.gaussian_spinor(dims, 802 + k)) for k in range(2)]
    kw = dict(ell=ell, tol=1e-300, mode="double", precision=precision, max_outer=3, fixed_iters=True)
    if precision == "mixed_df":
        kw["switch_resid"] = 1e-30
    ys, _ = fa.apply_f_batched(ctxs, srcs, **kw)
    for ctx, b, y in zip(ctxs, srcs, ys):
        ctx.set_hop_shape("narrow")
        assert np.array_equal(to_host(ctx.apply_f(b, gram_epilogue=False, **kw).y), to_host(y))


def test_double_float_conversion_outside_its_range():
    """Below 2^-74, near the largest FP32 number, infinite and NaN inputs keep their FP32
    meaning at least (site 0's output carries the diagonal term of its own input)."""
    dims = (2, 2, 2, 2)
    ctx = make_context(dims, inputs.unit_gauge(dims), -1.8, 0.0, 1.0)
    for x in (2.0 ** -140, 3.0 * 2.0 ** -90, 2.0 ** 126 * 0.3, np.inf, -np.inf, np.nan):
        v = inputs.point_source(dims, 0, 0) * 0.0
        v[0, 0, 0, 0, 0, 0] = x
        got = to_host(ctx.apply_dw(to_dev(v), precision="df"))[0, 0, 0, 0, 0, 0].real
        if np.isfinite(x):
            assert abs(got - 2.2 * x) <= 4e-7 * abs(x) + 2.0 ** -148, x
        else:
            assert not np.isfinite(got), x
