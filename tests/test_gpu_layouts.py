"""FP32 and double-float operator calls through the packing kernel (64-site
tiles) and the sweeps that write the canonical layout: ragged tiles against the
oracle, point sources (zeros), and scaled inputs, whose results must be the
scaled results bit for bit as long as every number stays normal (the packing
converts on the integer pipes)."""
import numpy as np
import pytest

import inputs
from fa_cases import make_context, rel, to_dev, to_host
from oracle import dirac

pytestmark = pytest.mark.gpu

BOUND = {"f32": 5e-6, "df": 1e-11}      # the operator tests' bounds


# 16 sites, 64, 65 = 64 + 1, 162 (ragged), 1216
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 2, 4), (13, 5, 2, 2), (3, 3, 3, 6), (4, 4, 4, 19)])
@pytest.mark.parametrize("precision", ["f32", "df"])
def test_layouts(dims, precision):
    U = inputs.su3_exp_gauge(dims, 0.5, 711)
    ctx = make_context(dims, U, -1.8, 0.17, 0.03)
    for v in (inputs.gaussian_spinor(dims, 712), inputs.point_source(dims, 2, 1, (1, 0, 1, 1))):
        for dagger in (False, True):
            D = dirac.dw_dagger if dagger else dirac.dw
            got = to_host(ctx.apply_dw(to_dev(v), dagger=dagger, precision=precision))
            assert rel(got, D(U, v, -1.8, 0.17)) < BOUND[precision]
        got = to_host(ctx.apply_A(to_dev(v), precision=precision))
        assert rel(got, dirac.apply_A(U, v, -1.8, 0.17, 0.03)) < BOUND[precision]


@pytest.mark.parametrize("precision,powers", [("f32", (-80, -40, 40)), ("df", (-40, 40))])
def test_scaled_inputs_give_scaled_results(precision, powers):
    dims = (3, 3, 3, 6)
    U = inputs.su3_exp_gauge(dims, 0.5, 713)
    ctx = make_context(dims, U, -1.8, 0.0, 0.03)
    v = inputs.gaussian_spinor(dims, 714)
    want = to_host(ctx.apply_dw(to_dev(v), precision=precision))
    for p in powers:
        got = to_host(ctx.apply_dw(to_dev(v * 2.0 ** p), precision=precision))
        assert np.array_equal(got, want * 2.0 ** p), p


def test_numbers_outside_the_integer_range():
    """Denormal, huge, infinite and NaN inputs keep their FP32 meaning: site 0's
    output carries the diagonal term of its own input."""
    dims = (2, 2, 2, 2)
    ctx = make_context(dims, inputs.unit_gauge(dims), -1.8, 0.0, 1.0)
    for x in (2.0 ** -140, 3.0 ** -90, 2.0 ** 126 * 0.3, np.inf, np.nan):
        v = inputs.point_source(dims, 0, 0) * 0.0
        v[0, 0, 0, 0, 0, 0] = x
        got = to_host(ctx.apply_dw(to_dev(v), precision="f32"))[0, 0, 0, 0, 0, 0].real
        xf = np.float64(np.float32(x))
        if np.isfinite(x):
            assert abs(got - 2.2 * xf) <= 4e-7 * abs(xf) + 2.0 ** -149, x
        else:
            assert not np.isfinite(got), x
