"""Operator calls whose input and output overlap in part (a shifted view of one
buffer) give what separate fields give: every precision works from a copy of
the input or has read it before it writes."""
import numpy as np
import pytest

import inputs
from fa_cases import make_context, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f64", "f32", "df"])
@pytest.mark.parametrize("shift", [1, 12, -5])
@pytest.mark.parametrize("dims", [(4, 4, 4, 8), (3, 3, 5, 7)])
def test_partly_overlapping_fields(dims, shift, precision):
    import torch
    v = to_dev(inputs.gaussian_spinor(dims, 791))
    n = v.numel()
    ctx = make_context(dims, inputs.su3_exp_gauge(dims, 0.5, 792), -1.8, 0.1, 0.03)
    for op in (ctx.apply_dw, ctx.apply_A):
        for dagger in (False, True):
            want = to_host(op(v, dagger=dagger, precision=precision))
            buf = torch.zeros(n + 32, dtype=torch.complex128, device="cuda")
            x, out = buf[16:16 + n].view(v.shape), buf[16 + shift:16 + shift + n].view(v.shape)
            x.copy_(v)
            op(x, dagger=dagger, precision=precision, out=out)
            assert np.array_equal(to_host(out), want)
