"""Blocks of the batched FP32 sweep that find all their systems finished leave no
trace record: the records of a batch are those of its outer iterations, without
the ones that were enqueued past convergence."""
import numpy as np
import pytest

import inputs
import paper_1010_2592_gb300 as fa
from fa_cases import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["double", "pseudo"])
def test_batched_sweep_records(mode):
    dims, ell = (4, 4, 4, 8), 2
    U = to_dev(inputs.su3_exp_gauge(dims, 0.5, 781))
    b = to_dev(inputs.gaussian_spinor(dims, 782))
    ctxs = []
    for k in range(3):
        ctx = fa.Context(dims)
        ctx.set_gauge(U) if k == 0 else ctx.share_gauge(ctxs[0])
        ctx.set_params(-1.8, 0.1, -1, 0.03)
        ctx.set_poles(*fa.neuberger_poles(4))
        ctxs.append(ctx)
    fa.trace_start(1 << 18)
    _, stats = fa.apply_f_batched(ctxs, [b, b, b], ell=ell, tol=1e-5, mode=mode, precision="f32", store_gb=1.0)
    rec, dropped = fa.trace_stop(1 << 18)
    m = stats[0]["outer_iters"]
    # the same source three times: all systems end at the same outer iteration; the host
    # enqueues eight at a time and looks at the flags a group later
    assert dropped == 0 and all(s["outer_iters"] == m for s in stats)
    sweeps = rec[(rec["kernel"] & 0xff) == 6]
    passes = 2 if mode == "double" else 1
    assert len(sweeps) == 4 * ell * m * passes * int(sweeps["grid"][0])
    assert np.all(sweeps["grid"] == sweeps["grid"][0])
