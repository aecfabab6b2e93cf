"""The single-pass MR step on small lattices splits the shifts over a cluster of
8, 4 or 2 blocks, of which one takes part in the convergence step: the flags
that the step clears are read by the others before it can run, so a shift that
freezes still gets its last update.  A batch gives all shifts of a tile to one
block, so both must agree bit for bit, however the blocks of a cluster fall
behind one another."""
import numpy as np
import pytest

import inputs
import paper_1010_2592_gb300 as fa
from fa_cases import to_dev, to_host

pytestmark = pytest.mark.gpu


# 512 sites (8 blocks on a 152-SM part), 1024 and 810 (4), 1050 and 2304 (2), 2312 (1)
@pytest.mark.parametrize("dims", [(4, 4, 4, 8), (4, 4, 8, 8), (3, 3, 9, 10), (5, 5, 6, 7), (4, 4, 12, 12), (17, 17, 2, 4)])
@pytest.mark.parametrize("ell,ns", [(1, 64), (2, 33), (4, 5)])
def test_clusters_equal_one_block(dims, ell, ns):
    U = to_dev(inputs.su3_exp_gauge(dims, 0.5, 741))
    om, sg = fa.neuberger_poles(ns)      # tan^2 from 1e-4 to 1e3: shifts freeze all through the solve
    ctxs = []
    for k in range(2):
        ctx = fa.Context(dims)
        ctx.set_gauge(U) if k == 0 else ctx.share_gauge(ctxs[0])
        ctx.set_params(-1.8, 0.1, -1, 0.03)
        ctx.set_poles(om, sg)
        ctxs.append(ctx)
    srcs = [to_dev(inputs.gaussian_spinor(dims, 742 + k)) for k in range(2)]
    kw = dict(ell=ell, tol=1e-9, mode="single", precision="f64", max_outer=400)
    ys, stats = fa.apply_f_batched(ctxs, srcs, **kw)
    for ctx, b, y, st in zip(ctxs, srcs, ys, stats):
        for _ in range(3):
            r = ctx.apply_f(b, **kw)
            assert np.array_equal(to_host(y), to_host(r.y))
            assert r.stats["iters_per_shift"] == st["iters_per_shift"]
            assert len(set(st["iters_per_shift"])) > 1
