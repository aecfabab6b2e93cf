"""The autotuner times the FP32 sweep that a solve runs: on small lattices the one
with two threads per site (a traced kernel; the operator calls' sweep is not), on
larger ones the listed shapes.  Cache entries from before that are timed again."""
import types

import numpy as np
import pytest

import paper_1010_2592_gb300 as fa


def test_entries_of_other_sweeps_are_timed_again(tmp_path):
    cache = str(tmp_path / "tune.json")
    ctx = object.__new__(fa.Context)
    ctx.dims, ctx.h, set_to = (8, 8, 8, 16), None, []
    ctx.set_hop_shape = set_to.append
    ctx.lib = types.SimpleNamespace(fa_autotune=lambda h, reps, times: fa.SHAPE_NARROW)
    key = fa.tune_key(ctx.dims, fa._device_name())
    fa.store_tune_cache(cache, key, {"shape": fa.SHAPE_WIDE, "times_ms": [0.02, 0.021]})
    r = ctx.autotune(cache=cache)
    assert not r["cached"] and r["shape"] == fa.SHAPE_NARROW and set_to == []
    r = ctx.autotune(cache=cache)
    assert r["cached"] and r["shape"] == fa.SHAPE_NARROW and set_to == [fa.SHAPE_NARROW]


@pytest.mark.gpu
@pytest.mark.parametrize("dims,split", [((8, 8, 8, 16), True), ((12, 16, 16, 19), True), ((12, 16, 16, 20), False)])
def test_autotune_times_the_solver_sweep(dims, split):
    """456 blocks of 128 sites are three per SM of a 152-SM part; one time slice more is not."""
    import torch
    import inputs
    from fa_cases import make_context, to_dev, to_host
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes are for 152 SMs")
    ctx = make_context(dims, inputs.unit_gauge(dims), -1.8, 0.1, 0.028)
    ctx.set_poles(*fa.neuberger_poles(4))
    b = to_dev(inputs.gaussian_spinor(dims, 771))
    kw = dict(ell=2, tol=1e-300, max_outer=3, fixed_iters=True, mode="double", precision="f32")
    want = to_host(ctx.apply_f(b, **kw).y)
    fa.trace_start(1 << 18)
    r = ctx.autotune(reps=2)
    rec, dropped = fa.trace_stop(1 << 18)
    names = {fa.trace_kernel_name(int(k)) for k in rec["kernel"]}
    assert dropped == 0 and names == ({"k_hop1<f32>"} if split else set())
    assert all(t > 0 for t in r["times_ms"])
    assert np.array_equal(to_host(ctx.apply_f(b, **kw).y), want)
