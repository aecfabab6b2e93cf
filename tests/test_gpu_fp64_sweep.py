"""The FP64 sweep at the edges of its tiles (32 sites) and of its split over
cluster blocks (four blocks per tile up to 38 tiles, two up to 76, one above),
in both layouts and both daggers, against the oracle."""
import numpy as np
import pytest

import inputs
from fa_cases import make_context, rel, to_dev, to_host
from oracle import dirac

pytestmark = pytest.mark.gpu


# 16 sites (half a tile), 32, 162 (ragged), 1216 = 38 tiles, 1225 (39, ragged), 2432 = 76 tiles, 2744 (86, ragged)
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 2, 4), (3, 3, 3, 6), (4, 4, 4, 19), (5, 5, 7, 7), (4, 4, 4, 38),
                                  (7, 7, 7, 8)])
def test_fp64_sweep_tiles(dims):
    U = inputs.su3_exp_gauge(dims, 0.5, 701)
    v = inputs.gaussian_spinor(dims, 702)
    ctx = make_context(dims, U, -1.8, 0.17, 0.03)
    # 1e-14: about 100 additions of rounding 1.1e-16 per component
    for dagger in (False, True):
        D = dirac.dw_dagger if dagger else dirac.dw
        A = dirac.apply_A_dagger if dagger else dirac.apply_A
        assert rel(to_host(ctx.apply_dw(to_dev(v), dagger=dagger)), D(U, v, -1.8, 0.17)) < 1e-14
        assert rel(to_host(ctx.apply_A(to_dev(v), dagger=dagger)), A(U, v, -1.8, 0.17, 0.03)) < 1e-14
