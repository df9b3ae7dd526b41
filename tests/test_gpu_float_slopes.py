"""Slopes of the float forms: a cell that is not finite is not limited away."""
import numpy as np
import pytest
import torch

import paper_1412_0934_gb300 as hy
import workloads
from hydro_testlib import ctx, dev, dts

pytestmark = pytest.mark.gpu

SHAPE = (14, 16, 18)
DX = 1.0 / 18


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("limiter", ["minmod", "mc"])
@pytest.mark.parametrize("axis", [1, 2, 3])
def test_a_nan_cell_reaches_both_sides(precision, limiter, axis):
    """A NaN density: its neighbours' fluxes use it, and so do their own slopes, on either side."""
    U = workloads.white_velocity_state(SHAPE, seed=7, p_jitter=0.2).numpy().copy()
    at = [0, 6, 7, 8]
    U[tuple(at)] = np.nan
    c = ctx(precision, limiter)
    a = dev(U, c.dtype)
    b = torch.empty_like(a)
    hy.hydro_step(c, hy.patch(a, 0, DX), hy.patch(b, 0, DX), dts(1e-3))
    assert hy.hydro_get_error(c)[1] & hy.EBIT_NONFINITE
    hy.hydro_finalize(c)
    for k in (-2, -1, 1, 2):
        p = list(at)
        p[axis] += k
        assert bool(torch.isnan(b[tuple(p)])), (axis, k)
