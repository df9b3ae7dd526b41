"""Slopes of the float forms: the forward step and its reverse select the same one, also where the product
of the two differences underflows, and a cell that is not finite is not limited away."""
import numpy as np
import pytest
import torch

import paper_1412_0934_gb300 as hy
import workloads
from hydro_testlib import ctx, dev, dts, normwise

pytestmark = pytest.mark.gpu

SHAPE = (14, 16, 18)
DX = 1.0 / 18


def _slow_gas(scale):
    """Gas of random density and pressure whose velocities are `scale` of the sound speed."""
    U = workloads.white_velocity_state(SHAPE, seed=6, p_jitter=0.2).numpy().copy()
    U[4] -= 0.5 * (U[1:4] ** 2).sum(0) / U[0]
    U[1:4] *= scale
    return U.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("limiter", ["minmod", "mc"])
@pytest.mark.parametrize("scale", [1e-24, 1e-12])
def test_reverse_step_selects_the_step_s_slopes(limiter, scale):
    """Velocity differences of 1e-24: the float gradient against the double one (whose sign tests never
    underflow), to the accuracy of the float gradient at ordinary speeds."""
    U = _slow_gas(scale)
    lam = np.random.default_rng(3).standard_normal(U.shape).astype(np.float32).astype(np.float64)
    got = {}
    for precision in ("fp32", "fp64"):
        c = ctx(precision, limiter)
        a, l = dev(U, c.dtype), dev(lam, c.dtype)
        out = torch.empty_like(a)
        hy.hydro_adjoint_step(c, hy.patch(a, 0, DX), dts(2e-3), hy.patch(l, 0, DX), hy.patch(out, 0, DX))
        assert hy.hydro_get_error(c) == (hy.HYDRO_OK, 0)
        got[precision] = out.double().cpu().numpy()
        hy.hydro_finalize(c)
    assert normwise(got["fp32"], got["fp64"]).max() <= 1e-4


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
