"""Sound speeds far from 1 in density and pressure.  Density and pressure may each be anywhere in the
range of the arithmetic; their product, which no formula of the scheme needs, may leave it."""
import numpy as np
import pytest
import torch

import paper_1412_0934_gb300 as hy
import workloads
from hydro_testlib import cfl, ctx, step_periodic

pytestmark = pytest.mark.gpu

N = 12
DX = 1.0 / N


def _gas(seed, mach):
    """Lognormal density and pressure around 1, white velocities; (5, N, N, N) conserved."""
    U = workloads.white_velocity_state(N, seed=seed, p_jitter=0.3).numpy().copy()
    kin = 0.5 * (U[1:4] ** 2).sum(0) / U[0]
    U[4] -= kin
    U[1:4] *= mach
    U[4] += mach * mach * kin
    return U


def _scaled(U, a, b):
    """Density times a, pressure times b (velocities times sqrt(b / a))."""
    return np.concatenate([a * U[:1], (np.sqrt(a) * np.sqrt(b)) * U[1:4], b * U[4:]])


@pytest.mark.parametrize("limiter", ["minmod", "mc", "ppm"])
@pytest.mark.parametrize("a,b,mach", [(2.0 ** -66, 2.0 ** -66, 0.0), (2.0 ** -66, 2.0 ** -62, 0.0),
                                      (2.0 ** 70, 2.0 ** 70, 0.0), (2.0 ** 66, 2.0 ** 62, 0.0),
                                      (2.0 ** 50, 2.0 ** 90, 1e-6)])
def test_double_float_at_far_scales(limiter, a, b, mach):
    """The step is covariant: the scaled state's step is the unit state's, scaled (dt by sqrt(a / b)).
    Every intermediate the double-float range names lies inside it, the momentum that the short step
    leaves too (its square 1e-14 of the pressure times the density); tolerance as for unit states."""
    U = _gas(3, mach)
    dt = 1e-7 * DX
    c = ctx("fp64", limiter=limiter, rho_floor=0.0, p_floor=0.0)
    want, dt_want = step_periodic(c, U, DX, dt, dt_next=True)
    hy.hydro_finalize(c)
    c = ctx("df64", limiter=limiter, rho_floor=0.0, p_floor=0.0)
    t = float(np.sqrt(a / b))
    got, dt_got = step_periodic(c, _scaled(U, a, b), DX, dt * t, dt_next=True)
    assert hy.hydro_get_error(c) == (hy.HYDRO_OK, 0)
    hy.hydro_finalize(c)
    got = _scaled(got, 1.0 / a, 1.0 / b)
    scale = np.abs(want).reshape(5, -1).max(1)
    scale[1:4] = np.sqrt(scale[0] * scale[4])  # a momentum of the gas: it may be at rest
    err = np.abs(got - want).reshape(5, -1).max(1) / scale
    assert err.max() <= 1e-12, err
    assert abs(dt_got / t - dt_want) <= 1e-12 * dt_want


@pytest.mark.parametrize("limiter", ["minmod", "ppm"])
@pytest.mark.parametrize("k", [-560, 540])
def test_double_at_far_scales(limiter, k):
    """Gas at rest, density and pressure times 2^k: every operation commutes with the scaling, so the
    results are the unit state's bits (the dt of the state at rest: the square of the momentum that the
    step leaves is out of range)."""
    U = _gas(4, 0.0)
    out = []
    for f in (1.0, 2.0 ** k):
        c = ctx("fp64", limiter=limiter, rho_floor=0.0, p_floor=0.0)
        g, _ = step_periodic(c, f * U, DX, 0.05 * DX)
        out.append((g / f, cfl(c, f * U, DX)))
        assert hy.hydro_get_error(c) == (hy.HYDRO_OK, 0)
        hy.hydro_finalize(c)
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]


def test_double_adjoint_at_far_scales():
    """With U' = S U, S diagonal, the reverse step of S^-1 lam is S^-1 times the unit state's: powers of
    two throughout, so the same bits."""
    U = _gas(5, 0.0)
    gen = torch.Generator().manual_seed(1)
    lam = torch.randn(U.shape, generator=gen, dtype=torch.float64).numpy()
    out = []
    for a, b in ((1.0, 1.0), (2.0 ** -400, 2.0 ** -640)):
        c = ctx("fp64", rho_floor=0.0, p_floor=0.0)
        dt = torch.full((1,), 0.05 * DX * float(np.sqrt(a / b)), dtype=torch.float64, device="cuda")
        Ud, Ld = (torch.as_tensor(x).cuda().contiguous() for x in (_scaled(U, a, b), _scaled(lam, 1 / a, 1 / b)))
        res = torch.empty_like(Ud)
        hy.hydro_adjoint_step(c, hy.patch(Ud, 0, DX), dt, hy.patch(Ld, 0, DX), hy.patch(res, 0, DX))
        assert hy.hydro_get_error(c) == (hy.HYDRO_OK, 0)
        hy.hydro_finalize(c)
        out.append(_scaled(res.cpu().numpy(), a, b))
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])
