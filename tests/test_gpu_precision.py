"""Rounding errors of double and double-float arithmetic, measured over many cells: no larger than those of
plain formulas in correctly rounded double operations and in normalising double-float operators.  The bounds
are those formulas' errors on the same inputs, measured once (the time step's and double-float's with 1%
added: rounding takes another course at each change)."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle
import paper_1412_0934_gb300 as hy
from hydro_testlib import GAMMA, ctx

pytestmark = pytest.mark.gpu

LD = np.longdouble
PATCHES, EDGE, DX = 3000, 6, 1.0 / 32


def _white(rng, shape, mach):
    rho, p = np.exp(0.5 * rng.normal(size=shape) - 0.125), np.exp(0.3 * rng.normal(size=shape))
    return _conserved(rho, mach * math.sqrt(GAMMA) * rng.normal(size=(3,) + shape), p)


def _conserved(rho, v, p):
    return np.stack([rho, *(rho * v), p / (GAMMA - 1) + 0.5 * rho * (v ** 2).sum(0)])


def _patches(kind, mach):
    """Ghosted 6^3 patches (5, PATCHES, 10, 10, 10): white noise, or cold gas in a linear flow."""
    rng = np.random.default_rng(3)
    shape = (PATCHES,) + (EDGE + 4,) * 3
    if kind == "white":
        return _white(rng, shape, mach)
    rho = np.exp(0.5 * rng.normal(size=shape) - 0.125)
    one, z = (3, PATCHES, 1, 1, 1), np.arange(EDGE + 4) / (EDGE + 4)
    v = rng.normal(size=one) + 0.02 * rng.normal(size=(3,) + shape)
    for axis in (z[:, None, None], z[None, :, None], z[None, None, :]):
        v = v + 0.3 * rng.normal(size=one) * axis
    return _conserved(rho, mach * math.sqrt(GAMMA * 1e-4) * v, 1e-4 * rho)


def _dt(U):
    """CFL dt of each patch's interior in extended precision."""
    U = U[:, :, 2:-2, 2:-2, 2:-2].astype(LD)
    ir = 1 / U[0]
    p = (LD(GAMMA) - 1) * (U[4] - LD(0.5) * (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) * ir)
    s = (abs(U[1]) + abs(U[2]) + abs(U[3])) * ir + 3 * np.sqrt(LD(GAMMA) * p * ir)
    return LD(0.8) * LD(DX) / s.reshape(PATCHES, -1).max(1)


def _on_gpu(U):
    return [torch.from_numpy(np.ascontiguousarray(U[:, i])).cuda() for i in range(PATCHES)]


@pytest.mark.parametrize("precision,kind,mach,bound", [
    ("fp64", "white", 0.3, 1.087e-16), ("fp64", "white", 1.0, 1.004e-16), ("fp64", "cold", 2.0, 1.387e-16),
    ("df64", "white", 0.3, 2.908e-15), ("df64", "white", 1.0, 2.621e-15), ("df64", "cold", 2.0, 6.002e-15),
    ("df64", "cold", 5.0, 1.904e-14)])
def test_time_step_error(precision, kind, mach, bound):
    U = _patches(kind, mach)
    c = ctx(precision, cfl=0.8)
    T = _on_gpu(U)
    dt = torch.empty(PATCHES, dtype=torch.float64, device="cuda")
    hy.hydro_cfl_dt(c, [hy.patch(t, 2, DX) for t in T], dt)
    want = _dt(U)
    err = ((dt.cpu().numpy().astype(LD) - want) / want).astype(np.float64)
    hy.hydro_finalize(c)
    assert math.sqrt((err ** 2).mean()) <= 1.01 * bound


@pytest.mark.parametrize("limiter", ["minmod", "mc"])
@pytest.mark.parametrize("kind,mach,bounds", [
    ("white", 1.0, (8.01e-16, 1.87e-15, 1.87e-15, 1.84e-15, 2.16e-15)),
    ("cold", 2.0, (1.628e-15, 2.964e-15, 2.920e-15, 2.867e-15, 4.151e-15)),
    ("cold", 5.0, (2.375e-15, 3.981e-15, 3.889e-15, 3.773e-15, 5.391e-15))])
def test_double_float_step_error(limiter, kind, mach, bounds):
    """Against the step in double, whose errors are 20 times smaller."""
    U = _patches(kind, mach)
    T = _on_gpu(U)
    dt = torch.from_numpy((_dt(U) * LD(0.7)).astype(np.float64)).cuda()
    out = {}
    for precision in ("fp64", "df64"):
        c = ctx(precision, limiter, cfl=0.8)
        O = torch.zeros((PATCHES, 5) + (EDGE,) * 3, dtype=torch.float64, device="cuda")
        hy.hydro_step(c, [hy.patch(t, 2, DX) for t in T], [hy.patch(o, 0, DX) for o in O], dt)
        out[precision] = O.transpose(0, 1).reshape(5, -1)
        hy.hydro_finalize(c)
    err = ((out["df64"] - out["fp64"]).norm(dim=1) / out["fp64"].norm(dim=1)).cpu().numpy()
    assert (err <= 1.01 * np.array(bounds)).all(), err


@pytest.fixture(scope="module")
def extended_step(tmp_path_factory):
    """The oracle's periodic step in extended precision: the same sources with long double for double."""
    d = tmp_path_factory.mktemp("extended")
    here = os.path.dirname(os.path.abspath(oracle.__file__))
    with open(str(d / "capi.cpp"), "w") as f:
        f.write("".join("#include <%s>\n" % h for h in ("algorithm", "cmath", "cstdint", "cstring", "vector", "type_traits")))
        f.write("#include <omp.h>\n#define double long double\n#include \"oracle_capi.cpp\"\n")
    so = str(d / "extended.so")
    subprocess.check_call(oracle._build.command([str(d / "capi.cpp")], so) + ["-I" + here])
    lib = ctypes.CDLL(so)

    class Config(ctypes.Structure):
        _fields_ = [(n, ctypes.c_longdouble) for n in ("gamma", "cfl", "rho_floor", "p_floor")] + [("limiter", ctypes.c_int)]

    vp, ld, i = ctypes.c_void_p, ctypes.c_longdouble, ctypes.c_int
    lib.oracle_step_periodic.argtypes = [ctypes.POINTER(Config), vp, vp, i, i, i, ld, ld]

    def step(U, dx, dt, limiter):
        U = np.ascontiguousarray(U, dtype=LD)
        out = np.empty_like(U)
        cfg = Config(GAMMA, 0.8, 1e-10, 1e-14, oracle.LIMITERS[limiter])
        assert lib.oracle_step_periodic(ctypes.byref(cfg), U.ctypes.data, out.ctypes.data, *U.shape[:0:-1], dx, dt) == 0
        return out

    return step


def test_double_step_error(extended_step):
    """White noise at Mach 3, where every face's wave speeds and contact matter."""
    n, total, norm = 32, np.zeros(5), np.zeros(5)
    c = ctx("fp64", cfl=0.8)
    for seed in range(4):
        U = _white(np.random.default_rng(seed), (n,) * 3, 3.0)
        a = torch.from_numpy(U).cuda()
        b, dt = torch.empty_like(a), torch.empty(1, dtype=torch.float64, device="cuda")
        hy.hydro_cfl_dt(c, hy.patch(a, 0, 1.0 / n), dt)
        hy.hydro_step(c, hy.patch(a, 0, 1.0 / n), hy.patch(b, 0, 1.0 / n), dt)
        want = extended_step(U, 1.0 / n, dt.item(), "minmod")
        err = (b.cpu().numpy() - want).astype(np.float64)
        total += (err ** 2).reshape(5, -1).sum(1)
        norm += (want ** 2).astype(np.float64).reshape(5, -1).sum(1)
    hy.hydro_finalize(c)
    err = np.sqrt(total / norm)
    assert (err <= np.array([6.079e-17, 9.613e-17, 9.596e-17, 9.335e-17, 1.186e-16])).all(), err
