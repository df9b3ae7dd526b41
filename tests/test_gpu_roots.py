"""The reciprocals, quotients and square roots that double and double-float arithmetic form from the
hardware's approximations, one by one against extended precision: the error bounds stated beside them,
over the stated exponent range, and what they give for zeros and NaN."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_1412_0934_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "df.cuh"
#include "hydro_device.cuh"
using namespace hydro;
__global__ void k_eval(int op, const double* a, const double* b, double* hi, double* lo, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double x = a[i], y = b[i];
  df r(0.f, 0.f);
  lo[i] = 0.0;
  switch (op) {
    case 0: hi[i] = rcp_(x); return;
    case 1: hi[i] = div_(x, y); return;
    case 2: hi[i] = rsqrt_(x); return;
    case 3: hi[i] = sound_speed(x, y); return;
    case 4: r = rcpu_(df(x)); break;
    case 5: r = quot_(df(x), df(y)); break;
    case 6: r = rootu_(df(x)); break;
    case 7: r = first_(rootq_(pair_(df(x), df(y)), pair_(df(y), df(x)))); break;
    case 8: r = second_(rootq_(pair_(df(y), df(x)), pair_(df(x), df(y)))); break;
    case 9: r = first_(rcpu_(pair_(df(x), df(y)))); break;
    case 10: r = second_(rootu_(pair_(df(y), df(x)))); break;
  }
  hi[i] = (double)r.h;
  lo[i] = (double)r.l;
}
extern "C" int roots_eval(int op, const double* a, const double* b, double* hi, double* lo, int n) {
  k_eval<<<(n + 255) / 256, 256>>>(op, a, b, hi, lo, n);
  return (int)cudaDeviceSynchronize();
}
"""
LD = np.longdouble
N = 1 << 20


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    d = tmp_path_factory.mktemp("roots")
    src, so = str(d / "roots.cu"), str(d / "roots.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.check_call([build.NVCC] + build.ARCH + build.FLAGS + ["-shared", "-o", so, src])
    lib = ctypes.CDLL(so)
    vp = ctypes.c_void_p
    lib.roots_eval.argtypes = [ctypes.c_int, vp, vp, vp, vp, ctypes.c_int]

    def run(op, a, b=None):
        a = torch.as_tensor(np.ascontiguousarray(a)).cuda()
        b = torch.ones_like(a) if b is None else torch.as_tensor(np.ascontiguousarray(b)).cuda()
        hi, lo = torch.empty_like(a), torch.empty_like(a)
        assert lib.roots_eval(op, a.data_ptr(), b.data_ptr(), hi.data_ptr(), lo.data_ptr(), a.numel()) == 0
        return hi.cpu().numpy().astype(LD) + lo.cpu().numpy().astype(LD)

    return run


def _numbers(seed, exponents):
    """Random mantissas over the exponents, with powers of two and their neighbours."""
    rng = np.random.default_rng(seed)
    x = np.ldexp(rng.uniform(1.0, 2.0, N), rng.integers(exponents[0], exponents[1] + 1, N))
    p = np.ldexp(1.0, rng.integers(exponents[0], exponents[1] + 1, N // 16))
    x[:3 * (N // 16)] = np.concatenate([p, np.nextafter(p, 0.0), np.nextafter(p, np.inf)])
    return x


def _pairs(x):
    """What a double-float holds of x."""
    h = x.astype(np.float32)
    return h.astype(LD) + (x - h).astype(np.float32).astype(LD)


def _worst(got, want):
    return float(np.abs((got - want) / want).max())


def test_double(evaluate):
    u = 2.0 ** -53
    x, y = _numbers(1, (-1018, 1018)), _numbers(2, (-1018, 1018))
    assert _worst(evaluate(0, x), 1 / x.astype(LD)) <= u + 2.0 ** -57
    assert _worst(evaluate(0, -x), -1 / x.astype(LD)) <= u + 2.0 ** -57
    assert _worst(evaluate(2, x), np.sqrt(x.astype(LD))) <= 1.5 * u + 2.0 ** -57
    assert _worst(evaluate(3, x, y), np.sqrt(x.astype(LD)) / np.sqrt(y.astype(LD))) <= 2 * u + 2.0 ** -55
    x, y = _numbers(3, (-450, 450)), _numbers(4, (-450, 450))
    assert _worst(evaluate(1, x, y), x.astype(LD) / y.astype(LD)) <= u + 2.0 ** -62
    assert _worst(evaluate(1, -x, y), -x.astype(LD) / y.astype(LD)) <= u + 2.0 ** -62


def test_double_zero_and_nan(evaluate):
    """A zero's root is zero; a NaN, of either sign, stays one."""
    nan = np.array([0x7ff8 << 48, 0xfff8 << 48, 2 ** 63 - 1, 2 ** 64 - 1], dtype=np.uint64).view(np.float64)
    one = np.ones_like(nan)
    assert np.isnan(nan).all()
    for r in (evaluate(0, nan), evaluate(1, nan, one), evaluate(1, one, nan), evaluate(2, nan), evaluate(3, nan, one),
              evaluate(3, one, nan)):
        assert np.isnan(r).all()
    zero = np.array([0.0, -0.0, 1e-310])
    assert (evaluate(2, zero) == 0).all() and (evaluate(3, zero, np.full(3, 2.0)) == 0).all()


def test_double_float(evaluate):
    """Operands and quotients between 2^-91 and 2^91: beyond about 2^-100 a low word leaves float's range."""
    x, y = _numbers(5, (-45, 45)), _numbers(6, (-45, 45))
    X, Y = _pairs(x), _pairs(y)
    assert _worst(evaluate(4, x), 1 / X) <= 2.0 ** -45
    assert _worst(evaluate(4, -x), -1 / X) <= 2.0 ** -45
    assert _worst(evaluate(9, x, y), 1 / X) <= 2.0 ** -45
    assert _worst(evaluate(5, x, y), X / Y) <= 2.0 ** -45
    assert _worst(evaluate(5, -x, y), -X / Y) <= 2.0 ** -45
    assert _worst(evaluate(6, x), np.sqrt(X)) <= 2.0 ** -45
    assert _worst(evaluate(10, x, y), np.sqrt(X)) <= 2.0 ** -45
    for op in (7, 8):
        assert _worst(evaluate(op, x, y), np.sqrt(X) / np.sqrt(Y)) <= 2.0 ** -43


def test_double_float_zero_and_nan(evaluate):
    nan, one, zero = np.full(4, np.nan), np.ones(4), np.zeros(4)
    for op in (6, 10):
        assert np.isnan(evaluate(op, nan)).all() and (evaluate(op, zero) == 0).all()
    for op in (7, 8):
        assert np.isnan(evaluate(op, nan, one)).all() and np.isnan(evaluate(op, one, nan)).all()
