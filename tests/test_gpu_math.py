"""Self-written FP32 functions against CUDA's FP64 ones, over the ranges that
their callers reach (math_errors.cu).  Bounds, with u = 2^-24:
  atan_unit    0.5 ulp for the last rounding and, at the top of its range (where
               1 ulp = u), u times what s = x^2 (0.143), x s (0.215) and Q's last step
               (1.3 x 0.215) carry over: 1.14; 2.4e-9 relative for the fit (0.04 ulp);
  recip_times  0.5 ulp, and the product of two 1.5 ulp errors;
  rsqrt_times  num r, x r (half of it) and the sum round once each: 2.5 u, and the
               square of the approximation's 2^-22.9;
  inv_sqrt     0.5 ulp, and 1.5 times the square of 2.5 ulp."""
import ctypes as C
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def error(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_11313_gb300 import build as b
    so = str(tmp_path_factory.mktemp("math") / "libmath_errors.so")
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-shared", os.path.join(HERE, "math_errors.cu"), "-o", so], check=True)
    fn = C.CDLL(so).math_error
    fn.argtypes = [C.c_int, C.c_ulonglong, C.POINTER(C.c_double)]

    def worst(what, n):
        v = C.c_double()
        assert fn(what, n, C.byref(v)) == 0
        print(f"worst error of {n}: {v.value:.4f} ({v.value * 2 ** 24:.3f} x 2^-24)")
        return v.value

    return worst


def test_arctangent(error):
    assert error(0, 0x0f800001) <= 1.2      # every float of [2^-31, 1], and its negative


def test_quotient(error):
    assert error(1, 1 << 28) <= 0.51


def test_quotient_by_square_root(error):
    assert error(2, 1 << 28) <= 2.51 * 2.0 ** -24


def test_inverse_square_root(error):
    assert error(3, 1 << 26) <= 0.51
