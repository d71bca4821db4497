"""The catalog recipe's reciprocal, quotient, square root and quotient by ln 2 (refined from the
hardware's approximations) against the IEEE operations, bit for bit: every mantissa, over the
exponents that the recipe reaches for any accepted parameters and beyond."""
import ctypes
import os
import subprocess

import pytest

from paper_2602_18560_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def differences(tmp_path_factory):
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    so = str(tmp_path_factory.mktemp("gen_arith") / "libgen_arith.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "gen_arith.cu")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I" + build.CSRC, "-shared", src, "-o", so],
                   check=True, capture_output=True, text=True)
    fn = ctypes.CDLL(so).gen_arith_differences
    fn.restype = ctypes.c_longlong
    return fn


@pytest.mark.parametrize("what, e0, e1", [
    (0, -110, 110),   # 1 / b: the incomplete gamma function's fractions reach 1e-30 and 1e30
    (1, -67, 72),     # sqrt: of 2^-23 .. 2^55 (polar method) and of logarithms
    (2, -100, 120),   # x / ln 2: any argument of exp whose quotient is not 0
    (3, -60, 60),     # a / b, four random dividends for every divisor
])
def test_equal_to_the_ieee_operation(differences, what, e0, e1):
    assert differences(what, e0, e1) == 0
