"""The kernels' own arithmetic against the operations it stands in for
(arithmetic.cu, built on the kernels' header): FP32 to FP64 over all FP32
patterns and FP64 to FP32 on, beside and halfway between them and over random
values of every exponent, bit for bit (a NaN for a NaN); 1/x within one
representable value of the division and 1/sqrt(x) within two of the root and
division, on both sides of the powers 2^-900 and 2^900 where they change over.

The bounds: two Newton steps from an approximation good to 2^-20 leave the
rounding of the last multiply-add, half a unit, so 1/x is at most one
representable value from the rounded quotient. For 1/sqrt(x) the step's product
y y is rounded too, which moves the result by 2^-54 of itself, and the root and
division it is compared with round twice: together 2.5 units of the smaller
spacing at a power of two, so at most two representable values."""
import subprocess

import pytest

from paper_2509_11100_gb300 import build

pytestmark = pytest.mark.gpu


def test_conversions_and_reciprocals(tmp_path):
    exe = tmp_path / "arithmetic"
    subprocess.run([build.nvcc()] + build.ARCH + build.NVFLAGS + [__file__.replace("test_gpu_arithmetic.py", "arithmetic.cu"),
                                                                  "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["0"] * 5, dict(zip(("widen", "narrow", "1/x", "1/sqrt(x)", "special"), out))
