"""The AdamW step's divisions and square root by Newton steps against CUDA's correctly rounded operations, directly.

tests/newton_check.cu is compiled against the library's device code: the two divisions for all 2^23 numerator mantissas
and 4096 divisor mantissas (those next to 1 and 2 and evenly spread ones; DSM_EXHAUSTIVE=1: all 2^46 pairs, about a
minute), the root for every mantissa at every exponent that it is used at, and the group of four against the step written
with the IEEE operations, bit for bit, with moments from every range that it tells apart: zeros, decayed and denormal
values, usual ones, huge ones and infinities, the ends of the ranges, whole groups of one kind and mixed ones.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu


def test_newton_forms_equal_the_ieee_operations(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2411_17866_gb300 import build
    exe = str(tmp_path / "newton_check")
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, os.path.join(ROOT, "tests", "newton_check.cu"), "-o", exe],
                   check=True, capture_output=True, timeout=300)
    divisors = 1 << 23 if os.environ.get("DSM_EXHAUSTIVE") else 4096
    r = subprocess.run([exe, str(divisors), str(1 << 24)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.split() == ["div_by", "0", "div_newton", "0", "sqrt_newton", "0", "adamw_group", "0"], r.stdout
