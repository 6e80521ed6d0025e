"""The FP64 quotient, reciprocal and square root that the kernels make from
approximations (GPU) against IEEE division and square root: never further than
the neighbouring number, over every density the contexts admit."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_against_ieee(tmp_path):
    from paper_1610_02733_gb300 import build_lib
    exe = str(tmp_path / "check")
    subprocess.check_call([build_lib.nvcc()] + build_lib.ARCH + [
        "-O3", "-std=c++17", "-w", "-I", build_lib.CSRC, "-I", os.path.join(ROOT, "include"), "-o", exe,
        os.path.join(ROOT, "tests", "fp64_quotient_check.cu")])
    *steps, q, inv, root, h = [float(v) for v in subprocess.check_output([exe], text=True).split()]
    assert h <= -19.0  # what the error bound of the quotient takes for the approximation
    assert max(steps) <= 1, steps
    # half a unit of the last place for the final rounding, and 2^-18 of one
    # (quotient) or what two more roundings of the residual's correction leave
    assert q <= 0.51 and inv <= 0.51 and root <= 0.51, (q, inv, root)
