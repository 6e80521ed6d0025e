"""The integer form of the FP64 collision, compiled for the host, against
quadruple precision: its error at every density it takes, and the densities it
leaves to the FP64 form."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytest.importorskip("numpy")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_1610_02733_gb300 import build_lib
    exe = str(tmp_path_factory.mktemp("fixed") / "check")
    subprocess.check_call([build_lib.nvcc()] + build_lib.ARCH + [
        "-O2", "-std=c++17", "-w", "-I", build_lib.CSRC, "-I", os.path.join(ROOT, "include"), "-o", exe,
        os.path.join(ROOT, "tests", "fixed_collision_check.cu")])
    return exe


@pytest.mark.parametrize("rho0", [1.0, 3.7e-9])
def test_error_and_range(program, rho0):
    nodes = 80
    rows = [[float(v) for v in line.split()]
            for line in subprocess.check_output([program, str(nodes), repr(rho0)], text=True).splitlines()]
    assert len(rows) == 22
    for rel, taken, rms, rms64, worst, mass, mass64 in rows:
        if rel < 0.305:  # below 5/16: FP64 is the more accurate
            assert taken == 0, rel
            continue
        if rel >= 0.33:  # (populations 5 % around their means: the density within 2 % of its own)
            assert taken == nodes, rel
        # no larger than the FP64 form's, 1.4e-17 of the density at the least
        assert rms <= 1.4e-17 and rms <= rms64, (rel, rms, rms64)
        # units of 2^(e - 60) beyond the result's own rounding: the populations'
        # rounding through the relaxation 3, the changes' rounding 2.5, their
        # division by 9 4.9, the last shift 0.5
        assert worst <= 12, (rel, worst)
        # 19 rounding errors of rms 5e-18 a node, 80 nodes: 2.5e-18; five times that
        assert abs(mass) <= 1.25e-17, (rel, mass)


def test_reciprocal_and_root(program):
    # 1/rho and sqrt(rho) over every density rho0 in 2^-60 .. 2^60 admits: half a
    # unit of the last place for the final rounding, and little else
    inv, root = [float(v) for v in subprocess.check_output([program, "factors"], text=True).split()]
    assert 0 < inv <= 0.51 and 0 < root <= 0.51, (inv, root)


def test_product_as_an_integer(program):
    # rounded right wherever it says it fits, fitting below 2^61, and never
    # fitting with a factor that is not finite, whatever the other one
    assert subprocess.check_output([program, "products"], text=True).split() == ["0", "0", "0"]
