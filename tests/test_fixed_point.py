"""The sweeps' fixed-point arithmetic on the host: csrc/fixed.cuh compiled by the C++ compiler and compared
with long double (exponential, conversions, the moments of one pass over the rule for flat and
peaked densities). The bounds are the rounding steps' own; see fixed_point_check.cpp."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2205_08417_gb300", "csrc")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fx") / "check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-I" + CSRC, "-o", exe, "-x", "c++",
                           os.path.join(HERE, "fixed_point_check.cpp")])

    def run(*args):
        ratio = float(subprocess.check_output([exe, *map(str, args)]))
        print("error / bound", ratio)
        return ratio
    return run


def test_exponential(check):
    assert check("exp") <= 1.0  # 2^-51 relative


def test_scaled_exponential(check):
    assert check("scaled") <= 1.0  # 2^-51 relative


def test_conversions(check):
    assert check("conv") <= 1.0  # half a unit


@pytest.mark.parametrize("N,order", [(1, 2), (1, 7), (2, 3), (2, 40), (3, 9), (3, 20), (3, 30), (4, 15), (5, 6), (5, 64)])
def test_moments(check, N, order):
    assert check("sums", N, order) <= 1.0
