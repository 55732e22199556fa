"""The three-part FP32 arithmetic of the direct sum on the CPU: the same
headers compiled for the host, over the scaled distances the kernel meets.

Tolerances, in units of 2^-53 (an FP64 rounding is up to 1): the third part
carries every rounding error of terms of size 2^-24 in FP32, so what is lost is
a few roundings of numbers of size 2^-31 at most (the logarithm's series: fewer
than eight, 2^-52 in the worst case, relative to max(1, |log|)) or 2^-42 (the
distance, the reciprocal root), and the same per term of a sum.  The tables'
last part is rounded to FP32 at 2^-35."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1609_08130_gb300", "csrc")

BOUNDS = {"table": 2.0 ** -6, "exponent": 2.0 ** -6, "dist2": 2.0 ** -6, "dist3": 2.0 ** -6, "log": 2.0,
          "rsqrt": 2.0 ** -5, "sum": 2.0 ** -5}


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path_factory.mktemp("direct_sum") / "host")
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-o", exe,
                           os.path.join(HERE, "direct_sum_host.cpp")])
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout
    return {k: float(v) for k, v in (line.split() for line in out.splitlines())}


@pytest.mark.parametrize("name", list(BOUNDS))
def test_error_is_below_an_fp64_rounding(errors, name):
    assert errors[name] <= BOUNDS[name], errors
