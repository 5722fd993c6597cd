"""The double-precision march's logarithm (csrc/f64_log.cuh, compiled for the host) against extended precision.

Bound: half an ulp of the last sum, a quarter of the sum before it (its value is at most the result's, one binade
lower where -ln c and the series nearly cancel), and less than 2^-6 of the series and the low parts: 0.77 ulp, below
the 1 ulp the library's log states."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2603_16623_gb300", "csrc")


def test_log_is_as_accurate_as_the_library_states(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "f64_log")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, os.path.join(HERE, "f64_log_host.cpp"),
                    "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
    worst = [float(v) for v in res.stdout.split()]
    assert len(worst) == 4 and max(worst) < 0.77, worst
