"""The on-chip re-sort's steps (csrc/key_sort.cuh, compiled for the host): whatever the radii hold -- NaNs and
infinities from an overflowing push among them -- the result is the stable sort's permutation of the rings, and no
access leaves a run."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2603_16623_gb300", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("key_sort") / "key_sort")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "key_sort_host.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("per_thread", [2, 4, 8])
@pytest.mark.parametrize("kind", ["near", "reversed", "shuffled", "ties", "one nan", "nan and inf", "all nan"])
def test_resort_is_a_permutation(program, per_thread, kind):
    res = subprocess.run([program, str(per_thread), kind], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-2000:]
