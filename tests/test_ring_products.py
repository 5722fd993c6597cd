"""The register marches' products of ring matrices (csrc/ring_jump.cuh, compiled for the host) in float, over uniform
rings out to 6, in the association of their scans, against double.

Bound on how far a solution's change over a distance of at most 1 is off: each of the two threads' products takes
three combinations at its full size (in the warp, over the block's warps, with the blocks before) of three roundings
of at most 2^-24 each, so 18 x 2^-24.  (Matrices rounded as they are, 1 + h r among them, were off by 3e-6 to 2e-5.)"""
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
    exe = str(tmp_path_factory.mktemp("ring_jump") / "ring_jump")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, os.path.join(HERE, "ring_jump_host.cpp"),
                    "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("per_thread", [1, 2, 3, 4])
@pytest.mark.parametrize("rings", [500, 3269, 6393, 8192])
def test_products_keep_the_difference_from_the_identity(program, rings, per_thread):
    res = subprocess.run([program, str(rings), str(per_thread)], capture_output=True, text=True, check=True)
    worst = [float(v) for v in res.stdout.split()]
    assert len(worst) == 2 and max(worst) < 18 * 2.0 ** -24, worst
