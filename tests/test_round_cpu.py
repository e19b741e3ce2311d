"""CPU: the order of a 128-thread group's MMA round trips (csrc/stf_round.h) on host
threads: whichever waits run out, every warp comes to the end of its rounds."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2305_05810_gb300", "csrc")


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("round") / "model")
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-pthread", "-I" + CSRC, os.path.join(HERE, "round_model.cpp"), "-o", exe])
    return exe


@pytest.mark.parametrize("tiles", [1, 2, 3])
def test_every_warp_comes_to_its_end(model, tiles):
    r = subprocess.run([model, str(tiles)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
