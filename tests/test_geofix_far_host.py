"""The fixed-point RK4 step (csrc/geofix.cuh) far from the hole, where the transverse momentum's scale 2^g
grows with r: rays from cameras at 1e5 to 1e12 M within the bounds that test_geofix_host.py states, and
random states out to there, with every shift count below its operand's width. No GPU is used."""
import os
import shutil
import subprocess
import tempfile

import pytest

from test_geofix_host import SRC


@pytest.fixture(scope="module")
def far():
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    text = SRC.replace("rc = 1000.0,", "rc = R_CAM,").replace("std::pow(10.0, 4 * U()) * rh", "std::pow(10.0, 12.04 * U()) * rh")
    assert text.count("R_CAM") == 1 and text.count("12.04") == 1
    with tempfile.TemporaryDirectory() as d:
        src = os.path.join(d, "t.cpp")
        open(os.path.join(d, "cuda_runtime.h"), "w").close()
        open(src, "w").write(text)

        def build(r_cam):
            out = os.path.join(d, "t" + r_cam)
            r = subprocess.run(["g++", "-O2", "-std=c++17", "-fwrapv", "-ffp-contract=off", "-fsanitize=shift-exponent",
                                "-fno-sanitize-recover=all", "-DR_CAM=" + r_cam, "-I", d, "-I",
                                os.path.join(root, "paper_2302_02733_gb300", "csrc"), "-o", out, src],
                               capture_output=True, text=True)
            assert r.returncode == 0, r.stderr
            return out

        yield build


@pytest.mark.parametrize("r_cam", ["1e5", "3e6", "5e6", "1e8", "1e10", "1e12"])
def test_far_rays(far, r_cam):
    r = subprocess.run([far(r_cam), "rays", "0.9375", "50", "4"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


def test_far_states(far):
    r = subprocess.run([far("1000.0"), "box", "400000"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
