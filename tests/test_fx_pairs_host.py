"""The two-lane double-float helpers of the particle kernel (packed FP32
instructions on the GPU), compiled for the host: lane by lane the bits of the
scalar helpers, and the fixed-point sum of an increment within one unit of
2^-56 up to the limits of its range."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_pair_helpers_on_host(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "fxpairs"
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-x", "c++",
                           os.path.join(HERE, "fx_pair_check.cpp"), "-o", str(exe), "-lm"])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert "bad 0" in out.stdout
