"""The range test of the fixed-point position sum, compiled for the host: an
increment with a NaN or an infinity in any one part is refused."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_increment_range_on_host(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "fxincrement"
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-x", "c++",
                           os.path.join(HERE, "fx_increment_check.cpp"), "-o", str(exe), "-lm"])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert "bad 0" in out.stdout
