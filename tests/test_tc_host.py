"""Index arithmetic of the tensor-core passes, compiled for the host
(tests/host_tc): the whole-sector loads of contiguous lines never leave the
field, whatever its length, line count and alignment, and lines inside the
field always take them."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2209_08437_gb300", "csrc")


def test_contiguous_loads_stay_in_the_field(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "check_loads")
    r = subprocess.run([cxx, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "tests", "host_fft", "shim"), "-I", CSRC,
                        "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "host_tc", "check_loads.cpp"),
                        "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
    loads, grouped = map(int, out.stdout.split())
    assert loads > 100000 and grouped > 0.9 * loads
