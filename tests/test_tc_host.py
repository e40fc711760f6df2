"""Host-side rules of the kernels, compiled for the host (tests/host_tc)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2209_08437_gb300", "csrc")


def build(name, tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / name)
    r = subprocess.run([cxx, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "tests", "host_fft", "shim"), "-I", CSRC,
                        "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "host_tc", name + ".cpp"),
                        "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    return exe


def test_contiguous_loads_stay_in_the_field(tmp_path):
    """The whole-sector loads of contiguous lines never leave the field, whatever
    its length, line count and alignment, and lines inside the field always take
    them."""
    out = subprocess.run([build("check_loads", tmp_path)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
    loads, grouped = map(int, out.stdout.split())
    assert loads > 100000 and grouped > 0.9 * loads


# Grids timed both ways on GB300 (us a call: FFT passes, direct sums).
DIAG_FFT = {(2048,): (124, 752), (1024,): (75, 219), (2048, 8): (148, 774), (8, 2048): (146, 811), (1024, 4): (90, 222),
            (1024, 32): (105, 224), (2047, 4): (142, 768), (4, 1000): (90, 218), (1500, 10): (149, 441), (700, 70): (103, 138),
            (2, 2, 2048): (144, 802), (4, 4, 1024): (106, 398), (8, 8, 512): (118, 231), (16, 16, 256): (119, 151),
            (3, 114, 256): (108, 249), (17, 29, 256): (108, 194), (63, 63, 63): (136, 148)}
DIAG_DIRECT = {(64,): (61, 33), (256,): (65, 45), (64, 64): (91, 32), (127, 127): (76, 34), (255, 255): (79, 69),
               (256, 256): (110, 69), (512, 64): (103, 82), (300, 40): (78, 58), (32, 32, 32): (119, 55),
               (64, 32, 16): (119, 57), (8, 8, 8): (86, 32), (100, 20, 30): (94, 71)}


def test_diagnostics_take_the_faster_route(tmp_path):
    def query(n):
        lens, inner = [], 1
        for l, v in enumerate(n):
            padded = not (v >= 4 and v & (v - 1) == 0) or (l > 0 and inner % 2 == 1)
            N = v
            if padded:
                N = 4
                while N < 2 * v - 1:
                    N *= 2
            lens.append(f"{N} {int(padded)}")
            inner *= v
        return " ".join([str(len(n)), *map(str, n), *lens])

    grids = [*DIAG_FFT, *DIAG_DIRECT]
    out = subprocess.run([build("check_diag_rule", tmp_path)], input="\n".join(map(query, grids)), capture_output=True,
                         text=True, timeout=60)
    got = dict(zip(grids, map(int, out.stdout.split())))
    assert [n for n in DIAG_FFT if got[n]] == [] and [n for n in DIAG_DIRECT if not got[n]] == []
