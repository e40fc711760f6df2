"""Build libsfac.so in-tree with nvcc for sm_103a (GB300).

The three translation units compile in parallel; the library links the CUDA
runtime statically, so it needs only the driver at run time.
"""
from __future__ import annotations

import os
import shutil
import subprocess

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OBJDIR = os.path.join(PKG, "_build")
LIBDIR = os.path.join(PKG, "lib")
LIB = os.path.join(LIBDIR, "libsfac.so")

SOURCES = ["sfac_plan.cu", "sfac_host.cu", "sfac_pass_f64.cu", "sfac_pass_f32.cu", "sfac_pass_pad_f64.cu",
           "sfac_pass_pad_f32.cu", "sfac_batch.cu",
           "sfac_batch_f32.cu", "sfac_batch_f64.cu", "sfac_server.cu",
           "sfac_noalloc.cu", "sfac_diag.cu", "sfac_pass_staged_f32.cu", "sfac_probe.cu", "sfac_steps.cu",
           "sfac_tc_build.cu", "sfac_tc_pass.cu", "sfac_tc_pass_f32.cu",
           "sfac_tc_steps.cu", "sfac_tc_long.cu"]
HEADERS = ["sfac_fft.cuh", "sfac_pass.cuh", "sfac_internal.h", "sfac_host.h", "sfac_batch.cuh",
           "sfac_batch_launch.h", "sfac_diag.h", "sfac_diag_rule.h", "sfac_tma.cuh", "sfac_steps.h",
           "sfac_tc.h", "sfac_tcgen05.cuh", "sfac_jq_fixed.cuh", "sfac_tc_tile.cuh", "sfac_tc_tile_f32.cuh", "sfac_tc_launch.cuh"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc_path() -> str:
    cand = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found: libsfac needs the CUDA toolkit to build")
    return cand


def _inputs():
    files = [os.path.join(CSRC, f) for f in SOURCES + HEADERS]
    files.append(os.path.join(INCLUDE, "sfac.h"))
    files.append(os.path.abspath(__file__))
    return files


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(f) > t for f in _inputs())


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile and link libsfac.so if it is missing or older than its sources."""
    if not force and not is_stale():
        return LIB
    nvcc = nvcc_path()
    os.makedirs(OBJDIR, exist_ok=True)
    os.makedirs(LIBDIR, exist_ok=True)
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC",
                    "-I", INCLUDE, "-I", CSRC]
    procs, objs = [], []
    for src in SOURCES:
        obj = os.path.join(OBJDIR, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [nvcc] + flags + ["-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd))
        procs.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    errors = []
    for cmd, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0:
            errors.append(" ".join(cmd) + "\n" + out.decode(errors="replace"))
        elif verbose and out:
            print(out.decode(errors="replace"))
    if errors:
        raise RuntimeError("libsfac build failed:\n" + "\n".join(errors))
    tmp = LIB + ".tmp"
    cmd = [nvcc] + ARCH + ["-shared", "-o", tmp] + objs
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    if r.returncode != 0:
        raise RuntimeError("libsfac link failed:\n" + r.stdout.decode(errors="replace"))
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
