"""Builds the C-ABI library ``libattn_b200.so`` in-tree with nvcc for sm_100a."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import tempfile
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
LIB = PKG / "libattn_b200.so"
SOURCES = ["api.cu", "attn_fwd_sm100.cu", "attn_rows_sm100.cu"]
HEADERS = ["ptx.cuh", "weight_map.cuh", "attn_kernel_common.cuh", "softmax_math.cuh", "../../include/attn.h"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and Path(cand).exists():
            return cand
    raise RuntimeError("nvcc not found")


def needs_build() -> bool:
    if not LIB.exists():
        return True
    t = LIB.stat().st_mtime
    return any((CSRC / f).stat().st_mtime > t for f in SOURCES + HEADERS)


def build(force: bool = False, verbose: bool = False) -> Path:
    if not force and not needs_build():
        return LIB
    tmp = LIB.with_suffix(f".so.tmp{os.getpid()}")
    flags = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
             "--ptxas-options=-v" if verbose else "-w"]
    with tempfile.TemporaryDirectory() as objs:
        # one compiler per source file, side by side
        jobs = [(f, subprocess.Popen([_nvcc(), *flags, "-c", "-o", f"{objs}/{f}.o", str(CSRC / f)],
                                     stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)) for f in SOURCES]
        logs = [job.communicate()[0] for _, job in jobs]
        for (f, job), log in zip(jobs, logs):
            if job.returncode != 0:
                raise RuntimeError(f"nvcc failed on {f}:\n{log}")
        link = subprocess.run([_nvcc(), "-shared", "-o", str(tmp), *(f"{objs}/{f}.o" for f in SOURCES), "-lcudart"],
                              capture_output=True, text=True)
        if link.returncode != 0:
            raise RuntimeError("nvcc failed at the link:\n" + link.stdout + link.stderr)
    if verbose:
        print("".join(logs))
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
