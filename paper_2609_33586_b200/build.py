"""Builds the C-ABI library ``libattn_b200.so`` (nvcc, sm_100a) and the host module ``_host`` in-tree."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig
import tempfile
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
LIB = PKG / "libattn_b200.so"
HOST = PKG / f"_host{sysconfig.get_config_var('EXT_SUFFIX')}"
SOURCES = ["api.cu", "attn_fwd_sm100.cu", "attn_fwd_split_sm100.cu", "attn_fwd_streams_sm100.cu", "attn_fwd_tau_sm100.cu", "attn_rows_sm100.cu"]
HEADERS = ["ptx.cuh", "kv_ring.cuh", "plan.h", "attn_fwd_kernel.cuh", "attn_streams_kernel.cuh", "weight_map.cuh", "attn_kernel_common.cuh", "softmax_math.cuh", "../../include/attn.h"]


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


def host_is_current(path: Path, torch_version: str) -> bool:
    """Whether the host module at `path` is newer than its sources and was built for this torch (its text says which)."""
    if not path.exists() or path.stat().st_mtime < max((CSRC / f).stat().st_mtime for f in ("host_binding.cpp", "../../include/attn.h")):
        return False
    return f"host module for torch {torch_version}\0".encode() in path.read_bytes()


def build_host(force: bool = False) -> Path:
    """The CPython module that does the per-call host work (csrc/host_binding.cpp)."""
    src = CSRC / "host_binding.cpp"
    import torch
    if not force and host_is_current(HOST, torch.__version__):
        return HOST
    troot = Path(torch.__file__).resolve().parent
    cuda = Path(_nvcc()).resolve().parent.parent
    tmp = HOST.with_suffix(f".so.tmp{os.getpid()}")
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-w", f'-DROWMAX_TORCH="{torch.__version__}"', f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           f"-I{sysconfig.get_paths()['include']}", f"-I{troot}/include", f"-I{troot}/include/torch/csrc/api/include",
           f"-I{cuda}/include", "-o", str(tmp), str(src), f"-L{troot}/lib", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda",
           "-ltorch_python", f"-Wl,-rpath,{troot}/lib"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed on host_binding.cpp:\n" + res.stdout + res.stderr)
    os.replace(tmp, HOST)
    return HOST


def build(force: bool = False, verbose: bool = False) -> Path:
    build_host(force)
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
        link = subprocess.run([_nvcc(), *flags[:2], "-shared", "-o", str(tmp), *(f"{objs}/{f}.o" for f in SOURCES), "-lcudart"],
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
