"""Builds in-tree the CUDA library, paper_2408_15766_b200/libhass_b200.so (sm_100a only), and the binding's native
calls, paper_2408_15766_b200/hass_host-<torch><Python>.so (against the installed torch)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from importlib.metadata import version

HERE = os.path.dirname(os.path.abspath(__file__))
SRC_DIR = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libhass_b200.so")
SOURCES = ["hass_api.cu"]


# every header under csrc/ and the public header: a change to any of them makes the library stale
def _headers() -> list:
    return sorted(f for f in os.listdir(SRC_DIR) if f.endswith((".cuh", ".h"))) + [os.path.join("..", "..", "include", "hass.h")]


# named after what its binary interface depends on: under another torch or Python it is not found, and built again, instead of loaded
HOST = os.path.join(HERE, f"hass_host-{version('torch')}{sysconfig.get_config_var('EXT_SUFFIX')}")
HOST_SOURCES = ["host_calls.cpp", os.path.join("..", "..", "include", "hass.h")]


def _stale(out, sources) -> bool:
    if not os.path.exists(out):
        return True
    t = os.path.getmtime(out)
    return any(os.path.getmtime(os.path.join(SRC_DIR, f)) > t for f in sources)


def build_host(force: bool = False) -> str:
    if not force and not _stale(HOST, HOST_SOURCES):
        return HOST
    from torch.utils.cpp_extension import include_paths, library_paths
    tmp = HOST + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-o", tmp, os.path.join(SRC_DIR, HOST_SOURCES[0])]
    cmd += ["-I" + p for p in include_paths("cuda") + [sysconfig.get_paths()["include"]]]
    cmd += ["-L" + p for p in library_paths("cuda")] + ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, HOST)
    return HOST


def build_library(force: bool = False, verbose: bool = False) -> str:
    if force or _stale(LIB, SOURCES + _headers()):
        _build_cuda(verbose)
    build_host(force)
    return LIB


def _build_cuda(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-o", tmp] + [os.path.join(SRC_DIR, s) for s in SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
