"""Builds in-tree libshotkv.so (the C-ABI library) with nvcc for sm_100a, and the binding's argument
marshalling module with the host compiler."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import warnings

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libshotkv.so")
SOURCES = ["shotkv_api.cu"]
MARSHAL_SOURCE = os.path.join(CSRC, "marshal.cpp")
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC,-fvisibility=hidden", "--expt-relaxed-constexpr",
    "-cudart", "shared", "-shared",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _stale(target: str, sources: list) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in sources + [os.path.join(PKG_DIR, "..", "include", "shotkv.h")])


def _run(cmd: list, what: str) -> subprocess.CompletedProcess:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError(f"{cmd[0]} failed building {what}")
    return res


def marshal_path() -> str:
    """Where the marshalling module for this Python and this torch lies.  It is compiled against the layout
    of their objects, so both are part of its name and one built for others is never loaded."""
    import sysconfig

    import torch
    return os.path.join(PKG_DIR, f"_marshal.torch-{torch.__version__}{sysconfig.get_config_var('EXT_SUFFIX')}")


def build_marshal(force: bool = False) -> str:
    """Compile the marshalling module next to this file, against the installed torch; returns its path."""
    path = marshal_path()
    if not force and not _stale(path, [MARSHAL_SOURCE]):
        return path
    import sysconfig

    import torch
    root = os.path.join(os.path.dirname(torch.__file__), "")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(_nvcc()) or _nvcc()))), "include")
    include = [root + "include", root + "include/torch/csrc/api/include", cuda, sysconfig.get_paths()["include"]]
    _run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
          f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *(x for i in include for x in ("-isystem", i)),
          MARSHAL_SOURCE, "-o", path, f"-L{root}lib", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"],
         "the marshalling module")
    return path


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile the CUDA sources into `libshotkv.so` next to this file; returns its path.  The marshalling
    module is built after it where that is possible: without it the binding goes through ctypes."""
    path = _build_cuda(force, verbose)
    try:
        build_marshal(force)
    except (ImportError, OSError, RuntimeError) as e:
        warnings.warn(f"the marshalling module was not built ({e}); calls go through ctypes")
    return path


def _build_cuda(force: bool, verbose: bool) -> str:
    if not force and not _stale(LIB_PATH, [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")]):
        return LIB_PATH
    cmd = [_nvcc(), *NVCC_FLAGS]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES]
    res = _run(cmd + ["-o", LIB_PATH], "libshotkv.so")
    if verbose:
        sys.stderr.write(res.stderr)
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force=True, verbose="-v" in sys.argv))
