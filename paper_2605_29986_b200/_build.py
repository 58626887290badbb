"""Compile the CUDA library in-tree with nvcc for sm_100a."""
from __future__ import annotations

import os
import shutil
import subprocess
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_HERE, "csrc")
_INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
LIB_PATH = os.path.join(_HERE, "libcfgzip.so")
CALLS_PATH = os.path.join(_HERE, "_calls.so")  # the per-step calls as Python functions

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo", "-shared",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
]


def _sources():
    return sorted(os.path.join(_CSRC, f) for f in os.listdir(_CSRC))


def needs_build() -> bool:
    if not (os.path.exists(LIB_PATH) and os.path.exists(CALLS_PATH)):
        return True
    built = min(os.path.getmtime(LIB_PATH), os.path.getmtime(CALLS_PATH))
    deps = _sources() + [os.path.join(_INCLUDE, "cfgzip.h")]
    return any(os.path.getmtime(p) > built for p in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Build ``libcfgzip.so`` and ``_calls.so`` next to this file if one is missing or older than the sources."""
    if not force and not needs_build():
        return LIB_PATH
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        raise RuntimeError("nvcc not found: the CFGzip CUDA library cannot be built")
    tmp = LIB_PATH + ".%d.tmp" % os.getpid()
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + [
        "-I", _INCLUDE, "-I", _CSRC, "-o", tmp, os.path.join(_CSRC, "cfgzip_api.cu"),
        os.path.join(_CSRC, "cfgzip_offline.cu")]
    subprocess.check_call(cmd)
    tmp_calls = CALLS_PATH + ".%d.tmp" % os.getpid()
    subprocess.check_call([shutil.which("gcc") or "cc", "-O2", "-shared", "-fPIC", "-Wall", "-I", _INCLUDE, "-I",
                           sysconfig.get_paths()["include"], "-o", tmp_calls, os.path.join(_CSRC, "calls.c")])
    os.replace(tmp, LIB_PATH)
    os.replace(tmp_calls, CALLS_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
