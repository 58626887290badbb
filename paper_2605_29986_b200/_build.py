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
# the per-step calls as Python functions, for this interpreter
CALLS_PATH = os.path.join(_HERE, "_calls" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo", "-shared",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
]


def _sources():
    return sorted(os.path.join(_CSRC, f) for f in os.listdir(_CSRC) if f != "calls.c")


def _stale(path: str, sources) -> bool:
    return not os.path.exists(path) or any(os.path.getmtime(p) > os.path.getmtime(path) for p in sources)


def needs_build() -> bool:
    return _stale(LIB_PATH, _sources() + [os.path.join(_INCLUDE, "cfgzip.h")])


def build_calls(force: bool = False) -> bool:
    """Build the native marshalling module if it is missing or older than its source. False where it cannot be built (no C
    compiler, no Python headers): the binding then passes the arguments through ctypes."""
    source = os.path.join(_CSRC, "calls.c")
    if not force and not _stale(CALLS_PATH, [source, os.path.join(_INCLUDE, "cfgzip.h")]):
        return True
    tmp = CALLS_PATH + ".%d.tmp" % os.getpid()
    try:
        subprocess.run([shutil.which("gcc") or "cc", "-O2", "-shared", "-fPIC", "-Wall", "-I", _INCLUDE, "-I",
                        sysconfig.get_paths()["include"], "-o", tmp, source], check=True, capture_output=True)
    except (OSError, subprocess.CalledProcessError):
        if os.path.exists(CALLS_PATH):
            os.remove(CALLS_PATH)  # of an older source
        return False
    os.replace(tmp, CALLS_PATH)
    return True


def build(force: bool = False, verbose: bool = False) -> str:
    """Build ``libcfgzip.so`` (and the marshalling module) next to this file if it is missing or older than the sources."""
    build_calls(force)
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
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
