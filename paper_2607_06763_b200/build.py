"""Builds ``libgdn_tree.so`` (``csrc/*.cu``, nvcc for sm_100a) and the extension module ``_gdn_call`` (``csrc/gdn_call.c``, the
binding's argument marshalling) in-tree; no GPU needed to compile."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libgdn_tree.so")
CALL_SRC = os.path.join(CSRC, "gdn_call.c")
CALL_LIB = os.path.join(_HERE, "_gdn_call" + sysconfig.get_config_var("EXT_SUFFIX"))   # one for each Python's ABI
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "--shared", "-I", os.path.join(_ROOT, "include"), "-I", CSRC,
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(_ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build_call_module(force: bool = False) -> str:
    if force or not os.path.exists(CALL_LIB) or os.path.getmtime(CALL_SRC) > os.path.getmtime(CALL_LIB):
        tmp = CALL_LIB + f".{os.getpid()}.tmp"
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"],
                               "-o", tmp, CALL_SRC])
        os.replace(tmp, CALL_LIB)
    return CALL_LIB


def build_library(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    build_call_module(force)
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc] + NVCC_FLAGS + list(extra_flags) + ["-o", tmp] + sources()
    if verbose:
        print(" ".join(cmd), flush=True)
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    flags = ["-Xptxas", "-v"] if "-v" in sys.argv else []
    print(build_library(force=True, verbose=True, extra_flags=flags))
