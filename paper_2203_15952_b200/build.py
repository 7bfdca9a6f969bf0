"""Build the CUDA library (libaqt.so) in-tree with nvcc for sm_100a, and the extension module through
which Python calls its per-layer entry points (_fastcall, under the suffix of the interpreter it is
built for) with the host compiler.

    python -m paper_2203_15952_b200.build [--force]
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_HERE, "csrc")
_INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
LIB_PATH = os.path.join(_HERE, "libaqt.so")
# The module's name carries the interpreter's tag: another interpreter does not find it, and builds its own.
FASTCALL_PATH = os.path.join(_HERE, "_fastcall" + sysconfig.get_config_var("EXT_SUFFIX"))
_FASTCALL_SRC = os.path.join(_CSRC, "host", "fastcall.c")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC"]


def _sources():
    files = [os.path.join(_CSRC, f) for f in sorted(os.listdir(_CSRC)) if f.endswith((".cu", ".cuh"))]
    files.append(os.path.join(_INCLUDE, "aqt.h"))
    return files


def _older(target, sources) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(f) > t for f in sources)


def is_stale() -> bool:
    return _older(LIB_PATH, _sources())


def _build_fastcall(force: bool) -> None:
    if force or _older(FASTCALL_PATH, [_FASTCALL_SRC, os.path.join(_INCLUDE, "aqt.h")]):
        tmp = FASTCALL_PATH + ".tmp.%d" % os.getpid()
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I" + sysconfig.get_paths()["include"],
                               _FASTCALL_SRC, "-o", tmp, "-ldl"])
        os.replace(tmp, FASTCALL_PATH)
    untagged = os.path.join(_HERE, "_fastcall.so")  # of earlier builds: any interpreter would load it
    if os.path.exists(untagged):
        os.remove(untagged)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/aqt_api.cu (one translation unit) into libaqt.so and csrc/host/fastcall.c into
    _fastcall where they are missing or out of date."""
    _build_fastcall(force)
    if force or is_stale():
        nvcc = os.environ.get("NVCC", "nvcc")
        tmp = LIB_PATH + ".tmp.%d" % os.getpid()
        cmd = [nvcc, *NVCC_FLAGS, os.path.join(_CSRC, "aqt_api.cu"), "-o", tmp]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        subprocess.check_call(cmd)
        os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
