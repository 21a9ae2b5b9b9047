"""Builds the CUDA library in-tree: paper_2601_22347_b200/libperq.so (sm_100a only)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
_CSRC = os.path.join(_PKG, "csrc")
LIB_PATH = os.path.join(_PKG, "libperq.so")
CALL_PATH = os.path.join(_PKG, "_perq_call" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))      # (another interpreter has another name)


def _sources():
    return sorted(os.path.join(_CSRC, f) for f in os.listdir(_CSRC) if f.endswith(".cu"))


def _deps():
    deps = [os.path.join(_CSRC, f) for f in os.listdir(_CSRC) if not f.endswith(".c")]
    deps.append(os.path.join(_ROOT, "include", "perq.h"))
    return deps


def needs_build() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    return any(os.path.getmtime(p) > t for p in _deps())


def build_call(force: bool = False) -> bool:
    """Compile the interpreter's direct entry to the two calls of the online path.  False where there are no headers for it or
    no compiler: these calls then go through ctypes, and an older file is taken away."""
    src, include = os.path.join(_CSRC, "perq_call.c"), sysconfig.get_paths()["include"]
    if not force and os.path.exists(CALL_PATH) and os.path.getmtime(src) <= os.path.getmtime(CALL_PATH):
        return True
    why, cc = "no Python.h", os.environ.get("CC", "gcc")
    if os.path.exists(os.path.join(include, "Python.h")):
        tmp = CALL_PATH + ".tmp.%d" % os.getpid()
        try:
            out = subprocess.run([cc, "-O2", "-shared", "-fPIC", "-I", include, "-o", tmp, src],
                                 stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
            if out.returncode == 0:
                os.replace(tmp, CALL_PATH)
                return True
            why = "%s failed\n%s" % (cc, out.stdout)
        except OSError as error:
            why = "%s: %s" % (cc, error)
    if os.path.exists(CALL_PATH):
        os.remove(CALL_PATH)
    sys.stderr.write("perq: without the interpreter's own entry, calls go through ctypes (%s)\n" % why)
    return False


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into one shared library for sm_100a, and the interpreter's entry to it."""
    build_call(force)
    if not force and not needs_build():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB_PATH + ".tmp.%d" % os.getpid()
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(_ROOT, "include"), "-I", _CSRC,
           "-o", tmp] + _sources()
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    out = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if out.returncode != 0:
        sys.stderr.write(out.stdout)
        raise RuntimeError("nvcc failed building libperq.so")
    if verbose:
        print(out.stdout)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB_PATH)
