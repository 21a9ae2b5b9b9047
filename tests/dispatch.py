"""Which kernel takes a call, by the library's own rules: the functions that decide between the tensor-core kernels for large
calls and the others are compiled here from their source."""
import ctypes
import functools
import os
import re
import subprocess
import tempfile

ROOT = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..")
LAUNCH = os.path.join(ROOT, "paper_2601_22347_b200", "csrc", "perq_tile_launch.cuh")
MODES = {("int4", False): 0, ("int4", True): 1, ("mxfp4", True): 2, ("fp4", False): 3, ("int4_asym", False): 4}


@functools.lru_cache(None)
def _rules():
    with open(LAUNCH) as f:
        text = f.read()
    functions = [re.search(r"^bool %s\(.*?^}\n" % name, text, re.S | re.M).group(0) for name in ("tile_is_better", "col_is_better")]
    with tempfile.TemporaryDirectory() as d:
        src, lib = os.path.join(d, "rules.cpp"), os.path.join(d, "rules.so")
        with open(src, "w") as f:
            f.write("namespace perq { enum { ROW_TOKEN = 0, ROW_GROUP = 1, ROW_MX = 2, ROW_FP4 = 3, ROW_ASYM = 4, SEG_ELEMS = 1024 }; }\n"
                    + "\n".join(functions)
                    + '\nextern "C" int tile_takes(int m, int d, int b, long long p) { return tile_is_better(m, d, b, p); }'
                      '\nextern "C" int column_takes(int m, int d, long long p) { return col_is_better(m, d, p); }\n')
        subprocess.run(["g++", "-shared", "-fPIC", "-o", lib, src], check=True)
        return ctypes.CDLL(lib)


def kernel_of(fmt, group, T, d, b, perm=False):
    """"tile", "column" or "other"."""
    ranges = fmt == "mxfp4" or (fmt == "int4" and group not in (0, d))
    if perm or b & (b - 1) or d % 128 or (fmt == "int4" and group not in (0, 128, d)):
        return "other"
    mode, pieces = MODES[(fmt, ranges)], ctypes.c_longlong(T * (d // 128))
    if b == d and b > 128:
        return "column" if d in (2048, 4096) and not ranges and _rules().column_takes(mode, d, pieces) else "other"
    if fmt == "int4_asym" or not 16 <= b <= 128 or (not ranges and not 1 <= 128 // (d // 128) <= 32):
        return "other"
    return "tile" if _rules().tile_takes(mode, d, b, pieces) else "other"


def most_rows(kernel, fmt, group, d, b, at_most):
    """The largest number of rows up to at_most for which the call is the kernel's."""
    T = at_most
    while T > 0 and kernel_of(fmt, group, T, d, b) != kernel:
        T = T * 15 // 16 if T > 4096 else T - 1
    return T
