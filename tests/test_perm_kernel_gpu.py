"""Parity of the kernel for many permuted rows with the oracle, at the edges of its sets, boxes and parts: widths of 5 pieces up to the
largest it takes, rows that end inside a set, sets that fill rounds of the grid exactly, leave a last round that is split
among CTAs, or are fewer than the SMs; base rows and flat rows of the tile kernel's tests.  The GPU runs the whole call, the
oracle the base rows it is made of; every repetition of a base row has to give the same bytes."""
import ctypes
import os
import re
import subprocess
import tempfile

import numpy as np
import pytest
import torch

from dispatch import LAUNCH
from parity import compare_quantized
from test_tile_kernel_gpu import BASE, FMT, B, base_rows, clean_error_word, flat_rows  # noqa: F401

pytestmark = pytest.mark.gpu


def takes(d, T):
    with open(LAUNCH) as f:
        rule = re.search(r"^bool perm_is_better\(.*$", f.read(), re.M).group(0)
    with tempfile.TemporaryDirectory() as tmp:
        src, lib = os.path.join(tmp, "rule.cpp"), os.path.join(tmp, "rule.so")
        with open(src, "w") as f:
            f.write("namespace perq { enum { SEG_ELEMS = 1024 }; }\n" + rule +
                    '\nextern "C" int takes(int d, long long T) { return perm_is_better(d, T); }')
        subprocess.run(["g++", "-shared", "-fPIC", "-o", lib, src], check=True)
        return ctypes.CDLL(lib).takes(d, ctypes.c_longlong(T))


def check(B, oracle, T, d, b, fmt, group, seed, make):
    assert takes(d, T) and not takes(d, 64) and not takes(1024, T)
    base = make(d, seed)
    rng = np.random.default_rng(seed)
    perm = rng.permutation(d).astype(np.int32)
    idx = (np.arange(T) + np.arange(T) // BASE) % BASE           # a base row meets different CTAs and places in a set
    idx_t = torch.from_numpy(idx).cuda()
    x = torch.from_numpy(base.view(np.int16)).cuda()[idx_t].view(torch.bfloat16)
    codes, scales = B.alloc_outputs(T, d, FMT[fmt], group, "cuda")
    codes.fill_(0x5a)
    torch.cuda.synchronize()
    B.perq_rotate_quantize(x, torch.from_numpy(perm).cuda(), b, FMT[fmt], group, codes, scales)
    torch.cuda.synchronize()
    first = torch.arange(BASE, device="cuda")
    for out in (codes, scales):
        out = out.reshape(T, -1).contiguous().view(torch.uint8)
        assert torch.equal(out, out[first][idx_t])
    ora = oracle.rotate_quantize(base, perm, b, FMT[fmt], group, want_pre=True)
    rep = compare_quantized(fmt, codes[:BASE].cpu().numpy(), scales[:BASE].cpu().numpy(), ora)
    assert rep["code_mismatch_exempt"] == 0


@pytest.mark.parametrize("fmt,group", [("mxfp4", 32), ("int4", 128)])
@pytest.mark.parametrize("b", [16, 32, 64, 128])
@pytest.mark.parametrize("T,d", [(592, 640), (1184, 1152), (1191, 4736), (2377, 3200), (600, 10112), (1500, 9728)])
def test_edges(B, oracle, fmt, group, b, T, d):              # noqa: F811
    check(B, oracle, T, d, b, fmt, group, 7100 + b + d, base_rows)


@pytest.mark.parametrize("fmt,group", [("mxfp4", 32), ("int4", 128)])
@pytest.mark.parametrize("b", [16, 32, 64, 128])
def test_flat_rows(B, oracle, fmt, group, b):                # noqa: F811
    check(B, oracle, 603, 1152, b, fmt, group, 7200 + b, flat_rows)
