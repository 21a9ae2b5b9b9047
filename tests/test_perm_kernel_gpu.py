"""Parity of the kernel for many permuted rows with the oracle, at the edges of its sets, boxes and parts: widths of 5 pieces up to the
largest it takes (86, four stages of its ring), rows that end inside a set, sets that fill rounds of the grid exactly, leave a last round that is split
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
from test_row_kernel_edges_gpu import _cancelling_rows, _rows_at_the_upper_end, _zero_quarter_rows, through
from test_tile_kernel_gpu import BASE, FMT, B, base_rows, clean_error_word, flat_rows  # noqa: F401

pytestmark = pytest.mark.gpu


def takes(d, T):
    """The launcher's rule, and its kernel's demand for four stages of the ring."""
    with open(LAUNCH) as f:
        text = f.read()
    rule = re.search(r"^bool perm_is_better\(.*$", text, re.M).group(0)
    stages = re.search(r"if \((lay\.stages < \d+)\) return -1;", text[text.index("int try_launch_perm("):]).group(1)
    with open(os.path.join(os.path.dirname(LAUNCH), "perq_perm.cuh")) as f:
        text = f.read()
    constants = "".join(m + "\n" for m in re.findall(r"^constexpr \w+ PERM_\w+ = .*$", text, re.M))
    layout = re.search(r"^struct PermLayout \{.*?^\};\n", text, re.S | re.M).group(0)
    with tempfile.TemporaryDirectory() as tmp:
        src, lib = os.path.join(tmp, "rule.cpp"), os.path.join(tmp, "rule.so")
        with open(src, "w") as f:
            f.write("#include <cstdint>\n#define __host__\n#define __device__\nnamespace perq { enum { SEG_ELEMS = 1024 };\n" + constants + layout + "}\n" + rule +
                    '\nextern "C" int takes(int d, long long T) { const perq::PermLayout lay(d, (d + perq::PERM_BOX - 1) / perq::PERM_BOX, 227 * 1024);'
                    " return perm_is_better(d, T) && !(%s); }" % stages)
        subprocess.run(["g++", "-shared", "-fPIC", "-o", lib, src], check=True)
        return ctypes.CDLL(lib).takes(d, ctypes.c_longlong(T))


def check(B, oracle, T, d, b, fmt, group, seed, make, gathered=False):
    """gathered: make gives the rows as they are after the permutation."""
    assert takes(d, T) and not takes(d, 64) and not takes(1024, T)
    base = make(d, seed)
    rng = np.random.default_rng(seed)
    perm = rng.permutation(d).astype(np.int32)
    if gathered:
        base = through(base, perm)
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


@pytest.mark.parametrize("fmt,group", [("mxfp4", 32), ("int4", 128)])
@pytest.mark.parametrize("d", [10368, 11008])
def test_widest_rows(B, oracle, fmt, group, d):              # noqa: F811
    """Five and four stages of the ring, 21 and 22 boxes; wider ones are not the kernel's."""
    assert not takes(11136, 600) and not takes(14208, 600)
    for b in (16, 32, 64, 128):
        check(B, oracle, 1190 if b == 32 else 600, d, b, fmt, group, 7300 + b + d, base_rows)


@pytest.mark.parametrize("b", [64, 128])
@pytest.mark.parametrize("T,d", [(600, 1152), (592, 4736)])
def test_groups_that_cancel(B, oracle, b, T, d):             # noqa: F811
    """(In blocks of 128 the exact zeros are noise in fp32, in blocks of 64 they are halves of groups that are not.)"""
    def rows(d, seed):
        bits = _zero_quarter_rows(BASE, d, b, seed)
        assert b == 64 or (oracle.rotate_quantize(bits, None, b, FMT["mxfp4"], 32)["scales"] == 0).mean() == 0.25
        return bits
    check(B, oracle, T, d, b, "mxfp4", 32, 7400 + b, rows, gathered=True)


@pytest.mark.parametrize("log2_ratio", [18, 22, 23])
@pytest.mark.parametrize("fmt,group", [("mxfp4", 32), ("int4", 128)])
def test_groups_far_below_their_block(B, oracle, fmt, group, log2_ratio):      # noqa: F811
    check(B, oracle, 600, 640, 128, fmt, group, 7500 + log2_ratio, lambda d, seed: _cancelling_rows(BASE, d, 128, log2_ratio, seed), gathered=True)


@pytest.mark.parametrize("fmt,group", [("mxfp4", 32), ("int4", 128)])
@pytest.mark.parametrize("b", [16, 32, 64, 128])
def test_rows_at_the_upper_end_of_the_range(B, oracle, fmt, group, b):         # noqa: F811
    check(B, oracle, 600, 1152, b, fmt, group, 7600 + b, lambda d, seed: _rows_at_the_upper_end(oracle, BASE, d, b, seed), gathered=True)
