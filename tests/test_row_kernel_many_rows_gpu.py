"""Parity of the row kernels with the oracle on calls in which every CTA serves at least five or six rows: the ring of two stages
is refilled (a refilled stage is read from a CTA's third row on), the stage parities flip, the lists and reduction words
of one row are those of the next.  The GPU runs the whole call, the oracle rows of every sixth of it.

A CTA's rows are blockIdx.x, blockIdx.x + grid, ...: a grid of at most 148 SMs times the rows that an SM's warps hold at
a time (ROW_SM_WARPS and ROW64_SM_WARPS of perq_row.cuh, a warp per 1024 channels or more).  Every case asserts the
rows from that bound, and that the call is not the column kernel's, so a change of the grid or the dispatch does not hollow
the tests out unnoticed.
"""
import numpy as np
import pytest
import torch

from paper_2601_22347_b200 import inputs

from dispatch import kernel_of
from parity import compare_quantized

pytestmark = pytest.mark.gpu

FMT = {"int4": 0, "mxfp4": 1, "fp4": 3, "int4_asym": 4}
SMS, SM_WARPS, SM_WARPS_64 = 148, 20, 16
MIN_ROWS = 6


@pytest.fixture(scope="module")
def B():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_22347_b200 import binding, build
    build.build()
    binding.load()
    return binding


@pytest.fixture(autouse=True)
def clean_error_word(B):
    B.perq_device_error_clear()
    yield
    assert B.perq_device_error() == 0


def rows_in_flight(d, fmt, group, b):
    fp64 = fmt == "int4" and 0 < group <= b and b >= 256 and b & (b - 1) == 0
    return SMS * max(1, (SM_WARPS_64 if fp64 else SM_WARPS) // -(-d // 1024))


@pytest.mark.parametrize("fmt,group", [("int4", 0), ("int4", 128), ("mxfp4", 32), ("fp4", 0), ("int4_asym", 0)])
@pytest.mark.parametrize("d,b,perm", [(14336, 14336, False), (14336, 14336, True), (6144, 6144, False), (3072, 3072, True),
                                      (16384, 16384, False), (8192, 8192, True), (4096, 4096, False), (4096, 2048, True),
                                      (2048, 2048, False), (1152, 128, True), (3072, 1024, True)])
def test_many_rows_per_cta(B, oracle, d, b, perm, fmt, group):
    flight = rows_in_flight(d, fmt, group, b)
    rows_each = MIN_ROWS
    if not perm and kernel_of(fmt, group, MIN_ROWS * flight + 3, d, b) != "other":
        rows_each -= 1                                        # (more rows are the column kernel's)
    T = rows_each * flight + 3
    assert T // flight >= rows_each and kernel_of(fmt, group, T, d, b, perm) == "other"
    base = inputs.laplace_outliers(192, d, max(1, d // 2048), 100.0, 20000 + d + b)[0]
    base[5] = 0
    idx = (np.arange(T) + np.arange(T) // 192) % 192         # a base row meets different CTAs and stages
    x = torch.from_numpy(base.view(np.int16)).cuda()[torch.from_numpy(idx).cuda()].view(torch.bfloat16)
    p = inputs.random_perm(d, 20001) if perm else None
    codes, scales = B.perq_rotate_quantize(x, None if p is None else torch.from_numpy(p).cuda(), b, FMT[fmt], group)
    torch.cuda.synchronize()
    rng = np.random.default_rng(20002)
    rows = np.unique(np.r_[0, T - 1, (np.arange(rows_each)[:, None] * flight + rng.integers(0, flight, (rows_each, 3))).ravel()])
    at = torch.from_numpy(rows).cuda()
    ora = oracle.rotate_quantize(base[idx[rows]], p, b, FMT[fmt], group, want_pre=True)
    compare_quantized(fmt, codes[at].cpu().numpy(), scales[at].cpu().numpy(), ora)
    # every repetition of a base row gives the same bytes
    first = torch.empty(192, dtype=torch.int64, device="cuda")
    idx_t = torch.from_numpy(idx).cuda()
    first[idx_t.flip(0)] = torch.arange(T - 1, -1, -1, device="cuda")
    assert torch.equal(codes, codes[first[idx_t]]) and torch.equal(scales, scales[first[idx_t]])
