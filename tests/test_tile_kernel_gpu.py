"""Parity of the tile and column kernels with the oracle: calls large enough to be theirs, with ragged numbers of rows, in which
every CTA serves several tiles (ring stages, accumulators and note slots are used again and change their phase).  The GPU
runs the whole call, the oracle the base rows it is made of; every repetition of a base row has to give the same bytes.

The base rows hold what each rule of these kernels meets: rows with outliers, rows without, zeros, one nonzero (every
output of its block ties), small integers (true rounding ties), a row near the lower end of the range that the formats
take and one near the upper end (the ends themselves: test_tensor_core_bounds.py).  Every case asserts that the call is the
kernel's.
"""
import numpy as np
import pytest
import torch

from paper_2601_22347_b200 import inputs

from dispatch import kernel_of
from parity import compare_quantized

pytestmark = pytest.mark.gpu

FMT = {"int4": 0, "mxfp4": 1, "fp4": 3, "int4_asym": 4}
BASE = 160


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


def bf16(v):
    return (np.ascontiguousarray(v, dtype=np.float32).view(np.uint32) >> 16).astype(np.uint16)


def base_rows(d, seed):
    rng = np.random.default_rng(seed)
    x = inputs.laplace_outliers(BASE, d, max(1, d // 1024), 200.0, seed)[0]
    x[40:80] = inputs.gaussian_outliers(40, d, 0, 1.0, seed + 1)[0]
    x[80:120] = inputs.student_t_outliers(40, d, 3.0, max(2, d // 256), 100.0, seed + 2)[0]
    x[7] = 0
    x[8] = bf16(np.eye(1, d, d // 3) * 3.0)                                    # one nonzero
    x[9] = bf16(rng.integers(-3, 4, d))                                        # small integers
    x[10] = bf16(np.where(rng.random(d) < 8.0 / d, rng.integers(1, 9, d), 0))  # a few of them
    x[11] = bf16(np.ones(d))
    x[12] = bf16(rng.standard_normal(d) * 2.0 ** -116)
    x[13] = bf16(rng.standard_normal(d) * 2.0 ** 116)
    x[14, d // 2:] = 0
    return x


def flat_rows(d, seed):
    rng = np.random.default_rng(seed)
    x = np.empty((BASE, d), np.uint16)
    for i in range(BASE):
        v = (np.ones(d), rng.integers(-3, 4, d), rng.choice([-1.0, 1.0], d), np.where(np.arange(d) % 128 == i % 128, 3.0, 0),
             np.repeat(2.0 ** rng.integers(-3, 4, d // 128), 128))[i % 5].astype(np.float64)
        if i % 2:                                                # pieces whose fp32 outputs are not exact
            v[(i % 128)::(128 if i % 4 == 1 else 384)] = 2.0 ** -30 * (i % 7 + 1)
        x[i] = bf16(v)
    return x


def check(B, oracle, T, d, b, fmt, group, seed, offset=0, make=base_rows):
    assert kernel_of(fmt, group, T, d, b) == ("column" if b > 128 else "tile")
    base = make(d, seed)
    idx = (np.arange(T) + np.arange(T) // BASE) % BASE           # a base row meets different CTAs, warps and stages
    idx_t = torch.from_numpy(idx).cuda()
    x = torch.from_numpy(base.view(np.int16)).cuda()[idx_t].view(torch.bfloat16)
    codes, scales = B.alloc_outputs(T, d, FMT[fmt], group, "cuda")
    if offset:                                                   # codes that are 16-byte but not 32-byte aligned
        codes = torch.zeros(T * d // 2 + offset, dtype=torch.uint8, device="cuda")[offset:].view(T, d // 2)
        assert codes.data_ptr() % 32 == 16
    B.perq_rotate_quantize(x, None, b, FMT[fmt], group, codes, scales)
    torch.cuda.synchronize()
    first = torch.empty(BASE, dtype=torch.int64, device="cuda")
    first[idx_t.flip(0)] = torch.arange(T - 1, -1, -1, device="cuda")
    assert torch.equal(codes, codes[first[idx_t]]) and torch.equal(scales, scales[first[idx_t]])
    rows = np.r_[np.arange(0, 16), np.random.default_rng(seed).choice(np.arange(16, BASE), 16 if b <= 128 else 6, replace=False)]
    at = first[torch.from_numpy(rows).cuda()]
    ora = oracle.rotate_quantize(base[rows], None, b, FMT[fmt], group, want_pre=True)
    compare_quantized(fmt, codes[at].cpu().numpy(), scales[at].cpu().numpy(), ora)


def rows_of(T, b, fmt, group):
    """Blocks of 128 with a scale per token are the kernel's from four times as many rows on."""
    return 4 * T + 1 if b == 128 and group == 0 else T


@pytest.mark.parametrize("fmt,group", [("int4", 0), ("int4", 128), ("mxfp4", 32), ("fp4", 0)])
@pytest.mark.parametrize("b", [16, 32, 64, 128])
def test_ragged_widths(B, oracle, b, fmt, group):
    # pieces per row: 6 (21 rows a tile), 76 and 111 (one), 9 (14, 126 of 128 lanes)
    for d, T in ((768, 6001), (9728, 691), (14208, 433), (1152, 5003)):
        check(B, oracle, rows_of(T, b, fmt, group), d, b, fmt, group, 30000 + d + b)


@pytest.mark.parametrize("d,fmt,group,b", [(d, "fp4", 0, b) for d in (512, 2048) for b in (16, 32, 64)] + [(512, "fp4", 0, 128)] +
                         [(512, "int4", 0, b) for b in (16, 32, 64, 128)])
def test_rows_inside_a_warp(B, oracle, d, fmt, group, b):
    """4 and 16 pieces per row: rows meet by shuffles, without a barrier, and settle by warps (512: all 32 rows of a tile)."""
    for make in (base_rows, flat_rows):
        check(B, oracle, rows_of(8195, b, fmt, group), d, b, fmt, group, 36000 + d + b, make=make)


@pytest.mark.parametrize("d,fmt,group,b", [(d, f, g, b) for d in (4096, 8192, 14336)
                                           for f, g, b in (("int4", 0, 64), ("int4", 128, 16), ("int4", 128, 128), ("mxfp4", 32, 32),
                                                           ("mxfp4", 32, 64), ("fp4", 0, 16), ("fp4", 0, 64))] +
                         [(14336, "int4", 0, 128), (14336, "fp4", 0, 128)] +
                         # 128, 24 and 48 pieces per row: one row, five and two of a tile
                         [(16384, "int4", 0, 64), (16384, "fp4", 0, 16), (3072, "int4", 0, 64), (3072, "fp4", 0, 32), (6144, "fp4", 0, 64),
                          (1024, "int4", 128, 64), (32768, "mxfp4", 32, 64)])
def test_whole_segments(B, oracle, d, fmt, group, b):
    check(B, oracle, (25 if b == 128 else 17) * 2 ** 20 // d, d, b, fmt, group, 31000 + d + b, offset=16)


@pytest.mark.parametrize("fmt", ["int4", "fp4", "int4_asym"])
@pytest.mark.parametrize("d,T", [(4096, 8195), (2048, 16389)])
def test_whole_row_rotations(B, oracle, d, T, fmt):
    check(B, oracle, T, d, d, fmt, 0, 32000 + d)


@pytest.mark.parametrize("fmt,group", [("int4", 0), ("int4", 128), ("mxfp4", 32), ("fp4", 0)])
@pytest.mark.parametrize("d,T", [(1536, 3001), (9728, 691), (4096, 4096)])
def test_flat_rows(B, oracle, d, T, fmt, group):
    # nearly every piece has more candidates or ties than are noted: lanes settle them, with exact fp32 outputs and without
    for b in (16, 128) if d % 1024 else {"int4": (64,) if group == 0 else (16, 64), "mxfp4": (32, 64), "fp4": (16, 64)}[fmt]:
        check(B, oracle, rows_of(T, b, fmt, group), d, b, fmt, group, 33000 + d + b, make=flat_rows)


@pytest.mark.parametrize("fmt", ["int4", "fp4", "int4_asym"])
@pytest.mark.parametrize("d,T", [(4096, 8195), (2048, 16389)])
def test_flat_whole_rows(B, oracle, d, T, fmt):
    check(B, oracle, T, d, d, fmt, 0, 33500 + d, make=flat_rows)


def zero_blocks(d, seed):
    """Blocks of 16 zeros beside blocks that are not, and channels of zeros at the end."""
    x = base_rows(d, seed)
    x[:, 16::64] = 0
    x[:, 32:48] = 0
    x[:, d - 80:] = 0
    return x


def pass_us(B, make, T, d, b, fmt, group, seed):
    x = torch.from_numpy(make(d, seed).view(np.int16)).cuda()[20:120].repeat(-(-T // 100), 1)[:T].view(torch.bfloat16).contiguous()
    codes, scales = B.alloc_outputs(T, d, FMT[fmt], group, "cuda")
    best = float("inf")
    for _ in range(5):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        e[0].record()
        for _ in range(10):
            B.perq_rotate_quantize(x, None, b, FMT[fmt], group, codes, scales)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]) * 100)
    return best


@pytest.mark.parametrize("fmt,group,d,T", [("fp4", 0, 4096, 4096), ("fp4", 0, 9728, 2048), ("mxfp4", 32, 9728, 2048)])
def test_blocks_of_zeros_beside_others(B, oracle, fmt, group, d, T):
    """The signs of their outputs are not in doubt: a call with some takes no longer than one without."""
    check(B, oracle, T, d, 16, fmt, group, 34000 + d, make=zero_blocks)
    dense, zeros = pass_us(B, base_rows, T, d, 16, fmt, group, 34001), pass_us(B, zero_blocks, T, d, 16, fmt, group, 34001)
    print("%s %d x %d: dense %.1f us, blocks of zeros %.1f us" % (fmt, T, d, dense, zeros))
    assert zeros < 2 * dense


def few_bits(d, seed):
    """Integers, and values of four significant bits: with b = 16 and 64 many outputs lie on E2M1 midpoints."""
    rng = np.random.default_rng(seed)
    x = rng.integers(-3, 4, (BASE, d)).astype(np.float64)
    x[BASE // 2:] = rng.integers(-15, 16, (BASE - BASE // 2, d)) * np.exp2(rng.integers(-3, 2, (BASE - BASE // 2, d)))
    return bf16(x)


@pytest.mark.parametrize("b,d,T", [(16, 9728, 2048), (64, 9728, 2048), (64, 4096, 4096)])
def test_many_midpoints(B, oracle, b, d, T):
    check(B, oracle, T, d, b, "mxfp4", 32, 35000 + b, make=few_bits)
    dense, ties = pass_us(B, base_rows, T, d, b, "mxfp4", 32, 35001), pass_us(B, few_bits, T, d, b, "mxfp4", 32, 35001)
    print("b = %d, %d x %d: dense %.1f us, midpoints %.1f us" % (b, T, d, dense, ties))
    assert ties < 18 * dense
