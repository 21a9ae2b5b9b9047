"""Error bounds of the kernels that rotate by chained tensor-core steps (tile and column kernel), against the oracle, on rows
whose fp32 outputs are as wrong as that arithmetic allows: a maximum, and a side of a rounding boundary, that fp32 hides."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2601_22347_b200 import inputs

from dispatch import LAUNCH, kernel_of
from mma_rows import (hadamard, chained_contraction, hidden_in_every_piece, hidden_maximum, hidden_side, hidden_step, losing_chunks, one_step_and_stages,
                      outputs, to_bf16)
from parity import compare_quantized

FMT = {"int4": 0, "mxfp4": 1, "fp4": 3, "int4_asym": 4}


@pytest.fixture(scope="module")
def B():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_22347_b200 import binding, build
    build.build()
    binding.load()
    binding.perq_device_error_clear()
    yield binding
    assert binding.perq_device_error() == 0


def bits(x):
    x = np.asarray(x, np.float32)
    assert np.array_equal(x, to_bf16(x))
    return inputs.f32_to_bf16_bits(x)


def whole_rows(d, seed):
    """Rows with one hidden output, moved to other places and magnitudes: an input's sign by a row of the Hadamard matrix
    moves all outputs, a shift of the inputs by XOR changes only their signs."""
    c = d // 128
    kinds = [hidden_maximum(d, 128, 110), hidden_maximum(d, 128, 95), hidden_in_every_piece(d, 94 * c), hidden_side(d, 128, 6.5 / 7, 10),
             hidden_side(d, 128, 5 / 7, 10), hidden_step(d, 128, 12, 10), hidden_step(d, 128, 11, 6)]
    rng, k = np.random.default_rng(seed), np.arange(d)
    rows = []
    for i in range(12):
        for x in kinds:
            m, s = (0, 0) if i == 0 else (int(rng.integers(d)), int(rng.integers(d)) & ~15)
            signs = 1.0 - 2.0 * (np.array([bin(v).count("1") for v in (k & m)]) & 1)
            rows.append((x * signs)[k ^ s] * 2.0 ** int(rng.integers(-20, 20)))
    return bits(np.array(rows))


def block_rows(d, b, seed):
    """Rows of one block that hides an output and others, at a quarter of its size and less, that do."""
    gap = 124 if b == 128 else 62
    kinds = [hidden_maximum(b, b, gap), hidden_maximum(b, b, gap - 8), hidden_side(b, b, 6.5 / 7, 10), hidden_side(b, b, 5 / 7, 10),
             hidden_side(b, b, 3.5 / 7, 10), hidden_step(b, b, 12, 10)]
    rng, k = np.random.default_rng(seed), np.arange(b)
    x = np.zeros((96, d // b, b))
    for i in range(len(x)):
        top = rng.integers(d // b)
        for j in range(d // b):
            signs = 1.0 - 2.0 * (np.array([bin(v).count("1") for v in (k & int(rng.integers(b)))]) & 1)
            size = 0 if j == top else int(rng.integers(-30, -2))
            x[i, j] = (kinds[(i + j) % 6 if j != top else i % 6] * signs)[k ^ (int(rng.integers(b)) & ~15)] * 2.0 ** size
        x[i] *= 2.0 ** int(rng.integers(-20, 20))
    return bits(x.reshape(len(x), d))


def run(B, oracle, base, T, b, fmt, group):
    """T rows made of the base rows, each of which is compared, and the same bytes at every repetition; in the kernels that
    rotate by chained steps."""
    n = len(base)
    assert kernel_of(fmt, group, T, base.shape[1], b) == ("column" if b > 128 else "tile")
    idx = (np.arange(T) + np.arange(T) // n) % n
    idx_t = torch.from_numpy(idx).cuda()
    x = torch.from_numpy(base.view(np.int16)).cuda()[idx_t].view(torch.bfloat16)
    codes, scales = B.perq_rotate_quantize(x, None, b, FMT[fmt], group)
    torch.cuda.synchronize()
    first = torch.empty(n, dtype=torch.int64, device="cuda")
    first[idx_t.flip(0)] = torch.arange(T - 1, -1, -1, device="cuda")
    assert torch.equal(codes, codes[first[idx_t]]) and torch.equal(scales, scales[first[idx_t]])
    ora = oracle.rotate_quantize(base, None, b, FMT[fmt], group, want_pre=True)
    compare_quantized(fmt, codes[first].cpu().numpy(), scales[first].cpu().numpy(), ora)


def test_rows_hide_what_they_say():
    """The model's fp32 outputs of the rows above: another maximum, another side."""
    h = hadamard(128)
    for d in (2048, 4096):
        for x, wrong in ((hidden_maximum(d, 128, 110), 46), (hidden_in_every_piece(d, 94 * d // 128), 90)):
            v = chained_contraction(x.reshape(-1, 128), h)
            u32 = hadamard(d // 128) @ v                       # (the later stages without rounding)
            top = np.abs(outputs(x)).max()
            at = np.unravel_index(np.abs(outputs(x)).argmax(), u32.shape)
            assert np.abs(u32).max() - abs(u32[at]) > (wrong - 1) * 2.0 ** -24 * top
        x = hidden_side(d, 128, 6.5 / 7, 10)
        v = (hadamard(d // 128) @ chained_contraction(x.reshape(-1, 128), h)).ravel()
        u = outputs(x)
        assert u[1] > 6.5 / 7 * u.max() and v[1] < 6.5 / 7 * v.max() * (1 - 30 * 2.0 ** -24)


def lost_at_most(x):
    """The column kernel's bound of what a piece of 128 loses, from its inputs."""
    e = np.floor(np.log2(np.abs(x).sum(1) * 1.001))
    n = ((x != 0) & (np.abs(x) < np.exp2(e - 16)[:, None])).sum(1)
    return (n + 5 * np.minimum(n, 8)) * np.exp2(e - 25)


@pytest.mark.parametrize("kind", ["gauss", "binades", "few", "coherent", "decreasing"])
def test_what_the_contraction_loses(kind):
    """No output of the model is further off than the bound (0.17 to 0.63 of it)."""
    rng, h, worst = np.random.default_rng(41000), hadamard(128), 0.0
    for it in range(6):
        x = rng.standard_normal((64, 128))
        if kind == "binades":
            x *= np.exp2(-rng.integers(0, 40, x.shape))
        elif kind == "few":
            x = np.where(rng.random(x.shape) < 0.1, x, 0.0) * np.exp2(-rng.integers(0, 26, x.shape))
        elif kind == "coherent":
            x = np.where(rng.random(x.shape) < 0.02, x, np.abs(x) * np.exp2(-rng.integers(14, 28, (64, 1))) * h[rng.integers(0, 128, 64)])
        elif kind == "decreasing":
            x *= np.exp2(-np.arange(128) / rng.integers(2, 12, (64, 1)))
        x = to_bf16(x)
        off = np.abs(chained_contraction(x, h) - x @ h).max(1)
        bound = lost_at_most(x)
        assert (off <= bound).all()
        worst = max(worst, (off / np.where(bound > 0, bound, 1)).max())
    assert worst > 0.1


@pytest.mark.gpu
@pytest.mark.parametrize("fmt", ["int4", "fp4", "int4_asym"])
@pytest.mark.parametrize("d,T", [(4096, 8195), (2048, 16389)])
def test_whole_row_rotations(B, oracle, d, T, fmt):
    run(B, oracle, whole_rows(d, 40000 + d), T, d, fmt, 0)


@pytest.mark.gpu
@pytest.mark.parametrize("fmt,group", [("int4", 0), ("int4", 128), ("fp4", 0), ("mxfp4", 32)])
@pytest.mark.parametrize("b", [64, 128])
def test_blocks(B, oracle, b, fmt, group):
    run(B, oracle, block_rows(1152, b, 42000 + b), 16 * 2 ** 20 // 1152 + 3, b, fmt, group)


def upper_end_rows(oracle, d, b, seed):
    """Largest unnormalised outputs in (2^125.98, 2^127.98]; and blocks in which the sum of the first inputs passes 2^128 although
    no output does."""
    rng = np.random.default_rng(seed)
    x = to_bf16(rng.standard_normal((48, d)) + 0.2)
    u = np.abs(oracle.rotate(bits(x), None, b)).max(axis=1) * np.sqrt(b)
    x *= np.exp2(np.floor(126.98 + np.arange(48) % 2 - np.log2(u)))[:, None]
    n = min(b, 128)
    if n >= 64:
        k, a = np.arange(n), 1.5 * 2.0 ** (121 if n == 128 else 122)
        for i in range(0, 48, 4):
            m = int(rng.integers(n))
            signs = 1.0 - 2.0 * (np.array([bin(v).count("1") for v in (k & m)]) & 1)
            x[i] = 0.0
            x[i, n * (i // 4 % (d // n)):][:n] = np.where(k < n - 16, a, -3 * a if n == 128 else -a) * signs
            if i % 8:
                x[i] += np.where(x[i] == 0, to_bf16(rng.standard_normal(d) * 2.0 ** 115), 0.0)
    return bits(x)


@pytest.mark.gpu
@pytest.mark.parametrize("fmt,group", [("int4", 0), ("int4", 128), ("fp4", 0), ("mxfp4", 32)])
@pytest.mark.parametrize("b", [16, 32, 64, 128])
def test_blocks_at_the_upper_end_of_the_range(B, oracle, b, fmt, group):
    run(B, oracle, upper_end_rows(oracle, 1152, b, 44000 + b), 16 * 2 ** 20 // 1152 + 3, b, fmt, group)


@pytest.mark.gpu
@pytest.mark.parametrize("fmt", ["int4", "fp4", "int4_asym"])
@pytest.mark.parametrize("d,T", [(4096, 8195), (2048, 16389)])
def test_whole_rows_at_the_upper_end_of_the_range(B, oracle, d, T, fmt):
    run(B, oracle, upper_end_rows(oracle, d, d, 45000 + d), T, d, fmt, 0)


def test_tile_err_covers_the_model():
    """|u32 - u| of the model against the tile kernel's constants (16, 20, 45 and 103 * 2^-24 of the block's largest output)."""
    rng = np.random.default_rng(43000)
    for b, err in ((16, 16), (32, 20), (64, 45), (128, 103)):
        h, worst = hadamard(b), 0.0
        rows = [rng.standard_normal((64, b)) * np.exp2(-rng.integers(0, 1 + 8 * t, (64, b))) for t in range(5)]
        if b >= 64:
            rows.append(np.array([hidden_maximum(b, b, 62), hidden_side(b, b, 6.5 / 7, 10), hidden_step(b, b, 12, 10)]))
        # one large input, and every other one just below what is kept beside it, agreeing in sign
        rows.append(np.where(np.arange(b) == 0, 1.0, h[rng.integers(0, b, 64)] * 1.9921875 * 2.0 ** -rng.integers(20, 26, (64, 1)).astype(float)))
        for x in rows:
            x = to_bf16(x)
            off = np.abs(chained_contraction(x, h) - x @ h).max(1) / np.abs(x @ h).max(1)
            worst = max(worst, off.max() * 2 ** 24)
        assert worst < err
        assert worst > (3 if b == 16 else 6 if b == 32 else 24 if b == 64 else 56)


# ------------------------------------------------------------------ the other attacks on the bounds, at these kernels' sizes

LARGE = [(1152, 16 * 2 ** 20 // 1152 + 3, b, fmt, group) for b in (16, 32, 64, 128) for fmt, group in (("int4", 0), ("int4", 128), ("fp4", 0), ("mxfp4", 32))]
LARGE += [(d, T, d, fmt, 0) for d, T in ((4096, 8195), (2048, 16389)) for fmt in ("int4", "fp4", "int4_asym")]


def flat_spectrum_rows(d, b, seed):
    """Signs whose rotation is as flat as it can be, times mantissas in [1, 2): the partial sums are as large as the outputs."""
    k, s = np.arange(b), 0
    for i in range(int(np.log2(b)) - 1):
        s = s ^ (k >> i) & (k >> (i + 1)) & 1
    rng = np.random.default_rng(seed)
    x = (1.0 + rng.integers(0, 128, (48, d // b, b)) / 128.0) * (1.0 - 2.0 * s)
    x *= np.exp2(rng.integers(-3, 4, (48, d // b, 1))) * rng.choice([-1.0, 1.0], (48, d // b, 1))
    x = x.reshape(48, d)
    x[::7] = to_bf16(rng.standard_normal((7, d)))
    return bits(x)


def small_and_shifted_rows(d, b, seed):
    """Rows at the lower end of the range (largest output 2^-119 and more), and rows far from symmetric (zero points of some 100)."""
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((48, d))
    x[1::3, :: max(1, d // 8)] *= 100.0
    x[2::3] += 40.0
    x[::3] *= np.exp2(-rng.integers(112, 118, (16, 1)))
    return bits(to_bf16(x))


def cancelling_rows(d, b, seed):
    """Blocks of four runs 3v, 4v, 5v, 4v: a quarter of the outputs is zero exactly, and fp32 leaves noise there."""
    rng = np.random.default_rng(seed)
    shape = (48, d // b, 1, b // 4)
    v = rng.integers(1, 16, shape) * np.exp2(rng.integers(-14, 15, shape)) * rng.choice([-1.0, 1.0], shape)
    return bits((v * np.array([3.0, 4.0, 5.0, 4.0])[None, None, :, None]).reshape(48, d))


def wide_rows(d, b, seed):
    """Inputs over 40 binades, and one large input with tiny ones of one sign."""
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((48, d)) * np.exp2(-rng.integers(0, 40, (48, d)))
    x[::2] = np.abs(rng.standard_normal((24, d))) * np.exp2(-rng.integers(16, 28, (24, 1)))
    x[np.arange(0, 48, 2), rng.integers(0, d, 24)] = 1.5
    return bits(to_bf16(x))


@pytest.mark.gpu
@pytest.mark.parametrize("make", [flat_spectrum_rows, small_and_shifted_rows, cancelling_rows, wide_rows])
@pytest.mark.parametrize("d,T,b,fmt,group", LARGE)
def test_large_calls(B, oracle, d, T, b, fmt, group, make):
    run(B, oracle, make(d, b, 46000 + b), T, b, fmt, group)


def vanishing_groups(d, b, seed):
    """Two large inputs that cancel in half of a block's outputs, and before the second one tiny inputs that fp32 loses
    beside the first: whole MX groups that are zero in fp32 and not in truth."""
    rng, k, h = np.random.default_rng(seed), np.arange(b), hadamard(b)
    x = np.zeros((48, d // b, b))
    for i in range(48):
        for j in range(d // b):
            tiny = (k > 0) & (k < b // 2) & (rng.random(b) < (1.0 if i % 3 else 0.2))
            x[i, j] = np.where(tiny, h[int(rng.integers(b))] * 0.9921875 * 2.0 ** -25, 0.0)
            x[i, j, 0] = x[i, j, b // 2] = 1.0
            x[i, j] *= 2.0 ** int(rng.integers(-20, 20))
    return bits(x.reshape(48, d))


@pytest.mark.gpu
@pytest.mark.parametrize("b", [64, 128])
def test_groups_that_vanish_in_fp32(B, oracle, b):
    run(B, oracle, vanishing_groups(1152, b, 47000 + b), 16 * 2 ** 20 // 1152 + 3, b, "mxfp4", 32)


def perm_err(b, ranges):
    """The permuted kernel's bound in 2^-24 of the block's largest output, from its source."""
    with open(os.path.join(os.path.dirname(LAUNCH), "perq_perm.cuh")) as f:
        rule = re.search(r"constexpr float perm_err\(int log2b, bool ranges\) \{ return \(ranges && log2b == 7 \? ([0-9.]+)f : ([0-9.]+)f \* log2b\) \* 0x1p-24f; \}", f.read())
    return float(rule.group(1)) if ranges and b == 128 else float(rule.group(2)) * np.log2(b)


@pytest.mark.parametrize("b", [16, 32, 64, 128])
def test_what_a_step_and_stages_lose(b):
    """The bound covers what the steps and the stages can lose, and with it what the model loses."""
    c = b // 16
    proven = 9.5 * np.sqrt(c) + sum(np.sqrt(2.0 ** k) for k in range(int(np.log2(c))))
    assert perm_err(b, True) >= proven and 2 * perm_err(b, False) >= proven
    rng, worst = np.random.default_rng(43000 + b), 0.0
    for make in [lambda: losing_chunks(512, b, rng)] * 20 + [lambda: rng.standard_normal((512, b)) * np.exp2(-rng.integers(0, 30, (512, b)))] * 5:
        x = to_bf16(make()).reshape(-1, b)
        u = x @ hadamard(b)
        worst = max(worst, (np.abs(one_step_and_stages(x) - u).max(1) / np.abs(u).max(1)).max() * 2.0 ** 24)
    assert 3 < worst <= proven


@pytest.mark.gpu
@pytest.mark.parametrize("fmt,group", [("int4", 128), ("mxfp4", 32)])
@pytest.mark.parametrize("b", [16, 32, 64, 128])
def test_permuted_rows_that_lose(B, oracle, b, fmt, group):
    d, n = 1152, 160
    rng = np.random.default_rng(44000 + b)
    x = losing_chunks(n * d // b, b, rng).reshape(n, d) * np.exp2(rng.integers(-20, 20, (n, 1)))
    perm = rng.permutation(d).astype(np.int32)
    base = np.empty((n, d), np.uint16)
    base[:, perm] = bits(x)
    xt = torch.from_numpy(np.tile(base, (4, 1)).view(np.int16)).cuda().view(torch.bfloat16)
    codes, scales = B.perq_rotate_quantize(xt, torch.from_numpy(perm).cuda(), b, FMT[fmt], group)
    torch.cuda.synchronize()
    ora = oracle.rotate_quantize(base, perm, b, FMT[fmt], group, want_pre=True)
    for part in range(4):
        rows = slice(n * part, n * part + n)
        compare_quantized(fmt, codes[rows].cpu().numpy(), scales[rows].cpu().numpy(), ora)
