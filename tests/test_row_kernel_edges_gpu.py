"""Parity with the oracle on inputs at the edges of the kernels' fp32 arithmetic: scale ranges that hold
small outputs of a block with large ones, MX groups that cancel exactly, rows at the upper end of the range,
rows in which many outputs tie."""
import numpy as np
import pytest
import torch

from paper_2601_22347_b200 import inputs

from parity import compare_quantized

pytestmark = pytest.mark.gpu

FMT = {"int4": 0, "mxfp4": 1, "fp4": 3, "int4_asym": 4}


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


def run(B, bits, perm, b, fmt, group):
    x = torch.from_numpy(bits.view(np.int16).copy()).cuda().view(torch.bfloat16)
    p = None if perm is None else torch.from_numpy(perm).cuda()
    codes, scales = B.perq_rotate_quantize(x, p, b, FMT[fmt], group)
    torch.cuda.synchronize()
    return codes.cpu().numpy(), scales.cpu().numpy()


def check(B, oracle, bits, perm, b, fmt, group):
    codes, scales = run(B, bits, perm, b, fmt, group)
    return compare_quantized(fmt, codes, scales, oracle.rotate_quantize(bits, perm, b, FMT[fmt], group, want_pre=True))


def through(bits, perm):
    """The rows whose gather through perm gives `bits`."""
    if perm is None:
        return bits
    out = np.empty_like(bits)
    out[:, perm] = bits
    return out


# ------------------------------------------------------------------ small outputs of a block with large ones

def _cancelling_rows(T, d, b, log2_ratio, seed):
    """Blocks whose upper half of outputs holds values 2^-log2_ratio of the lower half's: 16 large channels that occur
    in both halves of the block (and cancel in the upper outputs), 16 ordinary ones."""
    rng = np.random.default_rng(seed)
    x = np.zeros((T, d // b, b))
    for t in range(T):
        for j in range(d // b):
            k = rng.choice(b // 2, 16, replace=False)
            x[t, j, k] = x[t, j, k + b // 2] = rng.standard_normal(16) * 2.0 ** log2_ratio
            free = np.setdiff1d(np.arange(b), np.r_[k, k + b // 2])
            x[t, j, rng.choice(free, 16, replace=False)] = rng.standard_normal(16)
    return inputs.f32_to_bf16_bits(x.reshape(T, d).astype(np.float32))


# (up to 2^23: beyond, whole ranges vanish in fp32, and a range whose fp32 values are all zero gets scale 0)
@pytest.mark.parametrize("log2_ratio", [18, 20, 21, 22, 23])
@pytest.mark.parametrize("T,d,b,group,perm", [(40, 1024, 128, 32, False), (40, 1152, 128, 64, True), (60, 640, 64, 32, False),
                                              (9, 14336, 14336, 128, False), (20, 3072, 3072, 128, True), (20, 3072, 3072, 32, False),
                                              (20, 1024, 256, 64, True), (10, 4096, 2048, 128, True)])
def test_ranges_far_below_their_block(B, oracle, T, d, b, group, perm, log2_ratio):
    """The fp32 maximum of such a range is partly rounding noise: it does not pin a code to two neighbours, and at the
    higher ratios values that are zero in fp32 are among the candidates for the exact maximum."""
    p = inputs.random_perm(d, 81) if perm else None
    bits = through(_cancelling_rows(T, d, b, log2_ratio, 8000 + d + b + log2_ratio), p)
    check(B, oracle, bits, p, b, "int4", group)


# ------------------------------------------------------------------ MX groups that are exactly zero in a block that is not

def _zero_quarter_rows(T, d, b, seed):
    """Blocks of four runs 3v, 4v, 5v, 4v: the second quarter of the outputs is (3 - 4 + 5 - 4) H v = 0 exactly.  v spans
    29 binades, so that fp32 leaves noise there; the products are exact in bf16, all sums exact in fp64 (50 bits)."""
    rng = np.random.default_rng(seed)
    shape = (T, d // b, 1, b // 4)
    v = rng.integers(1, 16, size=shape) * np.exp2(rng.integers(-14, 15, size=shape)) * rng.choice([-1.0, 1.0], size=shape)
    x = (v * np.array([3.0, 4.0, 5.0, 4.0])[None, None, :, None]).reshape(T, d)
    bits = inputs.f32_to_bf16_bits(x.astype(np.float32))
    assert np.array_equal(inputs.bf16_to_f64(bits), x)
    return bits


def check_zero_groups(B, oracle, T, d, b, perm):
    p = inputs.random_perm(d, 82) if perm else None
    bits = through(_zero_quarter_rows(T, d, b, 8100 + d + b), p)
    zero = oracle.rotate_quantize(bits, p, b, FMT["mxfp4"], 32)["scales"] == 0
    assert zero.sum() * 4 == zero.size
    check(B, oracle, bits, p, b, "mxfp4", 32)


@pytest.mark.parametrize("T,d,b,perm", [(20, 1024, 256, True), (20, 1152, 128, False), (20, 1152, 128, True), (9, 3072, 3072, False),
                                        (6, 14336, 14336, True), (9, 2048, 2048, True), (7, 6144, 2048, False),
                                        (5, 16384, 16384, False), (9, 8192, 4096, True)])
def test_row_kernel_mx_groups_that_cancel(B, oracle, T, d, b, perm):
    check_zero_groups(B, oracle, T, d, b, perm)


@pytest.mark.parametrize("T,d,b,perm", [(20, 1024, 128, False), (20, 3072, 128, False), (20, 2048, 128, True), (20, 2048, 256, False),
                                        (9, 2048, 512, False), (9, 2048, 1024, False), (9, 1024, 1024, False), (9, 2048, 2048, False),
                                        (9, 4096, 4096, False), (9, 8192, 8192, False)])
def test_segment_kernels_mx_groups_that_cancel(B, oracle, T, d, b, perm):
    """The lean, the group (odd segment counts, permuted, blocks over lanes and warps) and the full-vector kernel."""
    check_zero_groups(B, oracle, T, d, b, perm)


# ------------------------------------------------------------------ rows at the upper end of the fp32 range

def _rows_at_the_upper_end(oracle, T, d, b, seed):
    """Rows whose largest unnormalised output lies in (2^125.98, 2^126.98] or (2^126.98, 2^127.98], alternating."""
    rng = np.random.default_rng(seed)
    x = inputs.bf16_to_f64(inputs.f32_to_bf16_bits((rng.standard_normal((T, d)) + 0.2).astype(np.float32)))
    u = np.abs(oracle.rotate(inputs.f32_to_bf16_bits(x.astype(np.float32)), None, b)).max(axis=1) * np.sqrt(b)
    x *= np.exp2(np.floor(126.98 + np.arange(T) % 2 - np.log2(u)))[:, None]
    bits = inputs.f32_to_bf16_bits(x.astype(np.float32))
    assert np.array_equal(inputs.bf16_to_f64(bits), x)
    return bits


@pytest.mark.parametrize("fmt,group", [("int4", 0), ("int4", 128), ("int4", 64), ("fp4", 0), ("int4_asym", 0), ("mxfp4", 32)])
@pytest.mark.parametrize("T,d,b", [(12, 1152, 128), (12, 2048, 2048), (12, 3072, 3072), (12, 4096, 4096), (6, 16384, 16384),
                                   (6, 14336, 14336)])
def test_rows_at_the_upper_end_of_the_range(B, oracle, T, d, b, fmt, group):
    """Outputs whose reciprocal, range or sum of two leaves the fp32 range where they themselves do not."""
    check(B, oracle, _rows_at_the_upper_end(oracle, T, d, b, 8200 + d + b), None, b, fmt, group)


# ------------------------------------------------------------------ flat rows: many outputs tie, fp32 is exact

def _flat_rows(T, d, b, seed):
    """One nonzero in the row, one in every block, few small integers, +-constant, constant, and rows just beyond the reach of
    exact fp32 arithmetic: a large and a tiny nonzero."""
    rng = np.random.default_rng(seed)
    x = np.zeros((T, d))
    for t in range(T):
        blk = x[t].reshape(d // b, b)
        if t % 6 == 0:
            x[t, rng.integers(d)] = -2.625
        elif t % 6 == 1:
            blk[:, rng.integers(b)] = 1.5 * (1 + np.arange(d // b) % 3)
        elif t % 6 == 2:
            x[t, rng.choice(d, 8, replace=False)] = np.arange(1, 9)
        elif t % 6 == 3:
            x[t] = np.where(rng.random(d) < 0.5, -1.25, 1.25)
        elif t % 6 == 4:
            x[t] = 1.2890625 * 2.0 ** rng.integers(-100, 100)
        else:
            x[t, rng.choice(d, 2, replace=False)] = 3.0, 2.0 ** -23
    return inputs.f32_to_bf16_bits(x.astype(np.float32))


@pytest.mark.parametrize("fmt,group", [("int4", 0), ("int4", 32), ("int4", 128), ("fp4", 0), ("int4_asym", 0), ("mxfp4", 32)])
@pytest.mark.parametrize("T,d,b,perm", [(18, 1152, 128, False), (18, 640, 32, True), (24, 1024, 128, False), (18, 3072, 1024, True), (12, 2048, 2048, False),
                                        (12, 4096, 4096, False), (12, 6144, 2048, True), (6, 8192, 8192, False), (12, 3072, 3072, False), (6, 14336, 14336, True)])
def test_flat_rows(B, oracle, T, d, b, perm, fmt, group):
    p = inputs.random_perm(d, 83) if perm else None
    check(B, oracle, through(_flat_rows(T, d, b, 8300 + d + b), p), p, b, fmt, group)
