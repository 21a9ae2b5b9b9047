"""The device MassDiff where its batched greedy can go wrong, against the host function."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_22347_b200 import binding, build
    build.build()
    binding.load()
    return binding


def device_perm(B, a, b):
    got = B.perq_massdiff_perm_device(torch.from_numpy(a).cuda(), b)
    torch.cuda.synchronize()
    return got.cpu().numpy()


@pytest.mark.parametrize("d,b", [(64, 32), (2080, 32), (4096, 2), (8192, 32), (1024, 1024)])
def test_masses_that_are_not_finite_and_non_negative(B, d, b):
    """A statistic of rows with NaN or infinities: NaN and negative masses count as 0, infinity as the largest float, and
    the result is a permutation (every list place is written; nothing is read that was not)."""
    rng = np.random.default_rng(9000 + d + b)
    a = rng.exponential(size=d).astype(np.float32)
    for share, value in ((0.05, np.nan), (0.03, np.inf), (0.05, -1.0), (0.02, -np.inf), (0.02, -0.0)):
        a[rng.random(d) < share] = value
    a[d // 2] = np.nan
    clean = np.minimum(np.where(a > 0, a, 0), np.finfo(np.float32).max).astype(np.float32)
    assert np.array_equal(device_perm(B, a, b), B.perq_massdiff_perm(clean, b))


@pytest.mark.parametrize("kind", ["exponential", "steep", "equal", "half_zero", "few_large"])
@pytest.mark.parametrize("d,b", [(32, 32), (64, 32), (96, 32), (1024, 32), (1056, 32), (2112, 64), (4096, 1024), (4096, 1), (8192, 8192),
                                 (6144, 48), (32768, 1024)])
def test_channels_one_by_one(B, kind, d, b):
    """1 to 32 blocks (never merged inside a window of 2048 channels), 33, and masses whose batches are too small."""
    rng = np.random.default_rng(9100 + d + b)
    a = {"exponential": rng.exponential(size=d), "steep": 1.02 ** -np.arange(d).clip(0, 4000), "equal": np.ones(d),
         "half_zero": rng.exponential(size=d) * (rng.random(d) < 0.5),
         "few_large": rng.exponential(size=d) * np.where(rng.random(d) < 0.01, 1e5, 1.0)}[kind]
    a = rng.permutation(a.astype(np.float32))
    assert np.array_equal(device_perm(B, a, b), B.perq_massdiff_perm(a, b))
