"""The device MassDiff up to 256 blocks (a block to a lane, sorted after every batch) at the sizes where it changes: 16 and 17 blocks, full
and part-filled warps, 256 and 257 blocks; masses whose batches are small, whose sums tie, and that are too small to change a
sum, so that blocks fill one after the other and no sum is near the smallest one."""
import numpy as np
import pytest
import torch

from massdiff_threads import KINDS, far_apart
from test_massdiff_device_gpu import B, device_perm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["statistic", "steep", "tiny", "noise", "integers", "rank", "zeros"])
@pytest.mark.parametrize("n,b", [(1, 32), (2, 16), (16, 8), (17, 40), (32, 3), (33, 64), (64, 1), (65, 32), (128, 24), (129, 2), (256, 32), (256, 128), (257, 32)])
def test_blocks_to_lanes(B, kind, n, b):                     # noqa: F811
    d = n * b
    rng = np.random.default_rng(9200 + d)
    a = {"statistic": np.abs(rng.standard_normal((64, d)).astype(np.float32)).sum(0) * np.where(rng.random(d) < 1 / 256, 30.0, 1.0),
         "steep": 1.02 ** -np.arange(d).clip(0, 300).astype(np.float64),
         "tiny": np.where(np.arange(d) < d // 2, 1.1 ** -np.arange(d).clip(0, 40).astype(np.float64), 1e-30),
         "noise": 1.0 + 1e-6 * rng.random(d), "integers": rng.integers(0, 20, d), "rank": 1.0 / (1.0 + np.arange(d)),
         "zeros": rng.exponential(size=d) * (rng.random(d) < 0.6)}[kind]
    a = rng.permutation(a.astype(np.float32))
    assert np.array_equal(device_perm(B, a, b), B.perq_massdiff_perm(a, b))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n,b", [(32, 16), (33, 128), (63, 32), (66, 16), (75, 128), (100, 32), (128, 16), (129, 48), (256, 16), (256, 32), (256, 128)])
def test_blocks_far_apart(B, kind, n, b):                    # noqa: F811
    for seed in range(30):
        a = far_apart(kind, n, b, seed)
        assert np.array_equal(device_perm(B, a, b), B.perq_massdiff_perm(a, b)), seed
