"""The sorting MassDiff kernel on the CPU, thread by thread (massdiff_threads.py), with warps ahead of each other."""
import numpy as np
import pytest

from massdiff_threads import FIRST, LAST, RANDOM, massdiff


@pytest.mark.parametrize("policy", [FIRST, LAST] + list(range(RANDOM, RANDOM + 4)))
@pytest.mark.parametrize("n,b", [(8, 16), (32, 16), (33, 16), (66, 16), (128, 8), (256, 32)])
def test_warps_meet_at_the_same_barriers(n, b, policy):
    """Masses whose lightest block becomes full while channels go one by one: the warp that serves them empties the head of the
    list, which the others may not have looked at yet."""
    d = n * b
    for masses in (np.random.default_rng(n).lognormal(0, 2, d), np.r_[np.full(n // 2, 1e6), 170, 150, np.ones(d - n // 2 - 2)]):
        status, perm = massdiff(masses.astype(np.float32), b, policy)
        assert status == 0
        assert np.array_equal(np.sort(perm), np.arange(d))
