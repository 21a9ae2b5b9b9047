"""The sorting MassDiff kernel on the CPU, thread by thread (massdiff_threads.py), with warps ahead of each other."""
import numpy as np
import pytest

from massdiff_threads import FIRST, KINDS, LAST, RANDOM, far_apart, massdiff


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


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n,b", [(20, 40), (32, 16), (33, 128), (48, 32), (66, 16), (75, 128), (128, 16), (256, 16), (256, 32)])
def test_the_permutation_of_the_host_function(n, b, kind):
    from paper_2601_22347_b200 import binding
    for seed in range(8):
        a = far_apart(kind, n, b, seed)
        status, perm = massdiff(a, b, seed % 3)
        assert status == 0 and np.array_equal(perm, binding.perq_massdiff_perm(a, b)), seed


@pytest.mark.parametrize("light", [1.0, 0.25])
def test_one_block_closes_between_two_others(light):
    """Block 32 is full while 30 blocks are out of reach, and the two that are next lie 34 to 67 masses above it."""
    from paper_2601_22347_b200 import binding
    a = np.r_[np.full(30, 1e6), 170, 150, np.full(33 * 128 - 32, light)].astype(np.float32)
    assert np.array_equal(massdiff(a, 128)[1], binding.perq_massdiff_perm(a, 128))
