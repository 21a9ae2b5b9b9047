"""The interpreter's own entry to the two calls: same arguments, same status as through ctypes, and the same refusals."""
import ctypes
import os

import numpy as np
import pytest


@pytest.fixture(scope="module")
def B():
    from paper_2601_22347_b200 import binding, build
    build.build()
    binding.load()
    if not os.path.exists(build.CALL_PATH):
        pytest.skip("no interpreter headers")
    return binding


@pytest.mark.parametrize("args", [(None, None, 0, 2048, 16, 0, 0, None, None, None), (None, None, 4, 2048, 16, 0, 0, None, None, None),
                                  (16, None, 4, 2048, 17, 0, 0, 16, 16, 0), (16, 6, 4, 2048, 16, 0, 0, 16, 16, 0), (16, None, -1, 2048, 16, 0, 0, 16, 16, 0),
                                  (16, None, 4, 2048, 16, 9, 0, 16, 16, 0), (16, None, 4, 2048, 16, 0, -5, 16, 16, 0), (8, None, 4, 2048, 16, 0, 0, 16, 16, 0),
                                  (2 ** 64 - 8, None, 4, 2048, 16, 0, 0, 16, 16, 0), (16, None, 0, 2 ** 32 + 2048, 16, 0, 0, 16, 16, 0)])
def test_status(B, args):
    """(All of these are decided before anything is launched.)"""
    assert B._rotate_quantize(*args) == B._lib.perq_rotate_quantize(*args)
    swiglu = (args[0],) + args
    assert B._swiglu_rotate_quantize(*swiglu) == B._lib.perq_swiglu_rotate_quantize(*swiglu)


@pytest.mark.parametrize("bad", [1.5, "16", None, np.float32(16), ctypes.c_int(16)])
def test_refusals(B, bad):
    with pytest.raises(TypeError):
        B._rotate_quantize(None, None, 0, 2048, bad, 0, 0, None, None, None)
    with pytest.raises(TypeError):
        B._rotate_quantize(None, None, 0)
    with pytest.raises(TypeError):
        B._swiglu_rotate_quantize(None, None, None, 0, 2048, bad, 0, 0, None, None, None)
