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


def ctypes_takes_the_calls(B, monkeypatch, path):
    from paper_2601_22347_b200 import build
    for name in ("_lib", "_rotate_quantize", "_swiglu_rotate_quantize"):
        monkeypatch.setattr(B, name, None)
    monkeypatch.setattr(build, "CALL_PATH", str(path))
    lib = B.load()
    return B._rotate_quantize is lib.perq_rotate_quantize and B._swiglu_rotate_quantize is lib.perq_swiglu_rotate_quantize


@pytest.mark.parametrize("content", [None, b"", b"another machine's file", b"\x7fELF" + bytes(200)], ids=["missing", "empty", "text", "header"])
def test_an_entry_that_cannot_be_loaded(B, monkeypatch, tmp_path, content):
    path = tmp_path / "_perq_call.so"
    if content is not None:
        path.write_bytes(content)
    assert ctypes_takes_the_calls(B, monkeypatch, path)
    assert B._rotate_quantize(None, None, 4, 2048, 16, 0, 0, None, None, None) == 1      # PERQ_ERR_NULL


@pytest.mark.parametrize("cc", ["/nowhere/cc", "false"])
def test_a_compiler_that_is_missing_or_fails(B, monkeypatch, tmp_path, cc):
    """The entry is left out, an older one taken away, and the library built as ever."""
    from paper_2601_22347_b200 import build
    path = tmp_path / "_perq_call.so"
    path.write_bytes(b"older")
    os.utime(path, (0, 0))
    monkeypatch.setattr(build, "CALL_PATH", str(path))
    monkeypatch.setenv("CC", cc)
    assert build.build() == build.LIB_PATH
    assert not path.exists()
