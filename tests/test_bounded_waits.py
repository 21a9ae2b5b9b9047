"""Bounded waits of the kernels whose warps meet at named barriers, by reading the sources (no wait is made to run out on a GPU):
each warp polls by itself, so a wait can run out for one of four and not for another.  They have to agree on that at a
barrier before any of them leaves or goes on to another."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2601_22347_b200", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def body(text, head):
    """The text from `head` to the end of its braces."""
    i = text.index(head)
    depth, k = 0, text.index("{", i)
    for j in range(k, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise ValueError(head)


def test_tile_kernel_agrees_before_its_barriers():
    text = source("perq_tile.cuh")
    epilogue = body(text, "bool tile_epilogue(")
    first = min(m.start() for m in re.finditer(r"named_barrier\w*\(", epilogue))
    assert epilogue[first:].startswith("named_barrier_all(bar, 128, true)")
    loop = body(body(text, "perq_tile_kernel("), "for (uint32_t j = (uint32_t)wg; j < n;")
    failed = body(loop, "if (!ok)")
    assert "named_barrier_all(1 + wg, 128, false)" in failed and failed.index("named_barrier_all") < failed.index("break")
    assert loop.index("if (!ok)") < loop.index("tile_epilogue<") and re.search(r"ok = tile_epilogue<[^;]*;\s*if \(!ok\) \{ give_up\(\); break; \}", loop)


def test_column_kernel_agrees_before_its_barriers():
    loop = body(body(source("perq_col.cuh"), "perq_col_kernel("), "for (uint32_t j = (uint32_t)wg, it = 0; j < n;")
    first = min(m.start() for m in re.finditer(r"named_barrier\w*\(", loop))
    assert loop[first:].startswith("named_barrier_all(bar, 128, ok)")
    assert loop.rindex("mbar_wait_fast") < first and "break" not in loop[:first]


@pytest.mark.parametrize("name", ["perq_tile.cuh", "perq_col.cuh"])
def test_a_wait_that_ran_out_sets_the_documented_bit(name):
    assert set(re.findall(r"atomicOr\(&g_perq_device_error, (\w+)\)", source(name))) == {"1u"}
