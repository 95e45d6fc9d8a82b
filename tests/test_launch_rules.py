"""Rules that every kernel keeps because it may start before the one ahead of it on the stream has ended: it lets its successor start, it
waits before it reads what its predecessors wrote, and it makes no promise that data in global memory stays as it is while it lives.
And one of the host code behind the C entries: nothing in it throws."""
import glob
import os
import re

import pytest

from paper_2605_14929_b200 import build as libbuild

SOURCES = libbuild.sources() + glob.glob(os.path.join(libbuild.CSRC, "*.cuh"))


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_load_outside_the_order_of_the_stream(path):
    # __ldg and const __restrict__ allow the non-coherent path, and a compiler may move such loads above the wait
    assert not re.search(r"__ldg\b|__restrict__|ld\.global\.nc", _code(path))


@pytest.mark.parametrize("path", libbuild.sources(), ids=os.path.basename)
def test_every_kernel_lets_its_successor_start_and_waits(path):
    for kernel in re.split(r"\b__global__\b", _code(path))[1:]:
        body = kernel[kernel.index("{"):]
        assert "pdl_trigger()" in body and "pdl_wait()" in body, kernel[:120]
        assert body.index("pdl_trigger()") < body.index("pdl_wait()")
        assert "return" not in body[:body.index("pdl_wait()")], kernel[:120]


@pytest.mark.parametrize("path", libbuild.sources(), ids=os.path.basename)
def test_nothing_behind_the_c_entries_throws(path):
    # containers of the C++ library and operator new throw when memory runs out; a caller through the C ABI cannot catch that
    assert not re.search(r"\bstd::|\bnew\s+[A-Za-z_]|\bthrow\b", _code(path))
