"""The device functions that stand for longer arithmetic or for rounded instructions, over whole ranges of their operands."""
import ctypes as C

import numpy as np
import pytest
import torch

from . import device_checks

pytestmark = pytest.mark.gpu


def _run(fn, *args):
    bad = torch.zeros(4, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert fn(*args, C.c_void_p(bad.data_ptr())) == 0
    return bad.tolist()


def test_the_fast_cosine_is_the_rounded_quotient_by_the_rounded_root():
    lib = device_checks.lib()
    rng = np.random.default_rng(1)
    one = 0x3F800000
    # every significand of x in two neighbouring binades (a root depends on x up to a power of four) against powers of two and other values
    dots = np.concatenate([[1.0, 0.5, 2.0 ** -20, 1.5, 2.0 - 2.0 ** -23, 1.0 + 2.0 ** -23, 1.0 / 3.0], rng.uniform(0.5, 2.0, 25)]).astype(np.float32)
    d = torch.from_numpy(dots).cuda()
    bad = _run(lib.check_cosine, C.c_uint(one), C.c_uint(1 << 24), C.c_void_p(d.data_ptr()), len(dots))
    assert bad[0] == 0 and bad[2:] == [2, 0], bad
    # the ends of the range of x
    for lo in (0x17800000, 0x67000000):
        bad = _run(lib.check_cosine, C.c_uint(lo), C.c_uint(1 << 24), C.c_void_p(d.data_ptr()), len(dots))
        assert bad[0] == 0 and bad[2:] == [2, 0], (hex(lo), bad)
    # every significand of the dot product against roots near a power of two, near all ones and of any kind
    every = torch.arange(1 << 23, dtype=torch.int32, device="cuda").add_(one).view(torch.float32)
    xs = [one, one + 1, one + 2, one + (1 << 24) - 3, one + (1 << 23), one + (1 << 23) - 1] + list(one + rng.integers(0, 1 << 24, 10))
    for x in xs:
        bad = _run(lib.check_cosine, C.c_uint(int(x)), C.c_uint(1), C.c_void_p(every.data_ptr()), every.numel())
        assert bad[0] == 0, (hex(int(x)), bad)


@pytest.mark.parametrize("exponent", [4, 5, 126, 127, 128, 249, 250])
def test_the_reciprocal_of_a_scale_is_rounded_to_nearest(exponent):
    # every significand; 4 .. 250 are the exponent fields that the sweep and the packer take this path for
    assert _run(device_checks.lib().check_reciprocal, C.c_uint(exponent))[0] == 0


@pytest.mark.parametrize("kind", [1, 2])
def test_the_conversion_instructions_quantise_and_encode_like_the_arithmetic(kind):
    # every finite fp32 pattern, in both places of the pair
    assert _run(device_checks.lib().check_quantize, C.c_int(kind))[:2] == [0, 0]
