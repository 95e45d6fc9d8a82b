"""The pass over the layer that derives the per-class shift: block counts that leave a thread with one to six blocks, block
maxima on both sides of every class's cut point, scales at the ends of the fp32 range (quotients that overflow or turn
subnormal), classes with and without a power-of-two range.  Shifts and max|W| are compared exactly."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_14929_b200 import inputs as I

from .test_gpu_parity import B, gpu_search  # noqa: F401  (B is a fixture)

pytestmark = pytest.mark.gpu


def _atoms():
    lut = np.linspace(-1.0, 1.0, 16).astype(np.float32)
    tables = [I.Atom(f"t{t}", 4, I.KIND_LUT, 0, 16, t, np.float32(t) * lut) for t in (np.float32(0.7), np.float32(1.9921875), np.float32(4.0))]
    return I.alphabet(["NF4"], fp=["E2M3", "E4M3"]) + tables


def _check(B, W, fmt_name):
    fmt, atoms = I.scale_format(fmt_name), _atoms()
    M, K = W.shape
    got = gpu_search(B, W, torch.ones(K), fmt, atoms)
    amax = W.float().abs().reshape(M * K // 16, 16).amax(dim=1).numpy()
    assert got["layer_absmax"] == amax.max()
    for i, a in enumerate(atoms):
        with np.errstate(over="ignore"):
            assert int(got["k"][i]) == oracle.f_layer(fmt, (amax / np.float32(a.tmax)).astype(np.float32)), (i, a.name)


@pytest.mark.parametrize("M,K", [(1, 16), (9, 48), (151553, 16), (1000, 4096), (850001, 16)])
def test_shifts_of_every_class(B, M, K):
    g = torch.Generator().manual_seed(M + K)
    W = torch.randn(M, K, generator=g).to(torch.bfloat16)
    _check(B, W, "E4M5")


@pytest.mark.parametrize("top", [-126, -110, 30, 118])
def test_scales_at_the_ends_of_the_range(B, top):
    # every mantissa as a block maximum, at exponents around `top`; subnormal weights among the smallest
    m = 1.0 + torch.arange(128, dtype=torch.float64) / 128.0
    e = torch.arange(top - 6, top + 3, dtype=torch.float64)
    amax = (m[None, :] * 2.0 ** e[:, None]).reshape(-1, 1)
    W = (amax * torch.linspace(-1.0, 0.5, 16, dtype=torch.float64)[None, :]).to(torch.float32).to(torch.bfloat16)
    _check(B, W, "UE4M4")
