"""GPU parity of the pool's per-cell sums, of the sorted tiles and of the iterations over them where they can go wrong: pools around a
tile of 384 blocks, cells that span many threads (nearly all elements alike), scales that saturate so that |u| passes 2 (and the
clamp of omega u at 256), more tiles in a CTA than it keeps the cell starts of.  The table bit for bit, the trace within 1e-6, for
Lloyd and the dynamic programme."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_14929_b200 import inputs as I

from .test_gpu_parity import B, REL, dev, gpu_lloyd  # noqa: F401  (B is a fixture)

pytestmark = pytest.mark.gpu


def _check(B, L, fmt_name, k, ranks, names=("NF4", "SH4")):
    fmt = I.scale_format(fmt_name)
    atoms = I.alphabet(list(names))
    c = oracle.channel_norms(L.X.numpy())
    r = oracle.pair_search(L.W, c, fmt, atoms, k_mode=oracle.K_AUTO if k is None else k, want_blocks=True)
    bc = torch.from_numpy(r["block_cos"]).to(dev())
    kk = int(r["k"][0])
    ne = len(atoms[0].lut)
    for rank in ranks:
        want = oracle.dd_lloyd(L.W, c, fmt, kk, r["block_cos"][0], rank, atoms[0].lut, 4)
        got = gpu_lloyd(B, L.W, c, fmt, atoms, bc, rank, 4, kk, 0)
        assert np.array_equal(got[0][:ne].view(np.uint32), want[0].view(np.uint32)) and got[2] == want[2], rank
        assert np.allclose(got[1], want[1], rtol=REL, atol=0), rank
        want = oracle.dd_grid_dp(L.W, c, fmt, kk, r["block_cos"][0], rank, ne)
        got = gpu_lloyd(B, L.W, c, fmt, atoms, bc, rank, 0, kk, 0, grid_dp=True)
        assert np.array_equal(got[0][:ne].view(np.uint32), want[0].view(np.uint32)) and got[2] == want[2], rank
        assert got[1][0] == pytest.approx(want[1], rel=REL, abs=1e-12)


@pytest.mark.parametrize("ranks", [(1, 2, 383), (384, 385, 767), (768, 769, 1152)])
def test_pools_around_a_tile(B, ranks):
    _check(B, I.tiny_layer(41, 72, 256), "UE4M4", None, ranks)


def test_a_cell_that_spans_many_threads(B):
    # blocks whose elements are +-1 and tiny values: three cells hold nearly everything
    L = I.tiny_layer(42, 100, 256)
    W = torch.where(torch.rand(100, 256, generator=torch.Generator().manual_seed(1)) < 0.3, torch.sign(L.W.float()), L.W.float() * 1e-4)
    _check(B, I.Layer(W.to(torch.bfloat16), L.X), "E5M6", None, (200, 1600))


@pytest.mark.parametrize("k", [9, 20])
def test_scales_that_saturate(B, k):
    # the shifted scale passes the format's largest value: u = w / scale reaches tens (k = 9) and tens of thousands
    L = I.tiny_layer(43, 40, 512)
    _check(B, L, "UE4M4", k, (300, 1280))


def test_more_tiles_than_a_cta_keeps_the_cell_starts_of(B):
    # 200 tiles on one iteration CTA (165 fit), in both launch forms
    L = I.outlier_channel_layer(44, 300, 4096, 16)
    fmt = I.scale_format("E5M6")
    atoms = I.alphabet(["NF4"])
    c = oracle.channel_norms(L.X.numpy())
    r = oracle.pair_search(L.W, c, fmt, atoms, want_blocks=True)
    NB = r["block_cos"].shape[1]
    assert NB == 200 * 384
    bc = torch.from_numpy(r["block_cos"]).to(dev())
    want = oracle.dd_lloyd(L.W, c, fmt, int(r["k"][0]), r["block_cos"][0], NB, atoms[0].lut, 3)
    B.dd4_lloyd_tuning(iter_ctas=1)
    try:
        for per_iteration in (False, True):
            got = gpu_lloyd(B, L.W, c, fmt, atoms, bc, NB, 3, int(r["k"][0]), 0, launch_per_iteration=per_iteration)
            assert np.array_equal(got[0][:16].view(np.uint32), want[0].view(np.uint32)) and got[2] == want[2]
            assert np.allclose(got[1], want[1], rtol=REL, atol=0)
    finally:
        B.dd4_lloyd_tuning()


def _levels(seed, M, K):
    """Weights of seven values per block (bf16 times a power of two), channel norms over many orders of magnitude."""
    g = torch.Generator().manual_seed(seed)
    v = torch.tensor([-256.0, -179.0, -77.0, 0.0, 77.0, 179.0, 256.0])[torch.randint(0, 7, (M, K // 16, 16), generator=g)] / 256.0
    v[..., 0] = 1.0
    W = (v * 2.0 ** torch.randint(-6, -2, (M, K // 16, 1), generator=g)).reshape(M, K).to(torch.bfloat16)
    return W, torch.exp(2.5 * torch.randn(K, generator=g)).numpy()


@pytest.mark.parametrize("per_iteration", [False, True])
def test_elements_on_their_entries_leave_no_distortion(B, per_iteration):
    # the table finds the seven values: the distortion is zero then, and rounding must not take it below (a negative last entry is the
    # mark of a call that did not finish)
    fmt, atoms = I.scale_format("E5M6"), I.alphabet(["NF4"])
    for seed in range(6):
        W, c = _levels(seed, 256, 1024)
        NB = W.numel() // 16
        bc = torch.rand(2, NB, generator=torch.Generator().manual_seed(seed)).to(dev())
        lut, dist, _ = gpu_lloyd(B, W, c, fmt, atoms, bc, NB // 2, 8, 0, 0, launch_per_iteration=per_iteration)
        assert set(np.array([-256, -179, -77, 0, 77, 179, 256], np.float32) / 256) <= set(lut[:16])
        assert (dist >= 0).all() and dist[8] == 0.0, dist


def test_a_layer_whose_least_cost_rounds_below_zero_is_handed_out(B):
    from paper_2605_14929_b200.pipeline import LayerSweep
    below = 0
    for seed in range(6):
        W, c = _levels(seed, 256, 1024)
        sw = LayerSweep(256, 1024, 2, I.scale_format("E5M6"), ["NF4"], device=dev(), grid_dp=True)
        sw.run(W.to(dev()), torch.from_numpy(np.stack([c, c])).to(dev()))
        below += sw.outputs().distortion[0] < 0
    assert below          # the sums of some of these layers round below zero
