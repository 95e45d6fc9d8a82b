"""GPU parity of the sweep's joint evaluation of table candidates where it can go wrong: more candidates of a class than one
group holds, an odd number of them, table values that are no bf16 numbers, lookup cells with three and with more decision
points, and block sums outside the range of the fast cosine.  Per-block values bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_14929_b200 import inputs as I

from .test_gpu_parity import B, check_search, gpu_search  # noqa: F401  (B is a fixture)

pytestmark = pytest.mark.gpu


def _table(name, lut, n_bits=4):
    return I.Atom(name, n_bits, I.KIND_LUT, 0, 16, float(np.abs(lut).max()), np.sort(np.asarray(lut, dtype=np.float32)))


def _dense(step, n):
    """16 entries, n + 1 of them `step` apart around 0.3 (n decision points `step` apart), the rest spread out."""
    return np.concatenate([np.linspace(-1.0, 0.1, 15 - n), 0.3 + step * np.arange(n + 1)[:n], [1.0]])


def _alphabet(kind):
    rng = np.random.default_rng(11)
    if kind == "twelve":          # one class, twelve candidates: a group of eight and one of four
        extra = [_table(f"r{i}", np.concatenate([[-1.0, 1.0], I.snap_bf16(rng.uniform(-0.95, 0.95, 14))])) for i in range(2)]
        return I.alphabet(["NF4", "SH4", "BOF4", "Split87"]) + [x for a in extra for x in (a, a.negation())]
    if kind == "odd":             # five candidates without negations, values with full fp32 significands
        return [_table(f"f{i}", np.concatenate([[-1.0, 1.0], rng.uniform(-0.99, 0.99, 14)])) for i in range(5)]
    if kind == "cell3":           # a cell with three decision points (cells are 2.5 / 640 wide)
        return [_table("c3", _dense(5e-4, 4))] + I.alphabet(["NF4"])
    if kind == "cell6":           # more than three: the group is searched
        a = _table("c6", _dense(2e-4, 7))
        return [a, a.negation()] + I.alphabet(["NF4", "SH4"])
    return I.alphabet(["NF5", "SH5", "BOF5", "E2M2"])      # two classes: six candidates and two


@pytest.mark.parametrize("kind,fmt_name", [("twelve", "E5M6"), ("odd", "UE4M4"), ("cell3", "E4M5"), ("cell6", "UE4M6"), ("classes", "E4M3")])
def test_groups_of_candidates_match_oracle(B, kind, fmt_name):
    check_search(B, I.tiny_layer(21, 37, 272), fmt_name, _alphabet(kind))


@pytest.mark.parametrize("fmt_name", ["E8M7", "UE4M4", "UE8M0"])
def test_block_sums_of_any_magnitude(B, fmt_name):
    # rows from 2^-64 to 2^60: norms and dot products from below 2^-80 to above 2^80 take the general cosine, the others the
    # fast one; a zero row, a row with one non-zero weight per block
    L = I.tiny_layer(22, 24, 256)
    W = L.W.float() * (2.0 ** torch.linspace(-64, 60, 24).round())[:, None]
    W[5] = 0
    W[6] = torch.where(torch.arange(256) % 16 == 3, W[6], torch.zeros(256))
    check_search(B, I.Layer(W.to(torch.bfloat16), L.X), fmt_name, I.alphabet(["NF4", "SH4"], fp=["E2M3", "E4M3"]))


@pytest.mark.parametrize("fmt_name", ["E8M7", "UE8M0"])
def test_a_norm_that_overflows_against_one_that_underflows(B, fmt_name):
    # per block one huge weight on a channel without activations and fifteen smaller ones that reconstruct as 1e-25: <w, w>
    # overflows, <q, q> underflows to zero, their product is no number and the cosine is zero
    L = I.tiny_layer(23, 24, 256)
    first = (torch.arange(256) % 16 == 0)
    W = torch.where(first, torch.full((), 2.0 ** 100), (L.W.float().abs() + 1.0) * 2.0 ** 66)
    X = torch.where(first, torch.zeros(()), L.X)
    a = _table("small", np.concatenate([np.linspace(-1.0, -0.1, 7), [1e-25], np.linspace(0.1, 1.0, 8)]))
    got, _ = check_search(B, I.Layer(W.to(torch.bfloat16), X), fmt_name, [a, a.negation()])
    assert not got["block_cos"].any()


@pytest.mark.parametrize("fmt_name", ["E8M7", "UE8M0"])
def test_element_formats_where_the_reciprocal_scale_overflows(B, fmt_name):
    # rows from 2^-136 to 2^-100 with zeros among the weights: scales of 2^-128 and below
    L = I.tiny_layer(24, 24, 256)
    W = L.W.float() * (2.0 ** torch.linspace(-131, -95, 24).round())[:, None]
    W = torch.where(torch.rand(24, 256, generator=torch.Generator().manual_seed(2)) < 0.4, torch.zeros(()), W)
    check_search(B, I.Layer(W.to(torch.bfloat16), L.X), fmt_name, I.alphabet([], fp=["E2M3", "E4M3", "E4M3^0"]), k_mode=0)


def test_a_norm_product_whose_root_is_all_ones(B):
    # <w, w> <q, q> = 4 - 2^-22 and <w, q> = 1 (table) or 1/4 (element format): the root rounds to 2 - 2^-23, the quotient of a power
    # of two by it is just above the middle of two numbers
    W, c = torch.zeros(2, 16), np.ones(16, np.float32)
    W[0, 0], W[0, 4], c[4] = 1.0, 0.125, 64.0 * (3.0 - 2.0 ** -22)           # the table reconstructs (1, 0.125) as (1, 0)
    W[1] = W[0]
    three = _table("three", np.array([-1.0, 0.0, 1.0]), n_bits=2)
    for atoms, fmt_name in (([three, three.negation()], "E5M6"), ([three], "UE4M4")):
        want = oracle.pair_search(W.to(torch.bfloat16), c, I.scale_format(fmt_name), atoms, want_blocks=True)
        got = gpu_search(B, W.to(torch.bfloat16), c, I.scale_format(fmt_name), atoms)
        assert want["block_cos"][0, 0] == np.float32(0.5 + 2.0 ** -24)
        assert np.array_equal(got["block_cos"].view(np.uint32), want["block_cos"].view(np.uint32))
    # E2M3 under the layer scale 1/4: (1, 2^-7) is (4, 2^-5) and reconstructs as (4, 0)
    W, c = torch.zeros(2, 16), np.ones(16, np.float32)
    W[:, 0], W[:, 4], c[0], c[4] = 1.0, 2.0 ** -7, 1.0 / 16.0, 2.0 ** 14 * (4.0 - 1.0 / 16.0 - 2.0 ** -22)
    pot = I.Atom("E2M3^0", 6, I.KIND_FP_E2M3, 0, I.SCOPE_LAYER_POT, 7.5)
    want = oracle.pair_search(W.to(torch.bfloat16), c, I.scale_format("UE4M4"), [pot], want_blocks=True)
    got = gpu_search(B, W.to(torch.bfloat16), c, I.scale_format("UE4M4"), [pot])
    assert want["block_cos"][0, 0] == np.float32((0.5 + 2.0 ** -24) / 4.0)
    assert np.array_equal(got["block_cos"].view(np.uint32), want["block_cos"].view(np.uint32))
