"""GPU parity of the packer where the winner comes from a sweep's values: every code width and container, block counts that end inside
a warp, a group of eight or a pair of blocks, rows with a stride, a table with two thresholds in one lookup cell and one with a
repeated entry, scales below the format's normal range.  Codes and words byte for byte, the padding of the words included."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_14929_b200 import inputs as I

from .test_gpu_parity import B, dev  # noqa: F401  (B is a fixture)

pytestmark = pytest.mark.gpu


def _fine():
    lut = np.concatenate([np.linspace(-1.0, -0.1, 6), [0.3, 0.302, 0.303, 0.304, 0.4, 0.5, 0.6, 0.7, 0.9, 1.0]]).astype(np.float32)
    return I.Atom("fine", 4, I.KIND_LUT, 0, 16, 1.0, I.snap_bf16(lut))


@pytest.mark.parametrize("M,K", [(1, 16), (3, 48), (5, 112), (37, 272)])
@pytest.mark.parametrize("kind,fmt_name,b", [("n4", "S1E4M4", 16), ("n4", "E4M3", 12), ("fine", "UE4M4", 12), ("n5", "UE4M4", 12), ("n5", "E5M6", 16),
                                             ("E2M2", "UE4M4", 16), ("E2M3", "UE4M4", 8), ("E4M3", "UE4M6", 12), ("E4M3^0", "UE4M4", 8)])
def test_packed_bytes_match_oracle(B, M, K, kind, fmt_name, b):
    L = I.tiny_layer(61, M, K)
    W = L.W.float()
    W[0, :16] *= 2.0 ** -40                       # a block below the format's normal range
    if M > 2:
        W[2] = 0
    W = W.to(torch.bfloat16)
    fmt = I.scale_format(fmt_name)
    c = oracle.channel_norms(L.X.numpy())
    if kind in ("n4", "n5", "fine", "E2M2"):
        bases = {"n4": ["NF4", "SH4"], "n5": ["NF5", "SH5"], "E2M2": ["NF5", "E2M2"]}.get(kind)
        atoms = I.alphabet(bases) if bases else [_fine(), _fine().negation()] + I.alphabet(["NF4"])
        a, bb, sign = 0, 2, 1 if fmt.sign_bits else 0
    else:
        atoms, a, bb, sign = [I.fp_atom(kind)], 0, B.NO_ATOM, 0
    wide = torch.zeros((M, K + 24), dtype=torch.bfloat16, device=dev())
    A, NB = len(atoms), M * K // 16
    cd = torch.as_tensor(c).to(dev())
    for Wd in (W.to(dev()), wide[:, :K].copy_(W.to(dev()))):
        pt, st, res = B.new_pair_table(A, dev()), B.new_pair_table(A, dev()), B.new_result(dev())
        bc, bs = torch.empty((A, NB), device=dev()), torch.empty((A, NB), device=dev())
        B.sop_pair_search(Wd, cd, fmt, atoms, pt, st, res, B.alloc_workspace(B.pair_search_workspace(M, K, A), dev()), block_cos=bc, block_sse=bs)
        r = B.read_result(res)
        n = atoms[a].n_bits
        codes = torch.full((NB * 2 * n + 64,), 0x5A, dtype=torch.uint8, device=dev())
        words = torch.full((B.words_nbytes(NB, b) + 64,), 0x5A, dtype=torch.uint8, device=dev())
        counts = torch.zeros(2, dtype=torch.int64, device=dev())
        B.sop_pack(Wd, cd, fmt, atoms, codes, words, index_a=a, index_b=bb, search_result=res, use_sign=sign, container_bits=b,
                   word_sign_bits=sign, counts=counts, block_cos=bc)
        pot = 0.0
        second = None if bb == B.NO_ATOM else atoms[bb]
        plain = torch.full_like(codes, 0x5A), torch.full_like(words, 0x5A), torch.zeros_like(counts)
        B.sop_pack(Wd, cd, fmt, atoms, plain[0], plain[1], index_a=a, index_b=bb, search_result=res, use_sign=sign, container_bits=b,
                   word_sign_bits=sign, counts=plain[2])               # every candidate evaluated in the packer
        assert torch.equal(codes, plain[0]) and torch.equal(words, plain[1]) and torch.equal(counts, plain[2])
        if kind == "E4M3^0":
            continue
        want = oracle.pack(W, c, fmt, atoms[a], int(r["k"][a]), second, 0 if second is None else int(r["k"][bb]), use_sign=sign,
                           container_bits=b, word_sign_bits=sign)
        assert np.array_equal(codes.cpu().numpy()[:NB * 2 * n].reshape(want["codes"].shape), want["codes"])
        assert np.array_equal(words.cpu().numpy()[:want["words"].size], want["words"])
        assert bool((codes[NB * 2 * n:] == 0x5A).all()) and bool((words[B.words_nbytes(NB, b):] == 0x5A).all())


@pytest.mark.parametrize("kind", ["E2M3", "E4M3"])
def test_both_packers_agree_where_the_reciprocal_scale_overflows(B, kind):
    # zeros among weights of 2^-136 and above at a format that has scales below 2^-128
    M, K = 24, 256
    W = I.tiny_layer(62, M, K).W.float() * (2.0 ** torch.linspace(-131, -95, M).round())[:, None]
    W = torch.where(torch.rand(M, K, generator=torch.Generator().manual_seed(3)) < 0.4, torch.zeros(()), W).to(torch.bfloat16).to(dev())
    atoms, fmt, NB = [I.fp_atom(kind)], I.scale_format("UE8M7"), M * K // 16
    cd = torch.ones(K, device=dev())
    bc = torch.zeros((1, NB), device=dev())
    out = []
    for metric in (bc, None):
        codes = torch.zeros(NB * 2 * atoms[0].n_bits, dtype=torch.uint8, device=dev())
        words = torch.zeros(B.words_nbytes(NB, 16), dtype=torch.uint8, device=dev())
        B.sop_pack(W, cd, fmt, atoms, codes, words, index_a=0, index_b=B.NO_ATOM, k_mode=0, container_bits=16, block_cos=metric)
        out.append((codes, words))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    if kind == "E4M3":
        assert int(((out[0][0] & 0x7F) == 0x7F).sum()) == 0           # no code that is not a number


@pytest.mark.parametrize("b", [8, 12, 16])
def test_both_packers_leave_the_same_words_where_there_is_no_pair(B, b):
    # a result without a pair: nothing is packed, a 12-bit stream is cleared, else its last 32 bits
    M, K = 37, 272
    fmt, atoms, NB = I.scale_format("UE4M3"), I.alphabet(["NF4", "SH4"]), M * K // 16
    W, cd, res = I.tiny_layer(63, M, K).W.to(dev()), torch.ones(K, device=dev()), B.new_result(dev())
    B.sop_pair_search(W, cd, fmt, atoms, B.new_pair_table(4, dev()), None, res, B.alloc_workspace(B.pair_search_workspace(M, K, 4), dev()),
                      singles_only=True, block_cos=torch.empty((4, NB), device=dev()), block_sse=torch.empty((4, NB), device=dev()))
    n, out = B.words_nbytes(NB, b), []
    for metric in (torch.zeros((4, NB), device=dev()), None):
        codes, words = torch.full((NB * 8,), 0x5A, dtype=torch.uint8, device=dev()), torch.full((n + 64,), 0x5A, dtype=torch.uint8, device=dev())
        counts = torch.zeros(2, dtype=torch.int64, device=dev())
        B.sop_pack(W, cd, fmt, atoms, codes, words, search_result=res, container_bits=b, counts=counts, block_cos=metric)
        assert counts.tolist() == [-1, -1] and bool((codes == 0x5A).all())
        out.append(words)
    assert torch.equal(out[0], out[1])
    assert int((out[0] == 0).sum()) == (n if b == 12 else 4) and bool((out[0][n:] == 0x5A).all())


@pytest.mark.parametrize("M,K", [(1, 16), (5, 112), (37, 272)])
@pytest.mark.parametrize("grid", [(3, 4, 3, 15.5), (2, 3, 1, 7.5), (2, 2, 1, 7.0), (3, 3, 3, 30.0)])      # 8, 6, 5 and 7 bits
def test_parametric_grids_in_both_packers(B, M, K, grid):
    x, y, bias, top = grid
    atoms, fmt, NB, n = [I.Atom("grid", 1 + x + y, I.KIND_FP_GRID, 0, 16, top, None, (x, y, bias, top))], I.scale_format("UE4M4"), M * K // 16, 1 + x + y
    W, cd, res = I.tiny_layer(64, M, K).W.to(dev()), torch.ones(K, device=dev()), B.new_result(dev())
    bc, bs = torch.empty((1, NB), device=dev()), torch.empty((1, NB), device=dev())
    B.sop_pair_search(W, cd, fmt, atoms, B.new_pair_table(1, dev()), None, res, B.alloc_workspace(B.pair_search_workspace(M, K, 1), dev()),
                      block_cos=bc, block_sse=bs)
    out = []
    for metric in (bc, None):
        codes, words = torch.full((NB * 2 * n + 64,), 0x5A, dtype=torch.uint8, device=dev()), torch.full((B.words_nbytes(NB, 12) + 64,), 0x5A, dtype=torch.uint8, device=dev())
        B.sop_pack(W, cd, fmt, atoms, codes, words, index_a=0, index_b=B.NO_ATOM, search_result=res, container_bits=12, block_cos=metric)
        out.append((codes, words))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
