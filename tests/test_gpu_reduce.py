"""The reduction of the per-block values into table entries, recomputed in FP64 from the per-block arrays of the same call: block
counts around a tile of 256 or 768 blocks and around one tile per SM, rows of the columns that start off a 16-byte boundary, and
alphabets whose entries make every kind of bundle (a rest of one, two or three candidates, one second candidate, many)."""
import numpy as np
import pytest
import torch

from paper_2605_14929_b200 import inputs as I

from .test_gpu_parity import B, dev  # noqa: F401  (B is a fixture)

pytestmark = pytest.mark.gpu

# fp32 sums of eight gaps or errors (relative 8 * 2^-24 of non-negative terms), everything after them in FP64
TOL = 8 * 2.0 ** -24


def _expect(cos, sse, atoms, signed, by_error):
    def pick(second, first):
        return sse[second] < sse[first] if by_error else cos[second] > cos[first]
    A, pair, four = len(atoms), {}, {}
    lut = [a.kind == I.KIND_LUT for a in atoms]
    for a in range(A):
        for b in range(a, A):
            if a != b and not (lut[a] and lut[b] and atoms[a].n_bits == atoms[b].n_bits):
                continue
            mu = pick(b, a)
            pair[a, b] = (np.where(mu, cos[b], cos[a]), np.where(mu, sse[b], sse[a]), int(mu.sum()), 0)
    base = [i for i in range(A - 1) if lut[i] and not atoms[i].negated and atoms[i + 1].negated] if signed else []
    best = {}
    for i in base:
        neg = pick(i + 1, i)
        best[i] = (np.where(neg, cos[i + 1], cos[i]), np.where(neg, sse[i + 1], sse[i]), neg)
    for x, i in enumerate(base):
        for j in base[x:]:
            (ci, ei, ni), (cj, ej, nj) = best[i], best[j]
            mu = (ej < ei if by_error else cj > ci) if i != j else np.zeros(len(ci), bool)
            four[i, j] = (np.where(mu, cj, ci), np.where(mu, ej, ei), int(mu.sum()), int(np.where(mu, nj, ni).sum()))
    return pair, four


@pytest.mark.parametrize("M,K", [(1, 16), (3, 64), (17, 240), (48, 256), (61, 1040), (1776, 1024), (1777, 1040)])
@pytest.mark.parametrize("rom,fp,by_error", [(["NF4"], [], False), (["NF4", "SH4", "BOF4", "Split87"], ["E2M3", "E4M3"], False),
                                             (["NF4", "SH4", "BOF4"], ["E2M3"], True)])
def test_table_entries_match_the_per_block_values(B, M, K, rom, fp, by_error):
    L = I.student_layer(5, 0, M, K, 4, 4.0, device="cuda")
    atoms = I.alphabet(rom, fp=fp)
    A, NB = len(atoms), M * K // 16
    c = torch.rand(K, device=dev()) + 0.1
    for fmt_name in ("E5M6", "UE4M4"):
        fmt = I.scale_format(fmt_name)
        pt, st, res = B.new_pair_table(A, dev()), B.new_pair_table(A, dev()), B.new_result(dev())
        bc, bs = torch.empty((A, NB), device=dev()), torch.empty((A, NB), device=dev())
        B.sop_pair_search(L.W, c, fmt, atoms, pt, st, res, B.alloc_workspace(B.pair_search_workspace(M, K, A), dev()), block_cos=bc, block_sse=bs,
                          select_mse=by_error)
        P, S = B.read_pair_table(pt, A), B.read_pair_table(st, A)
        pair, four = _expect(bc.cpu().numpy(), bs.cpu().numpy(), atoms, bool(fmt.sign_bits), by_error)
        for table, want in ((P, pair), (S, four)):
            for a in range(A):
                for b in range(A):
                    if (a, b) not in want:
                        assert table[a, b]["n_sel1"] == -1
                        continue
                    wc, we, n1, nn = want[a, b]
                    got = table[a, b]
                    assert (got["n_sel1"], got["n_neg"]) == (n1, nn), (a, b)
                    gap = 1.0 - wc.astype(np.float64)
                    assert abs((1.0 - got["acos"]) - gap.mean()) <= TOL * np.abs(gap).mean() + 4e-16, (a, b)
                    assert got["mse"] == pytest.approx(we.astype(np.float64).sum() / (M * K), rel=TOL), (a, b)


# more blocks than a lane of the reduction counts in 12 bits at one CTA per SM: with two candidates where as many CTAs as 12 bits
# ask for would not find room in the workspace (137,871,360 blocks), with sixteen where a warp has a bundle for itself
@pytest.mark.parametrize("M,K,tables", [(135300, 16384, 1), (20500, 16384, 8)])
def test_more_blocks_than_a_lane_counts_at_once(B, M, K, tables):
    rng = np.random.default_rng(4)
    bases = [I.rom_atom("NF4")] + [I.Atom(f"r{i}", 4, I.KIND_LUT, 0, 16, 1.0, np.sort(np.concatenate([[-1.0, 1.0], I.snap_bf16(rng.uniform(-0.95, 0.95, 14))]).astype(np.float32)))
                                   for i in range(tables - 1)]
    atoms = [x for a in bases for x in (a, a.negation())]
    A, NB = len(atoms), M * K // 16
    W = torch.randn((M, K), dtype=torch.bfloat16, device=dev(), generator=torch.Generator(device=dev()).manual_seed(1))
    c = torch.rand(K, device=dev(), generator=torch.Generator(device=dev()).manual_seed(2)) + 0.1
    pt, st, res = B.new_pair_table(A, dev()), B.new_pair_table(A, dev()), B.new_result(dev())
    bc, bs = torch.empty((A, NB), device=dev()), torch.empty((A, NB), device=dev())
    need = B.pair_search_workspace(M, K, A)
    ws = B.alloc_workspace(need + (1 << 22), dev())
    ws[need:] = 0x5A
    B.sop_pair_search(W, c, I.scale_format("E5M6"), atoms, pt, st, res, ws, block_cos=bc, block_sse=bs)
    P, S = B.read_pair_table(pt, A), B.read_pair_table(st, A)
    assert bool((ws[need:] == 0x5A).all())

    def entry(got, mu, x, y, n1, nn):
        cos = torch.where(mu, bc[y], bc[x])
        assert (got["n_sel1"], got["n_neg"]) == (n1, nn)
        assert abs(got["acos"] - float(cos.double().mean())) <= TOL * (1.0 - got["acos"]) + 1e-15
        assert got["mse"] == pytest.approx(float(torch.where(mu, bs[y], bs[x]).double().sum()) / (M * K), rel=TOL)
    for x in range(A):
        entry(P[x, x], torch.zeros(1, dtype=torch.bool, device=dev()), x, x, 0, 0)
        for y in range(x + 1, A):
            mu = bc[y] > bc[x]
            if y == x + 1 or tables == 1:
                entry(P[x, y], mu, x, y, int(mu.sum()), 0)
            else:
                assert P[x, y]["n_sel1"] == int(mu.sum())
    for x in range(0, A, 2):
        neg = bc[x + 1] > bc[x]
        entry(S[x, x], neg, x, x + 1, 0, int(neg.sum()))
        for y in range(x + 2, A, 2):
            negy = bc[y + 1] > bc[y]
            mu = torch.maximum(bc[y], bc[y + 1]) > torch.maximum(bc[x], bc[x + 1])
            assert (S[x, y]["n_sel1"], S[x, y]["n_neg"]) == (int(mu.sum()), int(torch.where(mu, negy, neg).sum()))


@pytest.mark.parametrize("M,K", [(3, 64), (2048, 4096)])
def test_a_call_that_forms_no_entry_keeps_the_tables(B, M, K):
    # every candidate loaded and every entry kept: the call closes over what an earlier one left (more than four tiles per CTA)
    L = I.student_layer(6, 0, M, K, 4, 4.0, device="cuda")
    atoms = I.alphabet(["NF4", "SH4"], fp=["E2M3"])
    A, NB = len(atoms), M * K // 16
    c = torch.rand(K, device=dev()) + 0.1
    pt, st, res, again = B.new_pair_table(A, dev()), B.new_pair_table(A, dev()), B.new_result(dev()), B.new_result(dev())
    bc, bs = torch.empty((A, NB), device=dev()), torch.empty((A, NB), device=dev())
    ws = B.alloc_workspace(B.pair_search_workspace(M, K, A), dev())
    B.sop_pair_search(L.W, c, I.scale_format("E5M6"), atoms, pt, st, res, ws, block_cos=bc, block_sse=bs)
    before = [t.clone() for t in (pt, st, bc, bs)]
    for kw in (dict(k_mode=B.K_FROM_RESULT, prev_result=res), dict()):
        again.zero_()
        B.sop_pair_search(L.W, c, I.scale_format("E5M6"), atoms, pt, st, again, ws, block_cos=bc, block_sse=bs, eval_mask=0,
                          load_mask=(1 << A) - 1, keep_loaded=True, **kw)
        assert all(torch.equal(x, y) for x, y in zip(before, (pt, st, bc, bs)))
        assert torch.equal(again, res)


@pytest.mark.parametrize("kind", ["NF4", "E4M3"])
def test_blocks_beyond_two_to_the_thirty(B, kind):
    # the byte offset of a block in a column passes 32 bits: only a few rows hold weights, among them some beyond 2^30, and each must
    # get its own value (43 GB)
    M, K = (1 << 30) + 64, 16
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB of device memory")
    rows = torch.tensor([0, 1, 5, 63, 64, (1 << 29) + 3, (1 << 30) - 1, 1 << 30, (1 << 30) + 1, (1 << 30) + 5, (1 << 30) + 63], device=dev())
    few = torch.randn((len(rows), K), device=dev(), generator=torch.Generator(device=dev()).manual_seed(7)).to(torch.bfloat16)
    W = torch.zeros((M, K), dtype=torch.bfloat16, device=dev())
    W[rows] = few
    c = torch.rand(K, device=dev(), generator=torch.Generator(device=dev()).manual_seed(8)) + 0.1
    atoms, out = [I.rom_atom("NF4") if kind == "NF4" else I.fp_atom("E4M3")], []
    for Wx in (few, W):
        NB = Wx.shape[0]
        pt, st, res = B.new_pair_table(1, dev()), B.new_pair_table(1, dev()), B.new_result(dev())
        bc, bs = torch.full((1, NB), -7.0, device=dev()), torch.full((1, NB), -7.0, device=dev())
        B.sop_pair_search(Wx, c, I.scale_format("E8M7"), atoms, pt, st, res, B.alloc_workspace(B.pair_search_workspace(NB, K, 1), dev()),
                          k_mode=0, block_cos=bc, block_sse=bs)
        out.append((bc, bs))
    for small, large in zip(*out):
        assert torch.equal(large[0, rows], small[0])
    rest = torch.ones(M, dtype=torch.bool, device=dev())
    rest[rows] = False
    assert bool((out[1][0][0][rest] == 1.0).all()) and not bool(out[1][1][0][rest].any())           # zero blocks: cosine 1, error 0
    assert B.read_pair_table(pt, 1)[0, 0]["mse"] == pytest.approx(float(out[0][1].double().sum()) / (M * K), rel=TOL)
