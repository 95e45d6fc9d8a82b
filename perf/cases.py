"""The work that users of this library have it do, as measurable cases.

A case names a path through the public entry points and its sizes:
  path "layer"   one layer at one scale format, launched call by call (``pipeline.LayerSweep.run``): channel norms, search,
                 DD atom (Lloyd iterations or the dynamic programme), search of the DD columns, pack; with ``opq`` / ``wr``
                 also the two sparse streams
  path "set"     one layer at several scale formats, replayed as one graph (``pipeline.LayerSetSweep``): the unit of a model
                 sweep
  path "search"  one search through the C-ABI binding with the per-block cosines and errors as outputs: a study of the
                 design axes or of element formats that reads the per-block values itself
  path "stream"  two host-resident layers through ``pipeline.LayerStream``: pinned inputs in, packed layers and tables out

Inputs follow the generators of ``paper_2605_14929_b200.inputs`` (heavy-tailed weights, lognormal channel scales, a few
outlier channels), made on the GPU from the seed.
"""
import math

import torch

from paper_2605_14929_b200 import binding as B
from paper_2605_14929_b200 import inputs as I
from paper_2605_14929_b200.pipeline import LayerSetSweep, LayerStream, LayerSweep

ROM4 = "NF4 SH4 BOF4 Split87"
ROM5 = "NF5 SH5 BOF5 E2M2"
ALL_FORMATS = " ".join(I.TABLE_SCALE_FORMATS)


def _case(path, M, K, T, formats, rom, fp="", iters=8, weights="student", grid_dp=False, opq=False, wr=False, select_mse=False, name=None):
    c = dict(path=path, M=M, K=K, T=T, formats=formats, rom=rom, fp=fp, iters=iters, weights=weights, grid_dp=grid_dp, opq=opq, wr=wr,
             select_mse=select_mse)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one small layer, no DD atom, signed scale words; launches and host work are what it costs
        _case("layer", 256, 1024, 128, "S1E4M4", "NF4 SH4 BOF4", iters=0, weights="rows", name="small_256x1024"),
        # an odd shape: a block count that is no multiple of four, a few tokens, a 12-bit signed word
        _case("layer", 771, 1040, 37, "E4M3", "NF4 SH4", name="ragged_771x1040"),
        # the key / value projection of a large model at the widest scale word
        _case("layer", 1024, 8192, 1024, "E8M7", ROM4, weights="channels", name="kv_1024x8192_E8M7"),
        # an attention projection with outlier channels, the whole 4-bit alphabet and two element formats beside it
        _case("layer", 4096, 4096, 512, "E5M6", ROM4, fp="E2M3 E4M3", weights="outliers", name="attention_4096x4096"),
        # element formats only (a promotion-profile comparison): no pair, no DD atom, the first one is packed
        _case("layer", 14336, 4096, 512, "UE4M4", "", fp="E2M3 E4M3^0", iters=0, name="fp_14336x4096"),
        # the 5-bit extension: 32-entry tables, sixteen Lloyd iterations
        _case("layer", 4096, 14336, 2048, "UE4M4", ROM5, iters=16, weights="laplace", name="n5_4096x14336"),
        # a large layer with both sparse streams
        _case("layer", 8192, 8192, 1024, "E5M6", ROM4, weights="channels", opq=True, wr=True, name="sparse_8192x8192"),
        # the DD atom by dynamic programming
        _case("layer", 2048, 4096, 256, "UE4M6", ROM4, grid_dp=True, name="grid_dp_2048x4096"),
        # the largest layer of a 70B-shaped model
        _case("layer", 28672, 8192, 1024, "UE5M7", ROM4, weights="channels", name="large_28672x8192"),
        # a model sweep: one layer at the eight scale formats, one graph
        _case("set", 8192, 8192, 1024, ALL_FORMATS, ROM4, weights="channels", name="formats8_8192x8192"),
        # a study that reads the per-block values: blocks assigned by squared error, parametric element grids
        _case("search", 4096, 1024, 256, "E4M5", ROM4, fp="E3M4 HIF7", iters=0, select_mse=True, name="axes_4096x1024"),
        # host-resident layers, copies overlapped with the sweeps
        _case("stream", 4096, 4096, 512, "UE4M4 E5M6", ROM4, name="stream_4096x4096"),
    ]


def draw(rng):
    path = rng.choice(["layer"] * 6 + ["set", "search", "stream"])
    most = {"layer": 1 << 27, "set": 1 << 25, "search": 1 << 26, "stream": 1 << 23}[path]
    K = 16 * round(math.exp(rng.uniform(math.log(12), math.log(1024))))
    M = max(40, round(math.exp(rng.uniform(math.log(40), math.log(16384)))))
    M = max(40, min(M, most // K))
    T = round(math.exp(rng.uniform(math.log(16), math.log(2048))))
    five = rng.random() < 0.2
    pool = (ROM5 if five else ROM4).split()
    rom = " ".join(pool[:rng.randint(2, 4)])
    fp = rng.choice(["", "", "E2M3", "E2M3 E4M3", "E4M3^0"])
    iters = rng.choice([4, 8, 8, 16])
    n_fmt = rng.randint(2, 4) if path == "set" else 2 if path == "stream" else 1
    formats = " ".join(rng.sample(I.TABLE_SCALE_FORMATS, n_fmt))
    weights = rng.choice(["student", "rows", "channels", "outliers", "laplace"])
    if path == "layer":
        kind = rng.choice(["dd", "dd", "dd", "dp", "rom", "fp", "sparse"])
        if kind == "rom":
            iters = 0
        if kind == "fp":
            rom, fp, iters = "", rng.choice(["E2M3", "E4M3 E2M3", "E2M3 E4M3^0"]), 0
        return _case(path, M, K, T, formats, rom, fp, iters, weights, grid_dp=kind == "dp", opq=kind == "sparse", wr=kind == "sparse")
    if path == "search":
        return _case(path, M, K, T, formats, rom, rng.choice(["", "E3M4 HIF7", "E2M3"]), 0, weights, select_mse=rng.random() < 0.5)
    return _case(path, M, K, T, formats, rom, fp, iters, weights)


def _layer(case, seed, device):
    M, K, T, kind = case["M"], case["K"], case["T"], case["weights"]
    if kind == "laplace":
        return I.laplace_outlier_layer(seed, 0, M, K, T, device=device)
    L = I.student_layer(seed, 0, M, K, T, 4.0 if kind == "outliers" else 5.0, 0.02, 1.2 if kind == "channels" else 0.0, device)
    g = torch.Generator(device=device)
    g.manual_seed(seed + 77)
    if kind == "rows":             # lognormal(0, 0.3) row scales
        rows = torch.exp(0.3 * torch.randn((M, 1), generator=g, device=device))
        return I.Layer((L.W.float() * rows).to(torch.bfloat16), L.X)
    if kind == "outliers":         # 1 % of the input channels twenty times as large, in the weights and the activations
        gain = torch.where(torch.rand((1, K), generator=g, device=device) < 0.01, 20.0, 1.0)
        return I.Layer((L.W.float() * gain).to(torch.bfloat16), L.X * gain)
    return L


def _table(t, n):
    """A table of ``sop_pair_stat``: its two doubles and its two counts per entry, as views."""
    return t.view(torch.float64).view(n, n, 4)[..., :2], t.view(torch.int64).view(n, n, 4)[..., 2:]


def _small(sw):
    """The results of one sweep that are its own when it shares its large buffers with others.  (The four-way table has
    entries only where the scale word has a sign.)"""
    n = len(sw.full_atoms)
    out = [*_table(sw.pair_table, n), sw.result.view(torch.int32), sw.counts]
    if sw.fmt.sign_bits:
        out += _table(sw.signed_table, n)
    return out + [sw.dd_lut, sw.distortion] if sw.iters > 0 else out


def _whole(sw):
    out = _small(sw) + [sw.c, sw.codes, sw.words]
    if sw.iters > 0:
        out += [sw.pool_count, sw.rom_result.view(torch.int32)]
    if sw.opq_m is not None:
        out += [sw.W_opq, sw.opq_row_start, sw.opq_records, sw.opq_count]
    if sw.wr_keep:
        out += [sw.wr_row_start, sw.wr_records, sw.wr_count, sw.wr_exp, sw.wr_tau]
    return out


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    M, K, T, path = case["M"], case["K"], case["T"], case["path"]
    fmts = [I.scale_format(f) for f in case["formats"].split()]
    rom, fp = case["rom"].split(), case["fp"].split()
    L = _layer(case, seed, str(dev))
    if path == "layer":
        sw = LayerSweep(M, K, T, fmts[0], rom, fp, case["iters"], device=dev, grid_dp=case["grid_dp"], opq_q=0.92 if case["opq"] else None,
                        wr_sigma=0.001 if case["wr"] else None, opq_capacity=M * K // 8 if case["opq"] else None)
        return dict(path=path, sweep=sw, W=L.W, X=L.X, out=_whole(sw))
    if path == "set":
        sset = LayerSetSweep([(M, K, T)], fmts, rom, fp, case["iters"], device=dev)
        sset.capture([(L.W, L.X)])
        out = _whole(sset.sweeps[0][-1])               # the packed layer is the last format's
        for sw in sset.sweeps[0][:-1]:
            out += _small(sw)
        return dict(path=path, set=sset, W=L.W, X=L.X, out=out)
    if path == "search":
        atoms = I.alphabet(rom, with_negations=True, fp=fp)
        n, nb = len(atoms), M * (K // 16)
        s = dict(path=path, W=L.W, X=L.X, atoms=B.make_atoms(atoms), fmt=B.make_fmt(fmts[0]), select_mse=case["select_mse"],
                 c=torch.empty(K, dtype=torch.float32, device=dev), pair=B.new_pair_table(n, dev), signed=B.new_pair_table(n, dev),
                 result=B.new_result(dev), cos=torch.empty((n, nb), dtype=torch.float32, device=dev),
                 sse=torch.empty((n, nb), dtype=torch.float32, device=dev),
                 ws_norm=B.alloc_workspace(B.channel_norms_workspace(T, K), dev), ws=B.alloc_workspace(B.pair_search_workspace(M, K, n), dev))
        s["out"] = [s["c"], *_table(s["pair"], n), *_table(s["signed"], n), s["result"].view(torch.int32), s["cos"], s["sse"]]
        return s
    first, sweeps = None, []
    for f in fmts:
        sweeps.append(LayerSweep(M, K, T, f, rom, fp, case["iters"], device=dev, share=first))
        first = first or sweeps[0]
    second = _layer(case, seed + 1, str(dev))
    host = [(x.W.cpu().pin_memory(), x.X.cpu().pin_memory()) for x in (L, second)]
    return dict(path=path, stream=LayerStream(sweeps, graphs=True), host=host, n=len(first.full_atoms), done=0)


def run(state):
    path = state["path"]
    if path == "layer":
        state["sweep"].run(state["W"], state["X"])
        return state["out"]
    if path == "set":
        state["set"].replay()
        return state["out"]
    if path == "search":
        s = state
        B.sop_channel_norms(s["X"], s["c"], s["ws_norm"])
        B.sop_pair_search(s["W"], s["c"], s["fmt"], s["atoms"], s["pair"], s["signed"], s["result"], s["ws"], block_cos=s["cos"],
                          block_sse=s["sse"], select_mse=s["select_mse"])
        return s["out"]
    stream, i = state["stream"], state["done"]
    for k, (W, X) in enumerate(state["host"]):
        stream.submit(i + k, W, X)
    state["done"] = i + len(state["host"])
    got = []
    for k in range(len(state["host"])):
        for o in stream.collect(i + k):
            got += [*_table(o["pair_table"], state["n"]), *_table(o["signed_table"], state["n"]), o["result"].view(torch.int32), o["codes"],
                    o["words"], o["distortion"]]
    return got


def work(case):
    """Bytes: the weights and activations read once, the packed layer (codes and scale words) of every format -- or, for a
    search, its per-block values -- written once, the sparse streams.  Operations: per element and format 8 for the block norm
    and the scaled value, 9 per candidate (the weighted products of its cosine, and its squared error)."""
    M, K, T = case["M"], case["K"], case["T"]
    E, layers, n_fmt = M * K, 2 if case["path"] == "stream" else 1, len(case["formats"].split())
    rom, fp = case["rom"].split(), case["fp"].split()
    n_cand = 2 * len(rom) + (2 if case["iters"] > 0 else 0) + len(fp)
    bits = I.rom_atom(rom[0]).n_bits if rom else I.fp_atom(fp[0]).n_bits
    out = 8.0 * n_cand / 16.0 if case["path"] == "search" else n_fmt * (bits / 8.0 + 1.0 / 16.0)
    extra = (2.0 if case["opq"] else 0.0) + (0.004 if case["wr"] else 0.0)
    return dict(bytes=layers * (E * (2.0 + out + extra) + 4.0 * T * K), flops=float(layers * n_fmt * E * (8 + 9 * n_cand) + layers * 2 * T * K))


def tolerance(case):
    """Whole numbers (counts, chosen pairs, packed bytes, records) are the same.  Floating outputs: channel norms and the DD
    table are fp32 values rounded once from wider sums (2^-24 = 6e-8 of the value); the FP64 tables against their own fp32
    per-block values summed in 64 bits differ by at most 1.1e-8 of the value (fp32 sums of eight blocks), the distortion trace by
    less.  Four times the largest of these."""
    return {"rel": 2.5e-7, "max": 2.5e-7, "differ": 0.0}
