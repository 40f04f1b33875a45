"""The fused layer kernel cuts a layer's rows into tiles of 32, 64 or 128 per CTA by how many rows there are: row counts on either
side of every cut, with the weights in tensor memory and streamed, against the layer's definition in fp64."""
import json
import re

import pytest
import torch

import paper_2202_02365_b200 as mg
from paper_2202_02365_b200 import inputs

pytestmark = pytest.mark.gpu

N = 40_000


@pytest.fixture(scope="module")
def graph():
    return inputs.rmat_graph(N, 6 * N, seed=31)


def last_layer(view, feats, ws, wn, b):
    """One layer over a one-hop sample in fp64: self rows, mean of the sampled neighbours, linear maps."""
    h = feats[view.node_ids.long()].double()
    off, n = view.nbr_offsets.long(), view.nbr_offsets.numel() - 1
    cnt = off[1:] - off[:-1]
    dst = torch.repeat_interleave(torch.arange(n, device=h.device), cnt)
    mean = torch.zeros((n, h.shape[1]), dtype=torch.float64, device=h.device).index_add(0, dst, h[view.repr_map.long()])
    mean = mean / cnt.clamp(min=1).double()[:, None]
    return h[h.shape[0] - n:] @ ws.double().cuda() + mean @ wn.double().cuda() + b.double().cuda()


# (148 SMs: one round of 64-row tiles holds 9,472 rows, of 128-row tiles 18,944); widths with K of one to three groups
@pytest.mark.parametrize("rows", [1, 64, 65, 129, 9_472, 9_473, 18_944, 18_945, 28_417, 37_889])
@pytest.mark.parametrize("d_in,d_out,half,fanout", [(128, 256, False, 4), (256, 100, False, 9), (384, 36, True, 3)])
def test_rows_on_either_side_of_the_tile_sizes(graph, rows, d_in, d_out, half, fanout):
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    feats = inputs.normal_features(N, d_in, seed=5, device="cuda", dtype=torch.float16 if half else torch.float32)
    ctx.load_features(feats)
    (layer,) = inputs.random_bias_layers([d_in, d_out], seed=6)
    dense = ctx.sample(inputs.distinct_targets(N, rows, seed=7), [fanout], seed=8)
    out = torch.full((rows + 1, d_out), 7.0, device="cuda")
    ctx.forward(ctx.model([layer]), dense, out[:rows])
    want = last_layer(dense.view(0), feats, *layer)
    # operands rounded to 10 bits (2^-11 each), sums of up to 768 products of random sign: rms error below 1e-3 of the rows' rms, the
    # largest of 10^7 values below 6 times that
    err = (out[:rows].double() - want).abs()
    rms = want.square().mean().sqrt()
    assert float(err.square().mean().sqrt() / rms) < 1e-3 and float((err / torch.maximum(want.abs(), rms)).max()) < 6e-3
    assert torch.equal(out[rows], torch.full_like(out[rows], 7.0))


# the rows may go into the table that they are made from: it is read before any of them is there, also where the layers run over a few
# mini-batches at a time
@pytest.mark.parametrize("hops,window", [(1, 0), (2, 0), (2, 1)])
def test_rows_written_over_the_table(graph, hops, window):
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    table = inputs.normal_features(N, 128, seed=5, device="cuda")
    ctx.load_features(table)
    ctx.set_layer_window(window)
    per, count = 9_000, 4
    targets = torch.cat([inputs.distinct_targets(N, per, seed=b) for b in range(count)])
    dense = ctx.sample_many(targets, [per * b for b in range(count + 1)], [5, 4][:hops], [1, 2, 3, 4])
    model = ctx.model(inputs.random_bias_layers([128] * (hops + 1), seed=6))
    want = torch.empty((per * count, 128), device="cuda")
    ctx.forward(model, dense, want)
    got = table[1_000:1_000 + per * count]
    ctx.forward(model, dense, got)
    assert torch.equal(got, want)


# tiles of 32 rows: one row, a full tile, one more, all that the SMs take in one round of them (148 SMs: 4,736), one more
@pytest.mark.parametrize("rows", [31, 32, 33, 63, 96, 4_736, 4_737])
@pytest.mark.parametrize("d_in,d_out,half,fanout", [(128, 256, False, 4), (256, 100, False, 9), (384, 36, True, 3)])
def test_rows_on_either_side_of_the_smallest_tiles(graph, rows, d_in, d_out, half, fanout):
    test_rows_on_either_side_of_the_tile_sizes(graph, rows, d_in, d_out, half, fanout)


# layers wider than the fused kernel's go through a product of their own: by tile, or (148 SMs: from 296 blocks of 256 rows x 256 columns on)
# by persistent CTA pairs; K of one and of eight slices, a ragged last block of rows and of columns
@pytest.mark.parametrize("rows", [37_632, 37_633, 39_999])
@pytest.mark.parametrize("d_in,d_out", [(16, 300), (128, 512), (100, 260)])
def test_rows_on_either_side_of_the_persistent_product(graph, rows, d_in, d_out):
    test_rows_on_either_side_of_the_tile_sizes(graph, rows, d_in, d_out, False, 4)


def layers_over(view, feats, layers, combine):
    """Layers over one mini-batch in fp64: combine(self rows, sum over their entries, how many, layer), a ReLU on all but the last."""
    nio, rep, off = view.node_id_offsets.tolist(), view.repr_map.long(), view.nbr_offsets.long()
    h = feats[view.node_ids.long()].double()
    for l, layer in enumerate(layers):
        first, drop = nio[l + 1] - nio[l], nio[l + 1] - nio[1]
        n = h.shape[0] - first
        lo, hi, cnt = int(off[drop]), int(off[drop + n]), off[drop + 1:drop + n + 1] - off[drop:drop + n]
        dst = torch.repeat_interleave(torch.arange(n, device=h.device), cnt)
        total = torch.zeros((n, h.shape[1]), dtype=torch.float64, device=h.device).index_add(0, dst, h[rep[lo:hi] - nio[l]])
        h = combine(h[first:], total, cnt.double()[:, None], [x.double().cuda() for x in layer])
        if l + 1 < len(layers):
            h = h.relu()
    return h


def uniform_attention(own, total, count, layer):
    return (own + total) / (count + 1) @ layer[0] + layer[3]


def mean_aggregator(own, total, count, layer):
    return own @ layer[0] + total / count.clamp(min=1) @ layer[1] + layer[2]


# the persistent product with a column block narrower than 256 (other boxes, MMA shapes, tensor-memory sizes and accumulator strides), which
# takes 296 blocks of 256 rows (148 SMs): the last row count by tile, one more, a ragged last block; K of a part of a slice to eight slices.
# An attention layer without attention is such a product of the rows' means.
@pytest.mark.parametrize("rows", [75_520, 75_521, 75_777])
@pytest.mark.parametrize("d_in,d_out", [(16, 4), (100, 16), (256, 36), (32, 96), (100, 100), (64, 132), (256, 200), (36, 224)])
def test_narrow_persistent_product(graph, rows, d_in, d_out):
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    feats = inputs.normal_features(N, d_in, seed=5, device="cuda")
    ctx.load_features(feats)
    ((w, _, b),) = inputs.random_bias_layers([d_in, d_out], seed=6)
    layer = (w, torch.zeros(d_out), torch.zeros(d_out), b)
    offs = [0, 38_000, rows]
    targets = torch.cat([inputs.distinct_targets(N, hi - lo, seed=lo) for lo, hi in zip(offs[:-1], offs[1:])])
    dense = ctx.sample_many(targets, offs, [3], [1, 2])
    out = torch.full((rows + 1, d_out), 7.0, device="cuda")
    ctx.gat_forward(ctx.gat_model([layer]), dense, out[:rows])
    want = torch.cat([layers_over(dense.view(i), feats, [layer], uniform_attention) for i in range(2)])
    # (as above: operands rounded to 10 bits, sums of up to 256 products)
    err, rms = (out[:rows].double() - want).abs(), want.square().mean().sqrt()
    assert float(err.square().mean().sqrt() / rms) < 1e-3 and float((err / torch.maximum(want.abs(), rms)).max()) < 6e-3
    assert torch.equal(out[rows], torch.full_like(out[rows], 7.0))


# the same product with a ReLU: the first of two layers, one wider than the fused kernel's and one of attention
@pytest.mark.parametrize("dims,attention", [([16, 300, 8], False), ([16, 100, 8], True), ([36, 320, 8], True)])
def test_persistent_product_before_a_relu(graph, dims, attention):
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    feats = inputs.normal_features(N, dims[0], seed=5, device="cuda")
    ctx.load_features(feats)
    layers = inputs.random_bias_layers(dims, seed=6)
    if attention:
        layers = [(w, torch.zeros_like(b), torch.zeros_like(b), b) for w, _, b in layers]
    per = 30_000
    targets = torch.cat([inputs.distinct_targets(N, per, seed=b) for b in range(3)])
    dense = ctx.sample_many(targets, [0, per, 2 * per, 3 * per], [3, 2], [1, 2, 3])
    assert int(dense.counts()[0][:, :2].sum()) > 75_520       # rows of the first layer
    out = torch.empty((3 * per, dims[-1]), device="cuda")
    if attention:
        ctx.gat_forward(ctx.gat_model(layers), dense, out)
    else:
        ctx.forward(ctx.model(layers), dense, out)
    want = torch.cat([layers_over(dense.view(i), feats, layers, uniform_attention if attention else mean_aggregator) for i in range(3)])
    # two layers, each with operands rounded to 10 bits: the bounds above twice
    err, rms = (out.double() - want).abs(), want.square().mean().sqrt()
    assert float(err.square().mean().sqrt() / rms) < 2e-3 and float((err / torch.maximum(want.abs(), rms)).max()) < 12e-3


# few rows of one mini-batch: the layers' kernels look the rows up in the sample themselves; a second mini-batch of one node makes them use
# the table made before, and the rows are the same bit for bit.  One to three hops, empty hops, a table in slots of a buffer
@pytest.mark.parametrize("rows,fanouts", [(1, [3]), (33, [9, 4]), (700, [5, 3, 2]), (2_000, [0, 2]), (4_737, [2])])
@pytest.mark.parametrize("slots", [False, True])
def test_rows_looked_up_by_the_layers(graph, rows, fanouts, slots):
    if 0 in fanouts:
        graph = inputs.build_csr(torch.tensor([3]), torch.tensor([4]), N)      # (no neighbours to speak of)
        fanouts = [1] * len(fanouts)
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.set_partitioning(4)
    feats = inputs.normal_features(N, 36, seed=5)
    if slots:
        ctx.load_features(feats.pin_memory(), capacity_parts=3, backing=mg.BACKING_HOST)
        ctx.set_resident([3, 0, 2])
        pool = torch.cat([torch.arange(0, N // 4), torch.arange(N // 2, N)])
    else:
        ctx.load_features(feats.cuda(), capacity_parts=4)
        ctx.set_resident([0, 1, 2, 3])
        pool = torch.arange(N)
    ids = pool[torch.randperm(len(pool), generator=torch.Generator().manual_seed(rows))[:rows + 1]].to(torch.int32)
    dims = [36] + [64] * (len(fanouts) - 1) + [20]
    model = ctx.model(inputs.random_bias_layers(dims, seed=6))
    one, two = torch.empty((rows, 20), device="cuda"), torch.empty((rows + 1, 20), device="cuda")
    before = ctx.kernel_launches()
    ctx.forward(model, ctx.sample(ids[:rows], fanouts, seed=8), one)
    alone = ctx.kernel_launches() - before
    ctx.forward(model, ctx.sample_many(ids, [0, rows, rows + 1], fanouts, [8, 9]), two)
    assert torch.equal(one, two[:rows])
    assert ctx.kernel_launches() - before - alone > alone


# the backward pass of such a pass makes the table itself
def test_backward_behind_rows_looked_up_by_the_layers(graph):
    got = []
    for keep in (False, True):
        ctx = mg.Context(0)
        ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
        ctx.load_features(inputs.normal_features(N, 36, seed=5, device="cuda"))
        ctx.keep_layer_outputs(keep)
        model = ctx.model(inputs.random_bias_layers([36, 64, 20], seed=6))
        dense = ctx.sample(inputs.distinct_targets(N, 500, seed=7), [5, 3], seed=8)
        ctx.forward(model, dense, torch.empty((500, 20), device="cuda"))
        got.append(ctx.backward(model, dense, inputs.normal_features(500, 20, seed=9, device="cuda")))
    for a, b in zip(*got):
        for x, y in zip(a, b):      # the same products of operands rounded to ten bits, summed in another order: a few 2^-24 of the norm
            assert float((x.double() - y.double()).norm() / y.double().norm()) < 1e-5


# rows of 9 to 16 entries on average keep their weights in tensor memory where the outputs are narrow, and stream them where they are not or where
# the rows are longer; against the streamed form, bit for bit, and the definition
@pytest.mark.parametrize("d_in,d_out", [(100, 100), (128, 128), (32, 4), (64, 132)])
@pytest.mark.parametrize("fanout", [12, 40])
def test_long_rows_of_narrow_outputs(monkeypatch, d_in, d_out, fanout):
    g = inputs.erdos_renyi_graph(N, 22 * N, seed=33)
    ctx = mg.Context(0)
    ctx.load_graph(g.row_offsets.cuda(), g.nbrs.cuda())
    feats = inputs.normal_features(N, d_in, seed=5, device="cuda")
    ctx.load_features(feats)
    (layer,) = inputs.random_bias_layers([d_in, d_out], seed=6)
    rows = 20_001
    dense = ctx.sample(inputs.distinct_targets(N, rows, seed=7), [fanout], seed=8)
    out, streamed = torch.empty((rows, d_out), device="cuda"), torch.empty((rows, d_out), device="cuda")
    ctx.forward(ctx.model([layer]), dense, out)
    monkeypatch.setenv("MG_FUSED_NO_TS", "1")
    ctx.forward(ctx.model([layer]), dense, streamed)
    assert torch.equal(out, streamed)
    want = last_layer(dense.view(0), feats, *layer)
    # (operands rounded to 10 bits: as in test_rows_on_either_side_of_the_tile_sizes)
    assert float((out.double() - want).norm() / want.norm()) < 1e-3


# the same of fp16 rows, of intermediates kept as fp16, of the sum and of both lists
@pytest.mark.parametrize("half,between,aggregator,direction", [(True, False, "mean", "in"), (False, True, "mean", "in"), (True, True, "mean", "inout"),
                                                               (False, False, "sum", "in"), (True, False, "sum", "inout")])
@pytest.mark.parametrize("rows", [1, 700, 1_300])
def test_rows_looked_up_by_the_layers_in_every_form(graph, rows, half, between, aggregator, direction):
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    if direction == "inout":
        other = inputs.transpose_csr(graph)
        ctx.load_out_graph(other.row_offsets.cuda(), other.nbrs.cuda())
        ctx.set_sample_direction(direction)
    ctx.load_features(inputs.normal_features(N, 72, seed=5, device="cuda", dtype=torch.float16 if half else torch.float32))
    ids = inputs.distinct_targets(N, rows + 1, seed=rows)
    model = ctx.model(inputs.random_bias_layers([72, 128, 20], seed=6))
    model.set_intermediates(torch.float16 if between else torch.float32)
    model.set_aggregator(aggregator)
    one, two = torch.empty((rows, 20), device="cuda"), torch.empty((rows + 1, 20), device="cuda")
    alone, both = ctx.sample(ids[:rows], [3, 2], seed=8), ctx.sample_many(ids, [0, rows, rows + 1], [3, 2], [8, 9])
    launches = [ctx.kernel_launches()]
    for dense, out in ((alone, one), (both, two)):
        ctx.forward(model, dense, out)
        launches.append(ctx.kernel_launches())
    assert torch.equal(one, two[:rows])
    assert launches[1] - launches[0] == 2 and launches[2] - launches[1] == 3      # (two layers; the table and two layers)


def layers_launched(call, tmp_path):
    """Template arguments (FIRST, HALF, F16, TS, ROWS, KEEP) of every layer kernel that `call` launches."""
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    prof.export_chrome_trace(str(tmp_path / "trace.json"))
    events = [e for e in json.load(open(tmp_path / "trace.json"))["traceEvents"] if e.get("cat") == "kernel" and "k_sage_layer_fused" in e["name"]]
    return [re.search(r"k_sage_layer_fused<(.*?)>", e["name"]).group(1).split(", ") for e in sorted(events, key=lambda e: e["ts"])]


# which layers keep their weights in tensor memory: rows of exactly as many entries as the rule allows and of one more; of 9 to 16, tiles of every height
# with one of them per CTA and several, two slices of weights and more, widths on either side of the rule's, fp16 rows and intermediates, layers that keep their
# outputs.  Where they are kept there, bit for bit what the streamed form gives.
@pytest.mark.parametrize("rows,tile", [(1_000, 32), (9_472, 64), (18_901, 128), (18_945, 64), (28_417, 128)])
@pytest.mark.parametrize("form,d_in,d_out,entries,kept", [
    ("fp32", 100, 128, 8, "yyyyy"), ("fp32", 100, 132, 8, "yyyyy"), ("fp32", 100, 132, 9, "nnnnn"), ("fp32", 100, 112, 16, "yyyyy"), ("fp32", 100, 112, 17, "nnnnn"),
    ("fp32", 100, 128, 9, "nnnyy"), ("fp32", 64, 128, 9, "ynnyy"), ("fp32", 32, 64, 9, "ynnnn"), ("fp32", 32, 100, 9, "ynnyy"), ("fp16", 256, 128, 16, "ynnyy"),
    ("fp16", 256, 64, 9, "yyyyy"), ("later", 32, 128, 9, "ynnyy"), ("later", 64, 128, 9, "yyyyy"), ("fp16 later", 128, 128, 16, "yyyyy"), ("kept", 64, 64, 9, "yynyn"),
    ("kept", 128, 64, 9, "yyyyy")])
def test_weights_in_tensor_memory_by_entries_and_width(monkeypatch, tmp_path, rows, tile, form, d_in, d_out, entries, kept):
    kept = kept[[1_000, 9_472, 18_901, 18_945, 28_417].index(rows)] == "y"
    half, later = "fp16" in form, form in ("later", "fp16 later", "kept")
    gen = torch.Generator().manual_seed(entries)
    g = inputs.build_csr(torch.randint(N, (N * entries,), generator=gen), torch.arange(N).repeat_interleave(entries), N)
    ctx = mg.Context(0)
    ctx.load_graph(g.row_offsets.cuda(), g.nbrs.cuda())
    width = 64 if later else d_in
    ctx.load_features(inputs.normal_features(N, width, seed=5, device="cuda", dtype=torch.float16 if half else torch.float32))
    ctx.keep_layer_outputs(form == "kept")
    model = ctx.model(inputs.random_bias_layers([width, d_in, d_out] if later else [width, d_out], seed=6))
    model.set_intermediates(torch.float16 if half else torch.float32)
    dense = ctx.sample(inputs.distinct_targets(N, rows, seed=7), [entries, 2] if later else [entries], seed=8)
    out, streamed = torch.empty((rows, d_out), device="cuda"), torch.empty((rows, d_out), device="cuda")
    last = layers_launched(lambda: ctx.forward(model, dense, out), tmp_path)[-1]
    assert last == [str(x).lower() for x in (not later, half, half, kept, tile, form == "kept")], last
    if kept:
        monkeypatch.setenv("MG_FUSED_NO_TS", "1")
        assert layers_launched(lambda: ctx.forward(model, dense, streamed), tmp_path)[-1][3] == "false"
        assert torch.equal(out, streamed)
