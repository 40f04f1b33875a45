"""The backward pass at the sizes where its gather is cut differently: source rows named by none, a few, tens and hundreds of
entries (a star graph's centre), widths of one to eight column blocks; against the layers' definition in fp64."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2202_02365_b200 as mg
from paper_2202_02365_b200 import api, inputs

pytestmark = pytest.mark.gpu

N = 6_000


def star_graph():
    """Node v aggregates from the centres 0 .. 3 by its id's divisors and from two nodes of a random graph; 0 from 20 others."""
    g = torch.Generator().manual_seed(3)
    v = torch.arange(4, N)
    dst = [v, v[::5], v[::40], v[::300], v, v, torch.zeros(20, dtype=torch.int64)]
    src = [torch.full_like(x, c) for c, x in enumerate(dst[:4])]
    src += [torch.randint(4, N, (len(v),), generator=g) for _ in range(2)] + [torch.arange(100, 120)]
    return inputs.build_csr(torch.cat(src), torch.cat(dst), N)


def reference(views, feats, layers, d_outs, aggregator):
    """Loss sum(d_out * H^k) differentiated by torch in fp64: weight gradients, and the rows' gradients by (mini-batch, node)."""
    params = [[p.double().requires_grad_() for p in layer] for layer in layers]
    rows, loss = [], 0.0
    for v, d_out in zip(views, d_outs):
        ids, nio = v.node_ids.cpu().long(), v.node_id_offsets.cpu().tolist()
        rep, off = v.repr_map.cpu().long(), v.nbr_offsets.cpu().long()
        h = feats[ids].double().requires_grad_()
        rows.append((ids, h))
        for l, (ws, wn, b) in enumerate(params):
            first = nio[l + 1] - nio[l]                  # rows of the farthest delta that is left: inputs only
            drop = nio[l + 1] - nio[1]                   # sampled nodes that are inputs only by now
            n_out = h.shape[0] - first
            lo, hi = off[drop], off[drop + n_out]
            cnt = off[drop + 1:drop + n_out + 1] - off[drop:drop + n_out]
            dst = torch.repeat_interleave(torch.arange(n_out), cnt)
            agg = torch.zeros((n_out, h.shape[1]), dtype=torch.float64).index_add(0, dst, h[rep[lo:hi] - nio[l]])
            if aggregator == "mean":
                agg = agg / cnt.clamp(min=1).double()[:, None]
            h = h[first:] @ ws + agg @ wn + b
            if l + 1 < len(params):
                h = torch.relu(h)
        loss = loss + (h * d_out.double().cpu()).sum()
    loss.backward()
    return params, rows


@pytest.mark.parametrize("dims,fanouts,aggregator", [([16, 8], [6], "mean"), ([132, 128, 12], [6, 4], "mean"), ([16, 260, 8], [6, 6], "sum"),
                                                     ([1024, 516, 4], [5, 6], "mean")])
def test_source_rows_named_by_few_and_by_many(dims, fanouts, aggregator):
    graph = star_graph()
    feats = inputs.normal_features(N, dims[0], seed=4)
    layers = inputs.random_bias_layers(dims, seed=5)
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.load_features(feats.cuda())
    ctx.keep_layer_outputs(True)
    sizes = [700, 0, 1, 90]
    targets = torch.cat([inputs.distinct_targets(N, s, seed=8 + i) for i, s in enumerate(sizes)])
    offs = np.concatenate([[0], np.cumsum(sizes)])
    dense = ctx.sample_many(targets, offs, fanouts, [1, 2, 3, 4])
    model = ctx.model(layers, mg.GEMM_FP32)
    model.set_aggregator(aggregator)
    out = torch.empty((len(targets), dims[-1]), device="cuda")
    ctx.forward(model, dense, out)
    d_out = torch.randn(out.shape, generator=torch.Generator("cuda").manual_seed(6), device="cuda")
    grads, g_rows, ids = ctx.backward(model, dense, d_out, want_h0_grad=True)
    views = [dense.view(b) for b in range(len(sizes))]
    params, rows = reference(views, feats, layers, [d_out[offs[b]:offs[b + 1]] for b in range(len(sizes))], aggregator)

    # fp32 sums of up to 800 rows x 700 entries' products in any order: sqrt(n) 2^-24 of the terms' norm, below 1e-5; where terms
    # cancel the result's norm is smaller, hence 1e-4
    def near(x, y):
        return float((x.double().cpu() - y).norm()) <= 1e-4 * max(float(y.norm()), 1e-12)

    for got, want in zip(grads, params):
        for x, p in zip(got, want):
            assert near(x.reshape(p.shape), p.grad)
    at = 0
    nodes, _ = dense.counts()
    for b, (want_ids, h) in enumerate(rows):
        n = int(nodes[b].sum())
        order = torch.argsort(ids[at:at + n].cpu())
        want = torch.argsort(want_ids)
        assert torch.equal(ids[at:at + n].cpu()[order].long(), want_ids[want])
        if n:
            assert near(g_rows[at:at + n].cpu()[order], h.grad[want])
            for i in torch.nonzero(want_ids[want] < 4).flatten().tolist():      # the centres' rows one by one
                assert near(g_rows[at:at + n].cpu()[order][i], h.grad[want][i])
        at += n


# one layer (no ReLU whose branch could differ): rows around a block of 32, around the rows that one CTA takes; widths of one to three
# groups of input columns and one to three tiles of output columns
@pytest.mark.parametrize("rows", [1, 31, 33, 257, 5_990])
@pytest.mark.parametrize("d_in,d_out,half,aggregator", [(4, 4, False, "mean"), (128, 256, False, "mean"), (132, 300, False, "sum"), (264, 36, True, "mean"),
                                                        (260, 516, False, "mean")])
def test_weight_gradients_on_the_tensor_cores(rows, d_in, d_out, half, aggregator):
    graph = star_graph()
    feats = inputs.normal_features(N, d_in, seed=4, dtype=torch.float16 if half else torch.float32)
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.load_features(feats.cuda())
    ctx.keep_layer_outputs(True)
    layers = inputs.random_bias_layers([d_in, d_out], seed=5)
    model = ctx.model(layers)
    model.set_aggregator(aggregator)
    dense = ctx.sample(inputs.distinct_targets(N, rows, seed=6), [6], 7)
    out = torch.empty((rows, d_out), device="cuda")
    ctx.forward(model, dense, out)
    d_out_rows = torch.randn(out.shape, generator=torch.Generator("cuda").manual_seed(8), device="cuda")
    grads, g_rows, ids = ctx.backward(model, dense, d_out_rows, want_h0_grad=True)
    (want,), ((want_ids, h),) = reference([dense.view(0)], feats.float(), layers, [d_out_rows], aggregator)
    # the tensor cores drop what is beyond ten bits of an operand that was not rounded before (gradient rows, the weights of dX): up to
    # 2^-10 relative for each of the two, all in one direction where a row stands alone, so 2^-9 of the result's norm
    for x, p in zip(grads[0], want):
        assert float((x.double().cpu().reshape(p.shape) - p.grad).norm()) <= 2 ** -9 * float(p.grad.norm())
    order, want_order = torch.argsort(ids.cpu()), torch.argsort(want_ids)
    assert float((g_rows.double().cpu()[order] - h.grad[want_order]).norm()) <= 2 ** -9 * float(h.grad.norm())


# the row metadata and the kept outputs are the old sample's: with another sample in the handle they would be read past their end
@pytest.mark.parametrize("precision", [mg.GEMM_TF32, mg.GEMM_FP32])
@pytest.mark.parametrize("fails", [False, True])
def test_sample_between_forward_and_backward_is_refused(precision, fails):
    graph = star_graph()
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.load_features(inputs.normal_features(N, 16, seed=4).cuda())
    ctx.keep_layer_outputs(True)
    model = ctx.model(inputs.random_bias_layers([16, 8], seed=5), precision)
    dense = ctx.sample(inputs.distinct_targets(N, 40, seed=6), [6], 7)
    out = torch.empty((40, 8), device="cuda")
    ctx.forward(model, dense, out)
    if fails:                                                # a sample that ends in an error leaves nothing to go back through either
        with pytest.raises(mg.MgError):
            ctx.sample(torch.tensor([1, 1], dtype=torch.int32), [6], 7, out=dense)
    else:
        ctx.sample(inputs.distinct_targets(N, 40, seed=6), [6], 8, out=dense)
    with pytest.raises(mg.MgError) as e:
        ctx.backward(model, dense, torch.ones_like(out))
    assert e.value.code == -2                                # MG_ERR_STATE
    if not fails:
        ctx.forward(model, dense, out)
        ctx.backward(model, dense, torch.ones_like(out))


# a wait of the scan that cuts the entry lists runs out (here at once): an error, and a context that goes on working
@pytest.mark.parametrize("precision", [mg.GEMM_TF32, mg.GEMM_FP32])
def test_scan_that_gives_up_ends_in_an_error(monkeypatch, precision):
    graph = star_graph()
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.load_features(inputs.normal_features(N, 16, seed=4).cuda())
    ctx.keep_layer_outputs(True)
    model = ctx.model(inputs.random_bias_layers([16, 12, 8], seed=5), precision)
    dense = ctx.sample(inputs.distinct_targets(N, 5_000, seed=6), [6, 4], 7)      # (more source rows than a tile of the scan has, 4,096)
    out = torch.empty((5_000, 8), device="cuda")
    ctx.forward(model, dense, out)
    d_out = torch.randn(out.shape, generator=torch.Generator("cuda").manual_seed(8), device="cuda")
    want, want_rows, _ = ctx.backward(model, dense, d_out, want_h0_grad=True)
    monkeypatch.setenv("MG_REV_POLLS", "0")
    with pytest.raises(mg.MgError, match="entry lists") as e:
        ctx.backward(model, dense, d_out, want_h0_grad=True)
    assert e.value.code == -7                                                     # MG_ERR_TIMEOUT
    monkeypatch.delenv("MG_REV_POLLS")
    got, got_rows, _ = ctx.backward(model, dense, d_out, want_h0_grad=True)
    for x, y in zip([t for layer in got for t in layer] + [got_rows], [t for layer in want for t in layer] + [want_rows]):
        assert float((x - y).norm()) <= 1e-5 * float(y.norm())                    # (sums over rows meet in any order)


# no memory for the pass's rows: it frees smaller buffers before it fails, and what it leaves is not to be gone back through
def test_backward_after_a_failed_forward_is_refused():
    graph = star_graph()
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.load_features(inputs.normal_features(N, 16, seed=4).cuda())
    ctx.keep_layer_outputs(True)
    model = ctx.model(inputs.random_bias_layers([16, 1024], seed=5))
    few, many = (ctx.sample(inputs.distinct_targets(N, n, seed=6), [6], 7) for n in (40, 5_990))
    out = torch.empty((5_990, 1024), device="cuda")
    d_out = torch.ones_like(out)
    ctx.forward(model, few, out)
    ctx.backward(model, few, d_out)
    held = []
    try:
        for size in (torch.cuda.mem_get_info()[0] - (64 << 20), 8 << 20, 2 << 20):
            try:
                while True:
                    held.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
            except torch.OutOfMemoryError:
                pass
        with pytest.raises(mg.MgError) as e:
            ctx.forward(model, many, out)                    # (24 MB of rows)
        assert e.value.code == -6                            # MG_ERR_OOM
    finally:
        held.clear()
        torch.cuda.empty_cache()
    for dense in (few, many):
        with pytest.raises(mg.MgError) as e:
            ctx.backward(model, dense, d_out)
        assert e.value.code == -2                            # MG_ERR_STATE
        with pytest.raises(mg.MgError):
            ctx.layer_output(model, dense, 1, 0, 40)
    ctx.forward(model, many, out)
    ctx.backward(model, many, d_out)


# the rows' gradients may go where the loss's gradient lies: it is read before any of them is written (rows named by hundreds of entries
# are cleared before they are added up)
@pytest.mark.parametrize("precision", [mg.GEMM_TF32, mg.GEMM_FP32])
@pytest.mark.parametrize("dims", [[16, 16], [16, 12, 16]])
def test_row_gradients_over_the_output_gradient(precision, dims):
    graph = star_graph()
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.load_features(inputs.normal_features(N, dims[0], seed=4).cuda())
    ctx.keep_layer_outputs(True)
    model = ctx.model(inputs.random_bias_layers(dims, seed=5), precision)
    dense = ctx.sample(inputs.distinct_targets(N, 4_000, seed=6), [6] * (len(dims) - 1), 7)
    out = torch.empty((4_000, dims[-1]), device="cuda")
    ctx.forward(model, dense, out)
    d_out = torch.randn(out.shape, generator=torch.Generator("cuda").manual_seed(8), device="cuda")
    want, want_rows, _ = ctx.backward(model, dense, d_out, want_h0_grad=True)
    both = torch.zeros(want_rows.numel(), device="cuda")
    both[:d_out.numel()] = d_out.flatten()
    at = ctypes.c_void_p(both.data_ptr())
    torch.cuda.synchronize()
    ctx._check(ctx.lib.mg_backward(ctx.handle, model.handle, dense.handle, at, at))
    w_self = ctypes.c_void_p(0)
    ctx._check(ctx.lib.mg_model_grads(model.handle, 1, ctypes.byref(w_self), None, None))
    got = torch.as_tensor(api._DeviceInts(w_self.value, want[0][0].numel()), device="cuda").view(torch.float32)
    for x, y in ((got, want[0][0].flatten()), (both, want_rows.flatten())):
        assert float((x - y).norm()) <= 1e-5 * float(y.norm())                    # (sums over rows meet in any order)


# a table and gradient rows that start anywhere (the step reads and adds 16 bytes at a time where it may)
@pytest.mark.parametrize("table_at,grad_at", [(0, 0), (1, 0), (0, 3), (2, 1)])
@pytest.mark.parametrize("dim", [4, 132])
def test_base_rows_step_at_any_alignment(table_at, grad_at, dim):
    graph = star_graph()
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    table = torch.zeros(N * dim + 4, device="cuda")[table_at:table_at + N * dim].view(N, dim)
    table.copy_(inputs.normal_features(N, dim, seed=4, device="cuda"))
    before = table.clone()
    ctx.load_features(table)
    sizes = [300, 0, 20]
    targets = torch.cat([inputs.distinct_targets(N, s, seed=8 + i) for i, s in enumerate(sizes)])
    dense = ctx.sample_many(targets, np.concatenate([[0], np.cumsum(sizes)]), [6, 4], [1, 2, 3])
    rows = int(dense.counts()[0].sum())
    grad = torch.zeros(rows * dim + 4, device="cuda")[grad_at:grad_at + rows * dim].view(rows, dim)
    grad.copy_(torch.randn((rows, dim), generator=torch.Generator("cuda").manual_seed(5), device="cuda"))
    ids = torch.empty(rows, dtype=torch.int32, device="cuda")
    ctx._check(ctx.lib.mg_dense_packed_ids(ctx.handle, dense.handle, ctypes.c_void_p(ids.data_ptr())))
    ctx.apply_embedding_sgd(dense, grad, 0.25)
    want = before.double().index_add(0, ids.long(), grad.double(), alpha=-0.25)
    assert float((table.double() - want).abs().max()) <= 4 * 2 ** -24 * 8      # (a handful of fp32 sums of magnitude below 8)


# what the forward pass leaves for the backward pass when it is asked to keep its layers (a bit for each output above zero; the aggregates of
# layers of several entries per row), against the same read and gathered again; rows around a row block and a tile, widths around a
# word, a 16-column step, a half tile of output columns
@pytest.mark.parametrize("sizes", [[1], [31, 2], [0, 33, 64], [700, 90], [5_000]])
@pytest.mark.parametrize("dims,aggregator", [([16, 4, 8], "mean"), ([20, 36, 100, 12], "sum"), ([128, 132, 256, 8], "mean"), ([12, 256, 64, 16], "mean")])
def test_what_the_forward_pass_keeps_for_the_backward_pass(sizes, dims, aggregator):
    graph = inputs.erdos_renyi_graph(N, 9 * N, seed=31)
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.load_features(inputs.normal_features(N, dims[0], seed=32, device="cuda"))
    targets = torch.cat([inputs.distinct_targets(N, s, seed=33 + i) for i, s in enumerate(sizes)])
    dense = ctx.sample_many(targets, np.concatenate([[0], np.cumsum(sizes)]), [7, 5, 4][:len(dims) - 1], list(range(len(sizes))))
    model = ctx.model(inputs.random_bias_layers(dims, seed=34))
    model.set_aggregator(aggregator)
    d_out = torch.randn((len(targets), dims[-1]), generator=torch.Generator("cuda").manual_seed(35), device="cuda")
    got = []
    for keep in (False, True):
        ctx.keep_layer_outputs(keep)
        out = torch.empty_like(d_out)
        ctx.forward(model, dense, out)
        grads, rows, ids = ctx.backward(model, dense, d_out, want_h0_grad=True)
        got.append([out, rows.clone(), ids.clone()] + [x.clone() for layer in grads for x in layer])
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][2], got[1][2])
    # the same operands; fp32 sums over up to 6,000 rows meet in any order: sqrt(6,000) 2^-24 of the terms' norm, where terms cancel more
    for x, y in zip(got[0][1:2] + got[0][3:], got[1][1:2] + got[1][3:]):
        assert float((x.double() - y.double()).norm()) <= 1e-4 * max(float(x.double().norm()), 1e-12)


# an aggregator that is set between the two passes: the backward pass takes its own, whatever the forward pass has left
def test_aggregator_set_between_the_passes():
    graph = inputs.erdos_renyi_graph(N, 9 * N, seed=31)
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.load_features(inputs.normal_features(N, 16, seed=32, device="cuda"))
    dense = ctx.sample(inputs.distinct_targets(N, 300, seed=33), [7, 5], seed=34)
    model = ctx.model(inputs.random_bias_layers([16, 32, 8], seed=35))
    d_out = torch.randn((300, 8), generator=torch.Generator("cuda").manual_seed(36), device="cuda")
    got = []
    for keep in (False, True):
        ctx.keep_layer_outputs(keep)
        model.set_aggregator("mean")
        ctx.forward(model, dense, torch.empty_like(d_out))
        model.set_aggregator("sum")
        got.append([x.clone() for layer in ctx.backward(model, dense, d_out) for x in layer])
    for x, y in zip(*got):      # (the same operands, sums in any order)
        assert float((x.double() - y.double()).norm()) <= 1e-4 * float(x.double().norm())


# what the forward pass leaves to save the backward pass work gives way where memory is short: to what the backward pass cannot do without, and it
# is not left at all where there is no room for it (no error of a call that succeeds); the results are the same
@pytest.mark.parametrize("short", ["backward", "forward"])
def test_what_is_kept_to_save_work_gives_way(short):
    graph = inputs.erdos_renyi_graph(N, 9 * N, seed=31)
    dims, per, count = [16, 256, 8], 3_000, 48
    targets = torch.cat([inputs.distinct_targets(N, per, seed=b) for b in range(count)]).cuda()
    d_out = torch.randn((per * count, 8), generator=torch.Generator("cuda").manual_seed(35), device="cuda")
    free = lambda: torch.cuda.mem_get_info()[0]

    def step(keep, held, leave_forward=None, leave_backward=None):
        def hold(leave):
            if leave is not None:
                held.append(torch.empty(free() - leave, dtype=torch.uint8, device="cuda"))
        ctx = mg.Context(0)
        ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
        ctx.load_features(inputs.normal_features(N, dims[0], seed=32, device="cuda"))
        ctx.keep_layer_outputs(keep)
        model = ctx.model(inputs.random_bias_layers(dims, seed=34))
        dense = ctx.sample_many(targets, per * np.arange(count + 1), [7, 4], list(range(count)))
        out = torch.empty_like(d_out)
        hold(leave_forward)
        at = [free()]
        ctx.forward(model, dense, out)
        at.append(free())
        assert ctx.lib.mg_last_error(ctx.handle) in (None, b"")
        if leave_forward is not None:
            held.clear()
            torch.cuda.empty_cache()
        hold(leave_backward)
        at.append(free())
        grads = [x.clone() for layer in ctx.backward(model, dense, d_out) for x in layer]
        at.append(free())
        ctx.close()
        return grads, at[0] - at[1], at[2] - at[3]

    held = []
    step(True, held)                                         # (kernels loaded, torch's own blocks there)
    want, forward, backward = step(False, held)
    _, forward_kept, backward_kept = step(True, held)
    kept = forward_kept - forward
    assert kept > 100 << 20 and backward_kept == backward > kept
    try:
        got, used, _ = step(True, held, forward + kept // 2 if short == "forward" else None, backward - kept // 2 if short == "backward" else None)
        assert used < forward + kept // 2 if short == "forward" else used == forward_kept
    finally:
        held.clear()
        torch.cuda.empty_cache()
    for x, y in zip(want, got):      # (the same operands; sums over rows meet in any order)
        assert float((x.double() - y.double()).norm()) <= 1e-4 * float(x.double().norm())
