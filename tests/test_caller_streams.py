"""Calls whose caller works on a stream of its own, or hands over host memory that a stream still writes: what is copied out for the
caller is the call's result however late the caller's stream runs, and what is read from the caller is what its stream wrote."""
import numpy as np
import pytest
import torch

import paper_2202_02365_b200 as mg
from paper_2202_02365_b200 import inputs

pytestmark = pytest.mark.gpu

N = 30_000
LATE = 200_000_000     # cycles that the caller's stream sleeps: a tenth of a second


@pytest.fixture(scope="module")
def graph():
    return inputs.erdos_renyi_graph(N, 8 * N, seed=41)


def context(graph, dim=32, stream=None):
    ctx = mg.Context(0, stream)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.load_features(inputs.normal_features(N, dim, seed=42, device="cuda"))
    torch.cuda.synchronize()
    return ctx


def arrays(view):
    return [x.cpu() for x in (view.node_ids, view.node_id_offsets, view.nbrs, view.nbr_offsets, view.repr_map)]


# up to 16,384 targets travel in the staging block of the call, more are copied
@pytest.mark.parametrize("count", [137, 20_000])
def test_pinned_targets_that_the_stream_still_writes(graph, count):
    ctx = context(graph)
    ids = inputs.distinct_targets(N, count, seed=1)
    want = arrays(ctx.sample(ids, [4, 3], 5).view(0))
    host = inputs.distinct_targets(N, count, seed=2).pin_memory()
    device = ids.cuda()
    torch.cuda.synchronize()
    torch.cuda._sleep(LATE)
    host.copy_(device, non_blocking=True)
    got = arrays(ctx.sample(host, [4, 3], 5).view(0))
    assert torch.equal(host, ids) and all(torch.equal(x, y) for x, y in zip(got, want))


def test_pinned_edges_that_the_stream_still_writes(graph):
    ctx = context(graph)
    rng = np.random.RandomState(3)
    edges = [torch.from_numpy(rng.randint(0, n, 5_000).astype(np.int32)) for n in (N, 50, N)]
    want = ctx.lp_prepare(*edges, 4, 100, seed=6).view()
    host = [torch.zeros(5_000, dtype=torch.int32).pin_memory() for _ in edges]
    device = [e.cuda() for e in edges]
    torch.cuda.synchronize()
    torch.cuda._sleep(LATE)
    for h, d in zip(host, device):
        h.copy_(d, non_blocking=True)
    got = ctx.lp_prepare(*host, 4, 100, seed=6).view()
    assert all(torch.equal(got[key], want[key]) for key in want)


@pytest.mark.parametrize("what", ["targets", "view"])
def test_arrays_of_a_freed_link_prediction_batch_copied_on_a_late_stream(graph, what):
    ctx = context(graph)
    rng = np.random.RandomState(3)
    batches = [[torch.from_numpy(rng.randint(0, n, 5_000).astype(np.int32)) for n in (N, 50, N)] for _ in range(3)]
    lps = [ctx.lp_prepare(*b, 4, 100, seed=6) for b in batches]
    take = (lambda lp: {"targets": lp.targets()}) if what == "targets" else (lambda lp: lp.view())
    want = [{k: x.cpu() for k, x in take(lp).items()} for lp in lps]
    for lp in lps:
        lp.free()
    got = []
    with torch.cuda.stream(torch.cuda.Stream()):
        torch.cuda._sleep(LATE)
        for b in batches:
            lp = ctx.lp_prepare(*b, 4, 100, seed=6)
            got.append(take(lp))
            lp.free()
    torch.cuda.synchronize()
    for g, w in zip(got, want):
        assert all(torch.equal(g[k].cpu(), w[k]) for k in w)


def training(graph, stream=None):
    ctx = context(graph, stream=stream)
    ctx.keep_layer_outputs(True)
    model = ctx.model(inputs.random_bias_layers([32, 16, 8], seed=7))
    dense = ctx.sample(inputs.distinct_targets(N, 300, seed=8), [5, 4], 9)
    out = torch.empty((300, 8), device="cuda")
    ctx.forward(model, dense, out)
    d_out = [torch.randn(out.shape, generator=torch.Generator("cuda").manual_seed(i), device="cuda") for i in (1, 2)]
    torch.cuda.synchronize()
    return ctx, model, dense, d_out


def test_gradients_of_two_passes_copied_on_a_late_stream(graph):
    ctx, model, dense, d_out = training(graph, torch.cuda.Stream())
    want = []
    for d in d_out:
        want.append(ctx.backward(model, dense, d))
        torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        torch.cuda._sleep(LATE)
        got = [ctx.backward(model, dense, d) for d in d_out]
    torch.cuda.synchronize()
    for g, w in zip(got, want):
        for x, y in zip((t for layer in g for t in layer), (t for layer in w for t in layer)):
            assert float((x - y).norm()) <= 1e-4 * float(y.norm())      # (sums over rows meet in any order)


def test_gradient_rows_in_memory_that_the_callers_stream_still_reads(graph):
    ctx, model, dense, d_out = training(graph, torch.cuda.Stream())
    rows = int(dense.counts()[0].sum())
    ctx.backward(model, dense, d_out[0], want_h0_grad=True)
    torch.cuda.synchronize()
    user = torch.cuda.Stream()
    with torch.cuda.stream(user):
        before = torch.full((rows, 32), 5.0, device="cuda")
        user.synchronize()
        at = before.data_ptr()
        (before * 1.0).sum()                         # (a kernel's first launch loads it, and waits)
        user.synchronize()
        torch.cuda._sleep(LATE)
        read = before * 1.0
        del before                                   # (the stream's own next allocation may take its place: it comes behind the read)
        _, g_rows, _ = ctx.backward(model, dense, d_out[0], want_h0_grad=True)
    torch.cuda.synchronize()
    assert g_rows.data_ptr() == at
    assert torch.equal(read, torch.full_like(read, 5.0))


@pytest.mark.parametrize("export", [False, True])
def test_views_copied_on_a_late_stream(graph, export):
    ctx = context(graph)
    offs = np.array([0, 200, 500, 650])
    samples = [ctx.sample_many(torch.cat([inputs.distinct_targets(N, n, seed=s + i) for i, n in enumerate(np.diff(offs))]), offs, [4, 3], [1, 2, 3])
               for s in (11, 21)]
    want = [[arrays(d.view(b)) for b in range(3)] for d in samples]
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        torch.cuda._sleep(LATE)
        if export:
            got = []
            for d in samples:
                d.export_many()
                got.append([d.export_view(b) for b in range(3)])
                d.export_many()      # (the same arrays, into the buffer that is still to be read)
        else:
            got = [[d.view(b) for b in range(3)] for d in samples]
    torch.cuda.synchronize()
    for g, w in zip(got, want):
        for x, y in zip(g, w):
            assert all(torch.equal(p, q) for p, q in zip(arrays(x), y))
