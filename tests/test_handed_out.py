"""What the binding hands out and takes in: tensors with a start and an autograd life of their own, sizes as they were given."""
import os

import numpy as np
import pytest
import torch

import paper_2202_02365_b200 as mg
from paper_2202_02365_b200 import api, build, inputs

N = 5_000


def test_fanouts_from_any_iterable():
    for given in ([5, 4], (5, 4), iter([5, 4]), (f for f in (5, 4)), np.array([5, 4]), torch.tensor([5, 4])):
        assert list(api._fanouts(given)) == [5, 4]


@pytest.mark.parametrize("too_large", [2 ** 31, 2 ** 32 + 5, -2 ** 31 - 1])
def test_fanouts_that_do_not_fit_are_refused(too_large):
    with pytest.raises((RuntimeError, OverflowError)):
        api._fanouts([5, too_large])


@pytest.fixture
def sample():
    graph = inputs.erdos_renyi_graph(N, 8 * N, seed=51)
    ctx = mg.Context(0)
    ctx.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    ctx.load_features(inputs.normal_features(N, 12, seed=52, device="cuda"))
    targets = torch.cat([inputs.distinct_targets(N, n, seed=n) for n in (101, 37, 1)])
    return ctx, ctx.sample_many(targets, np.array([0, 101, 138, 139]), [3, 5], [1, 2, 3])


@pytest.mark.gpu
@pytest.mark.parametrize("export", [False, True])
def test_arrays_start_on_their_own_and_live_on_their_own(sample, export):
    ctx, dense = sample
    if export:
        dense.export_many()
    for b in range(3):
        v = dense.export_view(b) if export else dense.view(b)
        for x in (v.node_ids, v.node_id_offsets, v.nbrs, v.nbr_offsets, v.repr_map):
            assert x.data_ptr() % 512 == 0 and x.is_contiguous() and x._base is None      # as an allocation of its own starts
        weight = torch.ones((N, 2), device="cuda", requires_grad=True)
        rows = torch.nn.functional.embedding(v.node_ids, weight)                          # keeps the ids for its backward pass
        v.nbrs.add_(1)
        rows.sum().backward()
        assert int(weight.grad.sum()) == 2 * len(v.node_ids)


# the same views where the native part was not built, and that it is missing is said
@pytest.mark.gpu
def test_export_views_without_the_native_part(sample, monkeypatch):
    ctx, dense = sample
    dense.export_many()
    keys = ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map")
    native = [dense.export_view(b) for b in range(3)]
    monkeypatch.setattr(api, "_views", None)
    monkeypatch.setattr(build, "views_path", lambda: os.path.join(build.HERE, "not_built.so"))
    with pytest.warns(RuntimeWarning, match="missing"):
        plain = [dense.export_view(b) for b in range(3)]
    for x, y in zip(native, plain):
        for key in keys:
            assert torch.equal(getattr(x, key), getattr(y, key)) and getattr(y, key).data_ptr() % 512 == 0
    with pytest.raises(mg.MgError):
        dense.export_view(3)


@pytest.mark.gpu
def test_gradients_may_be_changed_in_place(sample):
    ctx, dense = sample
    ctx.keep_layer_outputs(True)
    layers = inputs.random_bias_layers([12, 16, 4], seed=53)
    model = ctx.model(layers)
    out = torch.empty((139, 4), device="cuda")
    ctx.forward(model, dense, out)
    weight = torch.ones((12, 16), device="cuda", requires_grad=True)
    grads = ctx.backward(model, dense, torch.ones_like(out))
    assert all(x.data_ptr() % 16 == 0 for layer in grads for x in layer)
    kept = grads[0][0].clone()
    grads[0][0].add_(weight)                # a penalty's share, recorded by autograd
    assert torch.equal(grads[0][0].detach(), kept + 1) and not grads[0][1].requires_grad


@pytest.mark.gpu
def test_profile_counts_the_kernels_of_its_phases(sample):
    ctx, dense = sample
    model = ctx.model(inputs.random_bias_layers([12, 16, 4], seed=53))
    out = torch.empty((139, 4), device="cuda")
    rel = torch.ones((3, 4), device="cuda")
    lp = ctx.lp_prepare(torch.arange(40), torch.zeros(40), torch.arange(40, 80), 2, 20, seed=1)
    rows = torch.ones((lp.targets().numel(), 4), device="cuda")
    ctx.profile(True)
    ctx.profile_read(reset=True)
    before = ctx.kernel_launches()
    ctx.sample_many(torch.arange(139, dtype=torch.int32), [0, 139], [3, 5], [1], out=dense)
    dense.export_many()
    ctx.forward(model, dense, out)
    ctx.distmult_score(lp, rows, rel)
    phases = ctx.profile_read(reset=True)
    ctx.profile(False)
    assert sum(p["launches"] for p in phases.values()) == ctx.kernel_launches() - before
    assert all(p["launches"] for name, p in phases.items() if name != "gemm")      # (no phase that nothing enters; these layers need no separate product)
