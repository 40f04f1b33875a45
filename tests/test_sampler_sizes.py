"""The sampler's work is cut by the size of a hop (nodes per tile, buckets of the last hop, table density): the sizes on
either side of each cut, against the graph's own rows and against the same mini-batches sampled one at a time."""
import numpy as np
import pytest
import torch

import paper_2202_02365_b200 as mg
from paper_2202_02365_b200 import inputs

pytestmark = pytest.mark.gpu

N = 120_000


@pytest.fixture(scope="module")
def graph():
    return inputs.erdos_renyi_graph(N, 6 * N, seed=21)


@pytest.fixture(scope="module")
def ctx(graph):
    c = mg.Context(0)
    c.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    c.load_features(torch.zeros((N, 4), device="cuda"))
    return c


def batches(total):
    """`total` targets in ragged mini-batches of at most 100,000 distinct ids, an empty one among them."""
    sizes, left, s = [0], total, 0
    while left:
        n = min(left, 100_000 - 37 * s)
        sizes.append(n)
        left -= n
        s += 1
    ids = [inputs.distinct_targets(N, n, seed=300 + i) for i, n in enumerate(sizes)]
    return torch.cat(ids), np.concatenate([[0], np.cumsum(sizes)])


# one node; tiles of 32 (full, one more), 64, 128, 256, 512 and 1,024 nodes
@pytest.mark.parametrize("total", [1, 33, 32 * 740, 32 * 740 + 1, 64 * 740 + 1, 128 * 740 + 1, 512 * 1776 + 1, 1024 * 1776 + 1])
def test_hops_on_either_side_of_the_tile_sizes(graph, ctx, total):
    targets, offs = batches(total)
    off, nbrs = graph.row_offsets.numpy(), graph.nbrs.numpy()
    deg = np.diff(off)
    tg = targets.numpy()
    # every neighbour: the arrays hold the rows of the graph
    d = ctx.sample_many(targets.cuda(), offs, [int(deg.max())], list(range(len(offs) - 1)))
    for b in range(len(offs) - 1):
        t = tg[offs[b]:offs[b + 1]]
        v = d.view(b)
        rows = np.concatenate([[0], np.cumsum(deg[t])])
        assert np.array_equal(v.nbr_offsets.cpu().numpy(), rows)
        at = np.repeat(off[t] - rows[:-1], deg[t]) + np.arange(rows[-1])
        assert np.array_equal(v.nbrs.cpu().numpy(), nbrs[at])
        ids = v.node_ids.cpu().numpy()
        assert np.array_equal(ids[v.repr_map.cpu().numpy()], nbrs[at])
        assert np.array_equal(ids[:len(ids) - len(t)], np.setdiff1d(nbrs[at], t))
    d.free()
    # some of them, two hops: the same as the mini-batch alone
    d = ctx.sample_many(targets.cuda(), offs, [3, 2], [7 * b for b in range(len(offs) - 1)],
                        caps={"max_nodes_per_batch": N, "max_nodes_total": min(10 * total, N * (len(offs) - 1)) + 64, "max_entries_total": 18 * total + 64})
    b = len(offs) - 2
    one = ctx.sample(targets[offs[b]:offs[b + 1]], [3, 2], 7 * b)
    x, y = d.view(b), one.view(0)
    for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
        assert torch.equal(getattr(x, key), getattr(y, key)), key
    d.free()
    one.free()
