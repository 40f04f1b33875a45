"""The sampler's work is cut by the size of a hop (nodes per tile, buckets of the last hop, table density): the sizes on
either side of each cut, against the graph's own rows and against the same mini-batches sampled one at a time."""
import json

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


# many nodes: a thread draws and looks up a node's picks (fanouts of up to six, eleven to twenty); few: a group of lanes does.  Fanouts on either
# side, tiles of 128 and of 256 nodes, one list and both (degrees about 6 and, of the second list, about 20; rows shorter and longer than the fanout)
@pytest.mark.parametrize("total", [90_001, 128 * 740 + 257])
@pytest.mark.parametrize("direction", ["in", "inout"])
def test_picks_by_threads_and_by_groups_of_lanes(graph, total, direction):
    c = mg.Context(0)
    c.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    c.load_features(torch.zeros((N, 4), device="cuda"))
    if direction == "inout":
        other = inputs.rmat_graph(N, 20 * N, seed=22)
        c.load_out_graph(other.row_offsets.cuda(), other.nbrs.cuda())
        c.set_sample_direction("inout")
    per = 9_973
    sizes = [per] * (total // per) + [total % per]
    ids = [inputs.distinct_targets(N, n, seed=300 + i) for i, n in enumerate(sizes)]
    offs = np.concatenate([[0], np.cumsum(sizes)])
    for f in (1, 2, 4, 5, 6, 7, 11, 16, 17, 20, 21):
        d = c.sample_many(torch.cat(ids).cuda(), offs, [f], [2 ** 40 + 7 * b for b in range(len(sizes))])
        for b in (0, 1, len(sizes) - 1):
            one = c.sample(ids[b].cuda(), [f], 2 ** 40 + 7 * b)
            x, y = d.view(b), one.view(0)
            for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
                assert torch.equal(getattr(x, key), getattr(y, key)), (f, key)
            one.free()
        d.free()


# a thread per node in the last tiles of 256 and 512 nodes that are all in work at once, and one node more (148 SMs, four blocks each, five for fanouts of
# one and two), one list and both
@pytest.mark.parametrize("fanout,total", [(3, 151_552), (3, 151_553), (20, 303_104), (20, 303_105), (1, 189_441), (2, 378_881)])
@pytest.mark.parametrize("direction", ["in", "inout"])
def test_tiles_of_a_thread_per_node(graph, fanout, total, direction):
    c = mg.Context(0)
    c.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    if direction == "inout":
        other = inputs.transpose_csr(graph)
        c.load_out_graph(other.row_offsets.cuda(), other.nbrs.cuda())
        c.set_sample_direction("inout")
    sizes = [60_001] * (total // 60_001) + [total % 60_001]
    ids = [inputs.distinct_targets(N, n, seed=500 + i) for i, n in enumerate(sizes)]
    d = c.sample_many(torch.cat(ids).cuda(), np.concatenate([[0], np.cumsum(sizes)]), [fanout], [2 ** 40 + 7 * b for b in range(len(sizes))])
    for b in (0, len(sizes) - 2, len(sizes) - 1):
        one = c.sample(ids[b].cuda(), [fanout], 2 ** 40 + 7 * b)
        x, y = d.view(b), one.view(0)
        for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
            assert torch.equal(getattr(x, key), getattr(y, key)), (b, key)
        one.free()
    c.close()


def hops_launched(call, tmp_path):
    """(blocks, blocks that the SMs hold at once, shared memory of those on one SM) of every k_hop that `call` launches."""
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    prof.export_chrome_trace(str(tmp_path / "trace.json"))
    events = [e for e in json.load(open(tmp_path / "trace.json"))["traceEvents"] if e.get("cat") == "kernel" and "k_hop" in e["name"]]
    launched = []
    for e in sorted(events, key=lambda e: e["ts"]):
        registers, smem = -(-e["args"]["registers per thread"] // 8) * 8, e["args"]["shared memory"] + 1024      # (a kilobyte of every block is the system's)
        held = min(65536 // (256 * registers), 228 * 1024 // smem)
        launched.append((e["args"]["grid"][0], held * torch.cuda.get_device_properties(0).multi_processor_count, held * smem))
    return launched


# the blocks of a hop that may be picked by a thread per node are all on the SMs at once, whatever the hop turns out to have: without caps far
# less than its bound.  Tiles of every size in that form, fanouts on either side of its instances, one list and both
@pytest.mark.parametrize("direction", ["in", "inout"])
@pytest.mark.parametrize("targets", [4_200, 9_000, 30_000])
def test_later_hops_that_have_less_than_their_bound(graph, direction, targets, tmp_path):
    c = mg.Context(0)
    c.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    c.load_features(torch.zeros((N, 4), device="cuda"))
    other = inputs.rmat_graph(N, 20 * N, seed=22)
    if direction == "inout":
        c.load_out_graph(other.row_offsets.cuda(), other.nbrs.cuda())
        c.set_sample_direction("inout")
    ids = [inputs.distinct_targets(N, n, seed=n) for n in (targets - 1, 1)]
    pair = torch.cat(ids).cuda()
    for f in (1, 2, 3, 5, 6, 11, 16, 20):
        d = c.sample_many(pair, [0, targets - 1, targets], [40, f], [3, 4])
        one = c.sample(ids[1].cuda(), [40, f], 4)      # (the few nodes of the second mini-batch alone: a group of lanes per node)
        x, y = d.view(1), one.view(0)
        for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
            assert torch.equal(getattr(x, key), getattr(y, key)), (f, key)
        launched = hops_launched(lambda: c.sample_many(pair, [0, targets - 1, targets], [40, f], [3, 4], out=d), tmp_path)
        assert len(launched) == 2 and launched[1][0] <= launched[1][1], (f, launched)
        assert launched[1][2] <= 196 * 1024, (f, launched)      # (above, the look-ups have next to no L1)
        one.free()
        d.free()
    c.close()


# both lists in hops of more than a million nodes: tiles of 1,024, 512 and 256 nodes by what the picks leave of the shared memory, and fewer blocks
@pytest.mark.parametrize("fanout", [2, 4, 6, 12, 16, 20])
def test_picks_by_threads_in_tiles_that_leave_room_for_them(graph, fanout, tmp_path):
    c = mg.Context(0)
    c.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    other = inputs.transpose_csr(graph)
    c.load_out_graph(other.row_offsets.cuda(), other.nbrs.cuda())
    c.set_sample_direction("inout")
    n_batches, per = 700, 700
    rows = [inputs.distinct_targets(N, per - b % 2, seed=b) for b in range(n_batches)]
    offs = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    caps = {"max_nodes_per_batch": 60_000, "max_nodes_total": 16_000_000 + 4_000_000 * fanout, "max_entries_total": 16_000_000 + 6_000_000 * fanout}
    d = c.sample_many(torch.cat(rows), offs, [3, fanout], list(range(n_batches)), caps=caps)
    assert int(d.counts()[0][:, 1].sum()) > 1_818_624      # (tiles of 1,024 where they fit)
    launched = hops_launched(lambda: c.sample_many(torch.cat(rows), offs, [3, fanout], list(range(n_batches)), caps=caps, out=d), tmp_path)
    assert launched[1][0] <= launched[1][1] and launched[1][2] <= 196 * 1024, launched
    for b in (0, 1, n_batches // 2, n_batches - 1):
        one = c.sample(rows[b], [3, fanout], b)
        x, y = d.view(b), one.view(0)
        for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
            assert torch.equal(getattr(x, key), getattr(y, key)), (b, key)
        one.free()
    c.close()


# the last hop: through the global tables (little room in all); buckets in shared memory, one (a table of a few hundred nodes), several
# with tables for blocks of 256, 512 and 1,024 threads, as many tables as a mini-batch may need, and more (global tables again); ids that are multiples of a Fibonacci
# number, whose multiplicative hashes lie next to each other
@pytest.mark.parametrize("room,n_batches", [(300, 1), (N, 1), (300, 3_600), (4_000, 300), (12_000, 120), (N, 9), (370_000, 4), (420_000, 4)])
def test_last_hop_buckets(graph, ctx, room, n_batches):
    off, nbrs = graph.row_offsets.numpy(), graph.nbrs.numpy()
    per = max(1, min(room // 45, 2_000))
    ids = torch.arange(0, N, 987, dtype=torch.int32)
    rows = [torch.cat([ids[:min(per, len(ids)) // 2], torch.tensor([1], dtype=torch.int32)])]
    rows += [inputs.distinct_targets(N, per, seed=b) for b in range(1, n_batches)]
    offs = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    caps = {"max_nodes_per_batch": room, "max_nodes_total": 45 * per * n_batches + 256, "max_entries_total": 48 * per * n_batches + 256}
    d = ctx.sample_many(torch.cat(rows), offs, [4, 5], list(range(n_batches)), caps=caps)
    nodes, entries = d.counts()
    for b in (0, n_batches - 1):
        v = d.view(b)
        ids_b, rep, o = v.node_ids.cpu().numpy(), v.repr_map.cpu().numpy(), v.nbr_offsets.cpu().numpy()
        got = v.nbrs.cpu().numpy()
        assert len(np.unique(ids_b)) == len(ids_b) == int(nodes[b].sum())
        assert np.array_equal(ids_b[rep], got)
        src = ids_b[len(ids_b) - (len(o) - 1):]          # the sampled nodes, in order
        cnt = np.diff(o)
        deg = off[src + 1] - off[src]
        n0 = len(ids_b) - len(src)
        hop = np.where(np.arange(len(src)) >= len(src) - int(nodes[b, 0]), 4, 5)
        assert n0 == int(nodes[b, 2]) and np.array_equal(cnt, np.minimum(deg, hop))
        first = np.unique(got)                           # every node is a target or somebody's neighbour
        assert np.array_equal(np.unique(np.concatenate([first, rows[b].numpy()])), np.sort(ids_b))
    d.free()


# the last hop's tables in shared memory have slots for what their buckets hold, up to the room there is: mini-batches of none, one, few and many
# targets in one call, with just the room that the largest takes (16,009 nodes) each and with far more
@pytest.mark.parametrize("room", [16_009, 60_000, 300_000])
def test_last_hop_of_mini_batches_of_any_size(graph, ctx, room):
    sizes = [2_000, 0, 1, 3, 60, 700, 0, 1_500] * 10
    rows = [inputs.distinct_targets(N, n, seed=b) for b, n in enumerate(sizes)]
    rows[3] = torch.tensor([0, 1, N - 1], dtype=torch.int32)
    offs = np.concatenate([[0], np.cumsum(sizes)])
    caps = {"max_nodes_per_batch": room, "max_nodes_total": 1_500_000, "max_entries_total": 2_000_000}
    d = ctx.sample_many(torch.cat(rows), offs, [2, 3], list(range(len(sizes))), caps=caps)
    for b in (*range(8), len(sizes) - 1):
        one = ctx.sample(rows[b], [2, 3], b)
        x, y = d.view(b), one.view(0)
        for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
            assert torch.equal(getattr(x, key), getattr(y, key)), (b, key)
        one.free()
    d.free()


# entries go into the id tables 128 at a time, an entry per thread, or (hops with room for more than the SMs hold at once that way) 512 at
# a time: either form with blocks that touch a few mini-batches, and more mini-batches than a block keeps counts for
@pytest.mark.parametrize("per,fanout", [(1, 14), (4, 13), (4, 14)])
def test_id_table_blocks_over_many_mini_batches(graph, ctx, per, fanout):
    n_batches = 4_000
    rows = [inputs.distinct_targets(N, per, seed=b) for b in range(n_batches)]
    rows[17] = rows[17][:0]
    offs = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    d = ctx.sample_many(torch.cat(rows), offs, [fanout, 3], list(range(n_batches)), caps={"max_nodes_per_batch": 600})
    for b in (0, 16, 17, 18, 1_999, n_batches - 1):
        one = ctx.sample(rows[b], [fanout, 3], b)
        x, y = d.view(b), one.view(0)
        for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
            assert torch.equal(getattr(x, key), getattr(y, key)), (b, key)
        one.free()
    d.free()


# as many mini-batches as a call may have: where each stands in the export
def test_export_of_as_many_mini_batches_as_a_call_may_have(graph, ctx):
    n_batches = 4_096
    rows = [inputs.distinct_targets(N, 1 + b % 3, seed=b) for b in range(n_batches)]
    rows[17] = rows[17][:0]
    offs = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    d = ctx.sample_many(torch.cat(rows), offs, [3, 2, 2], list(range(n_batches)), caps={"max_nodes_per_batch": 200})
    d.export_many()
    views = [d.export_view(b) for b in range(n_batches)]
    for b in (0, 1, 16, 17, 18, 2_047, n_batches - 2, n_batches - 1):
        x, y = views[b], d.view(b)
        for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
            assert torch.equal(getattr(x, key), getattr(y, key)), (b, key)
    d.free()


# ids of 29 bits and mini-batches of 12: no part of a sample packs both into one word
def test_many_mini_batches_on_a_graph_of_many_nodes():
    n, n_batches = 2 ** 28 + 1, 2_049
    rows = torch.arange(n_batches, device="cuda") * ((n - 1) // (n_batches - 1))             # a target each, the first and the last node among them
    assert int(rows[-1]) == n - 1
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[rows + 1] = 3
    off = torch.cumsum(off, 0)
    nbrs = torch.stack([(rows + 1) % n, (rows + 12_345) % n, (rows + n // 2) % n], 1).sort(1).values
    c = mg.Context(0)
    c.load_graph(off, nbrs.flatten().to(torch.int32))
    del off
    d = c.sample_many(rows.to(torch.int32), list(range(n_batches + 1)), [3], list(range(n_batches)), caps={"max_nodes_per_batch": 16})
    d.export_many()
    for b in (0, 1, 1_024, n_batches - 1):
        for v in (d.export_view(b), d.view(b)):
            assert torch.equal(v.nbrs.long(), nbrs[b]) and int(v.node_ids[-1]) == int(rows[b])
            assert torch.equal(v.node_ids[v.repr_map.long()].long(), nbrs[b])
    c.close()
    torch.cuda.empty_cache()


# an export orders the ids of a delta bin by bin: deltas on either side of the number of bins (65), of what a warp compares (129), of what
# a block compares where the bin's range takes several bitmaps (1,025), ranges of one bitmap and of more, consecutive ids (one bin has all)
# and spread ones, before and behind the last hop (sampled nodes carry their entries along)
@pytest.mark.parametrize("stride", [1, 61, 200])
def test_export_orders_deltas_of_any_size_and_spread(stride):
    n, base = 2 ** 25 + 3, 5 * 2 ** 20 + 77
    sizes = [1, 64, 65, 128, 129, 1_000, 1_024, 1_025, 4_096, 4_097, 40_000, 0]
    tg = [np.arange(-(-m // 1_000), dtype=np.int64) + 100 * s for s, m in enumerate(sizes)]      # 1,000 of the delta's ids from each target
    counts = np.zeros(n, np.int32)
    inner = base + stride * np.arange(max(sizes))
    counts[inner] = np.arange(len(inner)) % 4
    for t, m in zip(tg, sizes):
        counts[t] = np.minimum(1_000, m - 1_000 * np.arange(len(t)))
    off = np.concatenate([[0], np.cumsum(counts, dtype=np.int64)])
    nbrs = np.empty(off[-1], np.int32)
    for t, m in zip(tg, sizes):
        if m: nbrs[off[t[0]]:off[t[0]] + m] = np.sort(inner[:m])
    for q in range(3):      # the last deltas: consecutive ids (stride 1) or spread ones
        has = np.nonzero(np.arange(len(inner)) % 4 > q)[0]
        nbrs[off[inner[has]] + q] = 2 ** 24 + stride * (2 * has + q)
    c = mg.Context(0)
    c.load_graph(torch.from_numpy(off).cuda(), torch.from_numpy(nbrs).cuda())
    rng = np.random.default_rng(3)
    targets = torch.from_numpy(np.concatenate([rng.permutation(t) for t in tg]).astype(np.int32))
    offs = np.concatenate([[0], np.cumsum([len(t) for t in tg])])
    room = 40 + 1_000 + 4 * 40_000
    d = c.sample_many(targets, offs, [1_000, 3], list(range(len(tg))), caps={"max_nodes_total": 3 * room, "max_entries_total": 3 * room, "max_nodes_per_batch": room})
    nodes, _ = d.counts()
    assert nodes[:, 1].tolist() == sizes
    d.export_many()
    views = [d.export_view(b) for b in range(len(tg))]
    for b, x in enumerate(views):
        y = d.view(b)
        for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
            assert torch.equal(getattr(x, key), getattr(y, key)), (b, key)
        at = x.node_id_offsets.tolist()
        for lo, hi in zip(at[:-2], at[1:-1]):
            assert bool((x.node_ids[lo:hi].diff() > 0).all())
        assert torch.equal(x.node_ids[x.repr_map.long()], x.nbrs)
    c.close()
    torch.cuda.empty_cache()


# the tables of k_hop over the mini-batches beside its largest tile: more shared memory than a kernel has without asking
@pytest.mark.parametrize("fanout", [9, 40])
def test_largest_tiles_with_as_many_mini_batches_as_a_call_may_have(graph, ctx, fanout):
    n_batches, per = 4_096, 40
    rows = [inputs.distinct_targets(N, per - b % 7, seed=b) for b in range(n_batches)]
    offs = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    d = ctx.sample_many(torch.cat(rows), offs, [fanout, fanout], list(range(n_batches)), caps={"max_nodes_per_batch": 4_000, "max_nodes_total": 4_000_000 * 3,
                                                                                              "max_entries_total": 4_000_000 * 3})
    for b in (0, 1, 2_047, n_batches - 1):
        one = ctx.sample(rows[b], [fanout, fanout], b)
        x, y = d.view(b), one.view(0)
        for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
            assert torch.equal(getattr(x, key), getattr(y, key)), (b, key)
        one.free()
    d.free()


# ids are as wide as the graph that was sampled has them, whatever the context has loaded since
@pytest.mark.parametrize("n_later", [500, 4 * N])
def test_arrays_of_a_sample_whose_graph_has_been_replaced(graph, n_later):
    c = mg.Context(0)
    c.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    rows = [inputs.distinct_targets(N, n, seed=n) for n in (700, 1, 90)]
    offs = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    keys = ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map")
    d = c.sample_many(torch.cat(rows), offs, [4, 3], [1, 2, 3])
    d.export_many()
    want = [{key: getattr(d.export_view(b), key).clone() for key in keys} for b in range(len(rows))]
    later = inputs.erdos_renyi_graph(n_later, 4 * n_later, seed=5)
    c.load_graph(later.row_offsets.cuda(), later.nbrs.cuda())
    d.export_many()
    for b, arrays in enumerate(want):
        for v in (d.export_view(b), d.view(b)):
            for key in keys:
                assert torch.equal(getattr(v, key), arrays[key]), (b, key)
    c.close()


# ... and deltas with as many bins as there are (131,073 nodes and more), spread and in one run of a graph of many nodes, and runs of ids that lie
# further apart than a bitmap reaches, several in a bin; targets with a thousand entries each and too few of them for a warp's share
@pytest.mark.parametrize("place,sizes,n", [(lambda i: 2 ** 18 * (i % 5) + i // 5, (64, 129, 1_000, 1_025, 4_097, 40_000), 2 ** 25),
                                           (lambda i: 61 * i, (131_072, 131_073, 150_000), 2 ** 26), (lambda i: i, (150_000,), 2 ** 27 - 1)],
                         ids=["runs", "long", "one-run"])
def test_export_orders_long_deltas_and_ids_in_runs(place, sizes, n):
    base, most = 5 * 2 ** 20 + 77, max(sizes)
    tg = [np.arange(-(-m // 1_000), dtype=np.int64) + 1_000 * s for s, m in enumerate(sizes)]      # 1,000 of the delta's ids from each target
    inner = base + place(np.arange(most, dtype=np.int64))
    has = np.nonzero(np.arange(most) % 4)[0]
    rows, ids = [], []
    for t, m in zip(tg, sizes):
        rows.append(np.repeat(t, np.minimum(1_000, m - 1_000 * np.arange(len(t)))))
        ids.append(inner[:m])
    for q in range(3):      # the last deltas: placed alike, up to three of their ids from each node
        at = has[has % 4 > q]
        rows.append(inner[at])
        ids.append(2 ** 24 + place(2 * at + q))
    rows, ids = np.concatenate(rows), np.concatenate(ids)
    assert inner.max() < 2 ** 24 and ids.max() < n
    off = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n), dtype=np.int64)])
    c = mg.Context(0)
    c.load_graph(torch.from_numpy(off).cuda(), torch.from_numpy(ids[np.lexsort((ids, rows))].astype(np.int32)).cuda())
    offs = np.concatenate([[0], np.cumsum([len(t) for t in tg])])
    room = 1_000 + 4 * most
    d = c.sample_many(torch.from_numpy(np.concatenate(tg).astype(np.int32)), offs, [1_000, 3], list(range(len(tg))),
                      caps={"max_nodes_total": 3 * room, "max_entries_total": 3 * room, "max_nodes_per_batch": room})
    assert d.counts()[0][:, 1].tolist() == list(sizes)
    d.export_many()
    for b in range(len(tg)):
        x, y = d.export_view(b), d.view(b)
        for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
            assert torch.equal(getattr(x, key), getattr(y, key)), (b, key)
        at = x.node_id_offsets.tolist()
        for lo, hi in zip(at[:-2], at[1:-1]):
            assert bool((x.node_ids[lo:hi].diff() > 0).all())
        assert torch.equal(x.node_ids[x.repr_map.long()], x.nbrs)
    c.close()
    torch.cuda.empty_cache()


# an export runs on the sampling stream, beside the layers of another sample and before the next one is drawn
def test_exports_beside_the_layers_of_other_samples(graph):
    c = mg.Context(0)
    c.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    c.load_features(inputs.normal_features(N, 32, seed=8, device="cuda"))
    model = c.model(inputs.random_bias_layers([32, 64, 64], seed=9))
    keys = ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map")
    n_batches, per = 24, 600
    offs = per * np.arange(n_batches + 1)
    rows = [torch.cat([inputs.distinct_targets(N, per, seed=100 * g + b) for b in range(n_batches)]).cuda() for g in range(5)]
    seeds = [[1_000 * g + b for b in range(n_batches)] for g in range(5)]
    outs, arrays = [], []
    for g in range(5):      # one behind the other
        d = c.sample_many(rows[g], offs, [8, 4], seeds[g])
        outs.append(c.forward(model, d, torch.empty((n_batches * per, 64), device="cuda")))
        arrays.append([{key: getattr(v, key).clone() for key in keys} for v in (d.view(b) for b in (0, 11, n_batches - 1))])
        d.free()
    held = [c.sample_many(rows[0], offs, [8, 4], seeds[0]) for _ in range(3)]
    for g in range(2):
        c.sample_many_begin(rows[g], offs, [8, 4], seeds[g], out=held[g])
    for g in range(5):
        d = held[g % 3]
        c.sample_many_end(d)
        d.export_many()
        if g + 2 < 5:
            c.sample_many_begin(rows[g + 2], offs, [8, 4], seeds[g + 2], out=held[(g + 2) % 3])
        assert torch.equal(c.forward(model, d, torch.empty((n_batches * per, 64), device="cuda")), outs[g])
        for want, b in zip(arrays[g], (0, 11, n_batches - 1)):
            v = d.export_view(b)
            for key in keys:
                assert torch.equal(getattr(v, key), want[key]), (g, b, key)
    c.close()


# the same tables beside a tile that has both directions: as many mini-batches as need no more shared memory than a kernel has without asking,
# one more, as many as a call may have
@pytest.mark.parametrize("n_batches", [1_408, 1_409, 4_096])
def test_largest_tiles_of_both_directions(graph, n_batches):
    c = mg.Context(0)
    c.load_graph(graph.row_offsets.cuda(), graph.nbrs.cuda())
    other = inputs.transpose_csr(graph)
    c.load_out_graph(other.row_offsets.cuda(), other.nbrs.cuda())
    c.set_sample_direction("inout")
    rows = [inputs.distinct_targets(N, 60 - b % 2, seed=b) for b in range(n_batches)]      # (hop 1: room for more nodes than 12 x 148 tiles of 1,024)
    offs = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    d = c.sample_many(torch.cat(rows), offs, [9, 1], list(range(n_batches)),
                      caps={"max_nodes_per_batch": 2_400, "max_nodes_total": 2_400 * n_batches, "max_entries_total": 2_400 * n_batches})
    for b in (0, 1, n_batches // 2, n_batches - 1):
        one = c.sample(rows[b], [9, 1], b)
        x, y = d.view(b), one.view(0)
        for key in ("node_ids", "node_id_offsets", "nbrs", "nbr_offsets", "repr_map"):
            assert torch.equal(getattr(x, key), getattr(y, key)), (b, key)
        one.free()
    c.close()
