"""What a program that uses this package has it do, as cases that can be timed: the sizes, the inputs, one pass of each.

A case names a task and its sizes; the tasks are
  infer   sample mini-batches (DENSE) and run the GraphSage layers over them
  export  sample mini-batches and take every mini-batch's arrays in the paper's canonical order
  train   one training step with fixed features: sample, layers, backward pass, Adagrad step of the weights
  embed   one training step with learned base representations: the same with an SGD step of the weights and of the rows
  lp      one link-prediction step: negatives and target union, a one-hop sample, one layer, DistMult scores
The graphs are the seeded stand-ins of `inputs.py` at sizes that can be made in about a second.
"""
import math

import numpy as np
import torch

import paper_2202_02365_b200 as mg
from paper_2202_02365_b200 import inputs

N_RELATIONS = 14_824      # relation types of the link-prediction workload


# ---- the cases ------------------------------------------------------------------------------------------------------
def _case(name, task, **sizes):
    """Every case carries every key of its task, so that a drawn one is made the same way."""
    c = {"task": task, "graph": "rmat", "nodes": 1_000_000, "edges": 20_000_000, "dim": 128, "half": False, "parts": 1, "resident": 1,
         "in_host_memory": False, "inout": False, "hops": 3, "fan0": 15, "fan1": 10, "fan2": 5, "batches": 1, "targets": 1000,
         "hidden": 256, "half_between": False, "host_io": False, "encoder": "sage", "heads": 1, "edges_scored": 0, "chunks": 1, "negatives": 0}
    c.update(sizes)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a first try of the package, or a small citation graph: one mini-batch, two narrow layers; all of it is launches and waits
        _case("tiny_graph", "infer", graph="er", nodes=10_000, edges=200_000, dim=16, hidden=16, hops=2, fan0=10, fan1=5, targets=512),
        # one mini-batch of node classification on a graph of a million nodes: what a loop without look-ahead waits for
        _case("one_mini_batch", "infer"),
        # a service that answers for some users at once: ids come from host memory, the rows go back there; odd widths
        _case("serve_from_host", "infer", nodes=300_007, edges=4_500_001, dim=100, hidden=100, hops=2, fan0=12, fan1=7, batches=3,
              targets=137, host_io=True),
        # the throughput configuration on a paper-citation graph: 128 mini-batches in one call (layer outputs over all nodes of a train set)
        _case("papers_group", "infer", nodes=16_000_000, edges=234_000_000, parts=16, resident=16, batches=128),
        # the same with the intermediate rows kept as fp16, a ragged group of ragged mini-batches
        _case("papers_half_between", "infer", nodes=4_000_037, edges=58_000_000, batches=37, targets=777, half_between=True),
        # neighbours from both edge directions: mini-batches many times larger, rows of up to thirty entries
        _case("papers_both_directions", "infer", nodes=8_000_000, edges=117_000_000, parts=16, resident=16, inout=True, batches=16),
        # wide half-precision rows out of core: the table stays in host memory, a third of the partitions is in the buffer
        _case("wide_rows_in_buffer", "infer", nodes=4_000_000, edges=43_000_000, dim=768, half=True, parts=32, resident=10,
              in_host_memory=True, batches=64),
        # the sampler feeding another framework's layers: every mini-batch's arrays in canonical order
        _case("sample_and_export", "export", nodes=8_000_000, edges=117_000_000, batches=32),
        # a training step of node classification (features are fixed)
        _case("train_step", "train", batches=8),
        # a training step that also learns the base representations
        _case("train_base_rows", "embed", nodes=2_000_000, edges=30_000_000, batches=24, targets=1000),
        # a link-prediction step on a knowledge graph: 50,000 edges against 1,000 shared negatives a chunk, both sides corrupted
        _case("link_prediction", "lp", nodes=8_000_000, edges=32_000_000, dim=100, parts=16, resident=8, hops=1, fan0=20, hidden=100,
              edges_scored=50_000, chunks=10, negatives=1000),
        # a smaller step of the same with graph attention as the encoder
        _case("link_prediction_attention", "lp", nodes=2_000_000, edges=8_000_000, dim=100, hops=1, fan0=20, hidden=100, encoder="gat",
              edges_scored=5_000, chunks=4, negatives=500),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def fanouts(both):
        # the fanouts of the configurations, and what lies about them; both directions double what a node gets
        hops = rng.choice((1, 2, 2, 3, 3))
        return {"hops": hops, "fan0": rng.randint(5, 15 if both else 20), "fan1": rng.randint(4, 10), "fan2": rng.randint(3, 5)}

    task = rng.choice(("infer", "infer", "infer", "export", "train", "embed", "lp"))
    if task == "lp":
        nodes = log_int(50_000, 8_000_000)
        parts = rng.choice((1, 16))
        chunks = rng.randint(1, 10)
        encoder = rng.choice(("sage", "sage", "gat"))
        dim = rng.choice((32, 64, 100, 128))
        return _case("", task, nodes=nodes, edges=4 * nodes, dim=dim, hidden=dim, parts=parts, resident=1 if parts == 1 else 8, hops=1,
                     fan0=rng.randint(10, 20), encoder=encoder, heads=rng.choice((1, 2)) if encoder == "gat" else 1, chunks=chunks,
                     edges_scored=log_int(1_000, 50_000), negatives=rng.choice((100, 250, 500, 1000, 997)))
    nodes = log_int(10_000, 8_000_000)
    small = nodes < 100_000 and rng.random() < 0.5
    c = _case("", task, graph="er" if small else "rmat", nodes=nodes, edges=int(nodes * rng.uniform(10, 20)),
              dim=rng.choice((16, 64, 100, 128, 128, 256)), hidden=rng.choice((16, 64, 100, 128, 256, 256)))
    c["batches"] = log_int(1, {"infer": 64, "export": 32, "train": 16, "embed": 16}[task])
    c["targets"] = min(log_int(64, 1000), nodes // 4)
    if task == "infer":
        option = rng.choice(("none", "none", "both", "between", "buffer", "host", "host"))
        c["host_io"] = option == "host"
        c["inout"] = option == "both"
        if option == "both":
            c["batches"] = min(c["batches"], 8)
        if option == "between":
            c["half_between"] = True
            c["hidden"] = rng.choice((128, 256))
        if option == "buffer":
            c.update(half=True, dim=rng.choice((128, 384, 768)), parts=32, resident=rng.randint(8, 12), in_host_memory=rng.random() < 0.5)
            c["nodes"] = min(max(c["nodes"], 200_000), 4_000_000)
            c["edges"] = int(c["nodes"] * rng.uniform(10, 15))
            c["graph"] = "rmat"
            c["targets"] = min(c["targets"], c["nodes"] // 16)
    c.update(fanouts(c["inout"]))
    return c


# ---- inputs and handles ---------------------------------------------------------------------------------------------
def _fanouts(case):
    return [case["fan0"], case["fan1"], case["fan2"]][:case["hops"]]


def _resident_parts(case, seed):
    g = torch.Generator().manual_seed(seed)
    return sorted(torch.randperm(case["parts"], generator=g)[:case["resident"]].tolist())


def _load_rows(ctx, case, seed, resident):
    """The table of base representations: fp32 or fp16, in device memory, or in pinned host blocks of one partition each."""
    n, dim = case["nodes"], case["dim"]
    dtype = torch.float16 if case["half"] else torch.float32
    std = 0.001 if case["task"] == "lp" else 1.0
    if case["parts"] > 1:
        ctx.set_partitioning(case["parts"])
    if not case["in_host_memory"]:
        table = inputs.normal_features(n, dim, seed, "cuda", dtype=dtype, std=std)
        if case["parts"] > 1:
            ctx.load_features(table, capacity_parts=case["resident"])
            ctx.set_resident(resident)
        else:
            ctx.load_features(table)
        return table
    ctx.load_features(None, capacity_parts=case["resident"], backing=mg.BACKING_HOST, dtype=dtype, dim=dim)
    size = inputs.contiguous_partition(n, case["parts"])
    block = torch.empty((size, dim), dtype=dtype, pin_memory=True)      # one staging block, refilled for every partition
    for i, p in enumerate(resident):
        rows = min(n, (p + 1) * size) - p * size
        block[:rows].copy_(inputs.block_features(rows, dim, seed, p, "cuda", dtype))
        ctx.set_partition_source(p, block)
        ctx.set_resident(resident[:i + 1])
        ctx.set_partition_source(p, None)
    return block


def _targets(case, seed, resident):
    """Distinct ids for every mini-batch, drawn among the nodes in the buffer."""
    n, b, t = case["nodes"], case["batches"], case["targets"]
    g = torch.Generator("cuda").manual_seed(seed)
    if case["parts"] > 1:
        size = inputs.contiguous_partition(n, case["parts"])
        pool = torch.cat([torch.arange(p * size, min(n, (p + 1) * size), device="cuda") for p in resident])
    else:
        pool = torch.arange(n, device="cuda")
    rows = []
    for _ in range(b):      # the first t distinct ones of a draw with a margin
        ids = pool[torch.randint(0, pool.numel(), (2 * t + 64,), generator=g, device="cuda")]
        ids, first = torch.unique(ids, return_inverse=True)
        at = torch.full((ids.numel(),), first.numel(), device="cuda").scatter_reduce_(0, first, torch.arange(first.numel(), device="cuda"), "amin")
        rows.append(ids[torch.argsort(at)[:t]])
    return torch.cat(rows).to(torch.int32)


def prepare(case, seed):
    task, n = case["task"], case["nodes"]
    ctx = mg.Context(0)
    make = inputs.erdos_renyi_graph if case["graph"] == "er" else inputs.rmat_graph
    graph = make(n, case["edges"], seed, "cuda", **({"n_relations": N_RELATIONS} if task == "lp" else {}))
    ctx.load_graph(graph.row_offsets, graph.nbrs)
    if case["inout"]:
        other = inputs.transpose_csr(graph)
        ctx.load_out_graph(other.row_offsets, other.nbrs)
        ctx.set_sample_direction("inout")
    resident = _resident_parts(case, seed + 1)
    s = {"case": case, "ctx": ctx, "table": _load_rows(ctx, case, seed + 2, resident), "dense": None, "seed": seed}
    dims = [case["dim"]] + [case["hidden"]] * case["hops"]
    layers = (inputs.glorot_layers if task == "lp" else inputs.random_bias_layers)(dims, seed + 3)     # (rows of 0.001: a bias would drown them)
    if case["encoder"] == "gat":
        g = torch.Generator().manual_seed(seed + 4)
        s["model"] = ctx.gat_model([(w, torch.randn(w.shape[1], generator=g) * 0.1, torch.randn(w.shape[1], generator=g) * 0.1, b)
                                    for w, _, b in layers])
        if case["heads"] > 1:
            s["model"].set_heads(case["heads"])
    else:
        s["model"] = ctx.model(layers)
        if case["half_between"]:
            s["model"].set_intermediates(torch.float16)
    if task == "lp":
        mask = inputs.resident_node_mask(n, case["parts"], resident, "cuda") if case["parts"] > 1 else None
        s["edges"] = inputs.lp_edges(graph, mask, case["edges_scored"], seed + 5)
        s["relations"] = inputs.normal_features(N_RELATIONS, case["dim"], seed + 6, "cuda")
        return s

    count = case["batches"] * case["targets"]
    targets = _targets(case, seed + 5, resident)
    s["targets"] = targets.cpu().pin_memory() if case["host_io"] else targets
    s["offsets"] = torch.arange(case["batches"] + 1) * case["targets"]
    s["seeds"] = [seed * 1000 + b for b in range(case["batches"])]
    # room for a sample, from a first one: the worst case would take many times the memory
    probe = ctx.sample_many(targets, s["offsets"], _fanouts(case), s["seeds"], caps=_first_caps(case))
    nodes, entries = probe.counts()
    probe.free()
    s["caps"] = {"max_nodes_total": int(nodes.sum() * 1.3) + 1024, "max_entries_total": int(entries.sum() * 1.3) + 1024,
                 "max_nodes_per_batch": int(nodes.sum(1).max() * 1.5) + 64,
                 "max_inner_nodes_per_batch": int(nodes[:, :-1].sum(1).max() * 1.5) + 64}
    if task == "export":
        hop_nodes, hop_entries, _ = _sizes(case)      # room for what the degrees give, and a fifth more
        room = {"node_ids": sum(hop_nodes), "nbrs": sum(hop_entries), "nbr_offsets": sum(hop_nodes[:-1]) + 1, "repr_map": sum(hop_entries),
                "node_id_offsets": case["hops"] + 2}
        s["arrays"] = {key: torch.zeros(int(1.2 * case["batches"] * r) + 4096, dtype=torch.int32, device="cuda") for key, r in room.items()}
    else:
        s["out"] = torch.empty((count, case["hidden"]), pin_memory=True) if case["host_io"] else torch.empty((count, case["hidden"]), device="cuda")
    if task in ("train", "embed"):
        ctx.keep_layer_outputs(True)
        g = torch.Generator("cuda").manual_seed(seed + 6)
        s["d_out"] = torch.randn((count, case["hidden"]), generator=g, device="cuda") / count      # the loss's gradient, a mean over the targets
    return s


def _first_caps(case):
    """Bounds for the first sample of a group: twice what the degrees of the graph give."""
    nodes, entries = _sizes(case)[:2]
    room = int(2 * max(sum(nodes), sum(entries))) + 8192
    return {"max_nodes_total": case["batches"] * room, "max_entries_total": case["batches"] * room, "max_nodes_per_batch": room}


# ---- one pass -------------------------------------------------------------------------------------------------------
def run(s):
    case, ctx = s["case"], s["ctx"]
    if case["task"] == "lp":
        return _run_lp(s)
    s["dense"] = dense = ctx.sample_many(s["targets"], s["offsets"], _fanouts(case), s["seeds"], caps=s["caps"], out=s["dense"])
    if case["task"] == "export":
        dense.export_many()
        views = [dense.export_view(b) for b in range(case["batches"])]
        for key, array in s["arrays"].items():      # the other framework's own arrays, one mini-batch behind the other
            parts = [getattr(v, key) for v in views]
            torch.cat(parts, out=array[:sum(p.numel() for p in parts)])
        return s["arrays"]
    out = ctx.forward(s["model"], dense, s["out"])
    if case["task"] == "infer":
        return out
    if case["task"] == "train":
        grads = ctx.backward(s["model"], dense, s["d_out"])
        ctx.adagrad_step(s["model"], lr=1e-3)
        return {"rows": out, "grads": grads}
    grads, g_rows, _ = ctx.backward(s["model"], dense, s["d_out"], want_h0_grad=True)
    ctx.sgd_step(s["model"], lr=1e-3)
    ctx.apply_embedding_sgd(dense, g_rows, lr=1e-1)
    return {"rows": out, "grads": grads, "table": s["table"]}


def _run_lp(s):
    case, ctx = s["case"], s["ctx"]
    src, rel, dst = s["edges"]
    lp = ctx.lp_prepare(src, rel, dst, case["chunks"], case["negatives"], seed=s["seed"])
    targets = lp.targets()
    s["dense"] = dense = ctx.sample(targets, _fanouts(case), seed=s["seed"], out=s["dense"])
    rows = torch.empty((targets.numel(), case["hidden"]), device="cuda")
    if case["encoder"] == "gat":
        ctx.gat_forward(s["model"], dense, rows)
    else:
        ctx.forward(s["model"], dense, rows)
    scores = ctx.distmult_score(lp, rows, s["relations"])
    lp.free()
    return scores


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def _groups(case):
    """Nodes by the number of ones in their R-MAT id: (how many, expected degree in the buffer, share of the edge ends)."""
    n, keep = case["nodes"], case["resident"] / case["parts"]
    if case["graph"] == "er":
        return [(n, case["edges"] / n, 1.0)]
    bits = max(1, math.ceil(math.log2(n)))
    q, fit = 0.24, n / 2 ** bits
    share = [math.comb(bits, j) * q ** j * (1 - q) ** (bits - j) for j in range(bits + 1)]
    return [(math.comb(bits, j) * fit, keep * case["edges"] * p / (math.comb(bits, j) * fit), p) for j, p in enumerate(share)]


def _mean_taken(rate, fanout):
    """Expected min(degree, fanout) for a Poisson degree."""
    if rate > 30 + 2 * fanout:
        return float(fanout)
    p, kept, left = math.exp(-rate), 0.0, 1.0
    for d in range(fanout):
        kept += d * p
        left -= p
        p *= rate / (d + 1)
    return kept + fanout * max(0.0, left)


def _sizes(case):
    """Expected (nodes first reached per hop, entries per hop) of one mini-batch, and the distinct nodes of a whole call."""
    groups, keep = _groups(case), case["resident"] / case["parts"]
    lists = 2 if case["inout"] else 1
    total = sum(g[0] for g in groups)
    targets = [case["targets"] * g[0] / total for g in groups]
    if case["task"] == "lp":      # the ends of the edges follow the degrees, the negatives do not
        drawn, negatives = 2 * case["edges_scored"], case["chunks"] * case["negatives"]
        targets = [g[0] * keep * -math.expm1(-(drawn * g[2] + negatives * g[0] / total) / (g[0] * keep)) for g in groups]
    first = sum(targets)
    nodes, entries, ends, at = [first], [], 0.0, [t / first for t in targets]
    reached, level = first, first
    for f in _fanouts(case):
        e = level * lists * sum(w * _mean_taken(g[1], f) for w, g in zip(at, groups))
        ends += e
        seen = sum(g[0] * keep * -math.expm1(-ends * g[2] / (g[0] * keep)) for g in groups)
        level = max(0.0, min(first + seen, total * keep) - reached)
        reached += level
        nodes.append(level)
        entries.append(e)
        at = [g[2] for g in groups]
    drawn = case["batches"] * ends
    distinct = sum(g[0] * keep * -math.expm1(-(drawn * g[2] + case["batches"] * first * g[0] / total) / (g[0] * keep)) for g in groups)
    return nodes, entries, distinct


def work(case):
    """Bytes of the inputs read once (row bounds, picked ids, base rows, weights) and the outputs written once; flops of the linear maps."""
    nodes, entries, distinct = _sizes(case)
    b, hops, lists = case["batches"], case["hops"], 2 if case["inout"] else 1
    row = case["dim"] * (2 if case["half"] else 4)
    dims = [case["dim"]] + [case["hidden"]] * hops
    sampled = min(distinct, b * sum(nodes[:hops]))
    moved = 4 * b * nodes[0] + 16 * lists * sampled + 4 * b * sum(entries)
    maps = [2 * dims[l - 1] * dims[l] for l in range(1, hops + 1)]
    rows_of = [b * sum(nodes[:hops - l + 1]) for l in range(1, hops + 1)]      # output rows of layer l
    flops = sum(2 * r * m for r, m in zip(rows_of, maps))
    if case["task"] == "export":
        return {"bytes": moved + 4 * b * (sum(nodes) + sum(nodes[:hops]) + 2 * sum(entries)), "flops": 0}
    moved += distinct * row + 4 * sum(maps) + b * nodes[0] * dims[-1] * 4
    if case["task"] in ("train", "embed"):      # the loss's gradient in, the weights' gradients and the updated weights out
        moved += b * nodes[0] * dims[-1] * 4 + 3 * 4 * sum(maps)
        flops += sum(2 * r * m for r, m in zip(rows_of, maps)) + sum(2 * r * m for r, m in list(zip(rows_of, maps))[1:])
        if case["task"] == "embed":             # the rows' gradients, and the rows written back
            moved += distinct * row
            flops += 2 * rows_of[0] * maps[0]
    if case["task"] == "lp":
        scores = 2 * case["edges_scored"] * case["negatives"]
        flops = flops // (2 if case["encoder"] == "gat" else 1) + 2 * scores * case["dim"]
        moved += 12 * case["edges_scored"] + 4 * (scores + case["edges_scored"]) + 4 * N_RELATIONS * case["dim"] - nodes[0] * dims[-1] * 4
    return {"bytes": float(moved), "flops": float(flops)}


def tolerance(case):
    """Measured: the same cases on fp32 products (GEMM_FP32) against the default.  TF32 and fp16 operands keep ten bits: rows 3e-4 to 4.6e-4,
    scores 3e-4.  A gradient sees that twice, and where a row of a ReLU lies within rounding of zero its branch may change: 2.4e-2
    between fp32 and TF32 products, a hundredth between two that both round to ten bits."""
    if case["task"] == "export":
        return "exact"
    return {"rel": 1e-2 if case["task"] in ("train", "embed") else 2e-3}
