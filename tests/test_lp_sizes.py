"""Link prediction at the sizes where its kernels are cut: nodes around the tiles of the target union's bitmap (65,536), few and
many edges per warp of the positive scores."""
import numpy as np
import pytest
import torch

import paper_2202_02365_b200 as mg
from paper_2202_02365_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,edges,chunks,negs", [(33, 1, 1, 1), (65_535, 37, 2, 16), (65_536, 4_000, 3, 100), (65_537, 5, 5, 0), (2_300_000, 50_001, 7, 333)])
def test_target_union(nodes, edges, chunks, negs):
    ctx = mg.Context(0)
    g = inputs.erdos_renyi_graph(nodes, 2 * nodes, seed=1, device="cuda")
    ctx.load_graph(g.row_offsets, g.nbrs)
    ctx.load_features(torch.zeros((nodes, 4), device="cuda"))
    rng = np.random.RandomState(2)
    src, dst = (torch.from_numpy(rng.randint(0, nodes, edges).astype(np.int32)) for _ in range(2))
    src[0], dst[-1] = 0, nodes - 1          # the first and the last bit
    lp = ctx.lp_prepare(src, torch.zeros(edges, dtype=torch.int32), dst, chunks, negs, seed=3)
    v = {k: x.cpu().numpy() for k, x in lp.view().items()}
    ids = np.concatenate([src.numpy(), dst.numpy(), v["neg_ids"].ravel()])
    assert np.array_equal(v["targets"], np.unique(ids))
    assert np.array_equal(v["targets"][v["src_idx"]], src.numpy()) and np.array_equal(v["targets"][v["dst_idx"]], dst.numpy())
    assert np.array_equal(v["targets"][v["neg_idx"]], v["neg_ids"])


@pytest.mark.parametrize("dim,edges", [(4, 1), (100, 5), (128, 37), (60, 40_003)])
def test_positive_scores_beside_the_operand_images(dim, edges):
    nodes = 70_000
    ctx = mg.Context(0)
    g = inputs.erdos_renyi_graph(nodes, 2 * nodes, seed=1, device="cuda")
    ctx.load_graph(g.row_offsets, g.nbrs)
    ctx.load_features(torch.zeros((nodes, 4), device="cuda"))
    rng = np.random.RandomState(4)
    src, dst, rel = (torch.from_numpy(rng.randint(0, n, edges).astype(np.int32)) for n in (nodes, nodes, 50))
    lp = ctx.lp_prepare(src, rel, dst, 1, 24, seed=5)
    v = lp.view()
    h = inputs.normal_features(v["targets"].numel(), dim, seed=6, device="cuda")
    r = inputs.normal_features(50, dim, seed=7, device="cuda")
    pos, nd, ns = ctx.distmult_score(lp, h, r)
    s, o, w = h[v["src_idx"].long()].double(), h[v["dst_idx"].long()].double(), r[rel.cuda().long()].double()
    n = h[v["neg_idx"][0].long()].double()
    # fp32: two roundings a product and at most 128 of them summed, 2^-24 each, against the norm of the terms
    terms = (s * w * o).square().sum(1).sqrt()
    assert float(((pos.double() - (s * w * o).sum(1)).abs() / terms).max()) < 1e-5
    for got, want in ((nd, (s * w) @ n.T), (ns, (o * w) @ n.T)):
        assert float((got.double() - want).norm() / want.norm()) < 1e-3      # operands rounded to ten bits


# tiles of both sides in one launch: none left over a round of 148, some that are cut into parts, too many to cut; parts of unequal
# runs of negatives; one side alone
@pytest.mark.parametrize("edges,chunks,negs,corrupt", [(9_472, 1, 40, mg.CORRUPT_BOTH), (20_000, 1, 600, mg.CORRUPT_BOTH), (18_000, 9, 130, mg.CORRUPT_BOTH),
                                                       (3_001, 2, 1_000, mg.CORRUPT_SRC), (127, 1, 333, mg.CORRUPT_DST)])
def test_negative_scores_by_the_number_of_tiles(edges, chunks, negs, corrupt):
    nodes, dim = 30_000, 36
    ctx = mg.Context(0)
    g = inputs.erdos_renyi_graph(nodes, 2 * nodes, seed=1, device="cuda")
    ctx.load_graph(g.row_offsets, g.nbrs)
    ctx.load_features(torch.zeros((nodes, 4), device="cuda"))
    rng = np.random.RandomState(4)
    src, dst, rel = (torch.from_numpy(rng.randint(0, n, edges).astype(np.int32)) for n in (nodes, nodes, 50))
    lp = ctx.lp_prepare(src, rel, dst, chunks, negs, seed=5)
    v = lp.view()
    h = inputs.normal_features(v["targets"].numel(), dim, seed=6, device="cuda")
    r = inputs.normal_features(50, dim, seed=7, device="cuda")
    _, nd, ns = ctx.distmult_score(lp, h, r, corrupt)
    w = r[rel.cuda().long()].double()
    chunk = torch.arange(edges, device="cuda") * chunks // edges
    for got, keep in ((nd, v["src_idx"]), (ns, v["dst_idx"])):
        assert (got is None) == (not corrupt & (mg.CORRUPT_DST if keep is v["src_idx"] else mg.CORRUPT_SRC))
        for c in range(chunks if got is not None else 0):
            mine = chunk == c
            want = (h[keep.long()][mine].double() * w[mine]) @ h[v["neg_idx"][c].long()].double().T
            # operands rounded to ten bits, sums of 36 products: below 1e-3 of the norm, no value off by 1 % of the rows' rms
            err = got[mine].double() - want
            assert float(err.norm() / want.norm()) < 1e-3 and float(err.abs().max() / want.square().mean().sqrt()) < 1e-2


# rows of scores that start 32-byte aligned (stored as they are), 16-byte aligned, and neither; widths that end inside a slice of 32 columns
@pytest.mark.parametrize("edges,chunks,negs", [(500, 2, 8), (131, 1, 104), (1_000, 3, 500), (300, 1, 996), (300, 1, 1_001)])
def test_negative_scores_by_the_alignment_of_their_rows(edges, chunks, negs):
    test_negative_scores_by_the_number_of_tiles(edges, chunks, negs, mg.CORRUPT_BOTH)


# rows of whole 128-byte lines, which are stored by lines: within one slice of 32 columns and one block of them, several of each; every second row on a line
@pytest.mark.parametrize("edges,chunks,negs", [(131, 1, 32), (300, 2, 128), (257, 3, 1_504), (300, 1, 2_048), (300, 1, 1_008)])
def test_negative_scores_in_rows_of_whole_lines(edges, chunks, negs):
    test_negative_scores_by_the_number_of_tiles(edges, chunks, negs, mg.CORRUPT_BOTH)


# batches are prepared while the scores of the ones before are computed, in the blocks of freed batches: growing, shrinking, two alive at once
@pytest.mark.parametrize("sizes", [[40_000] * 6, [100, 40_000, 300, 50_000, 20_000, 60_000]])
def test_batches_prepared_beside_scores(sizes):
    nodes, dim = 400_000, 64
    ctx = mg.Context(0)
    g = inputs.erdos_renyi_graph(nodes, 2 * nodes, seed=1, device="cuda")
    ctx.load_graph(g.row_offsets, g.nbrs)
    ctx.load_features(torch.zeros((nodes, 4), device="cuda"))
    r = inputs.normal_features(50, dim, seed=7, device="cuda")
    table = inputs.normal_features(nodes, dim, seed=6, device="cuda")
    rng = np.random.RandomState(4)
    batches = [tuple(torch.from_numpy(rng.randint(0, n, e).astype(np.int32)) for n in (nodes, 50, nodes)) for e in sizes]

    def score(i, wait):
        lp = ctx.lp_prepare(*batches[i], 4, 500, seed=i)
        h = table[lp.targets().long()]
        if wait:
            torch.cuda.synchronize()
        out = ctx.distmult_score(lp, h, r)
        if wait:
            torch.cuda.synchronize()
        return lp, out

    got, held = [], None
    for i in range(len(sizes)):
        lp, out = score(i, False)
        got.append(out)
        if i % 3 == 1:
            held = lp                       # freed a batch later
        else:
            lp.free()
            if held is not None:
                held.free()
                held = None
    for i in range(len(sizes)):
        lp, want = score(i, True)
        lp.free()
        for x, y in zip(got[i], want):
            assert torch.equal(x, y), i


# neither side corrupted: only the positives, from rows that may start anywhere
@pytest.mark.parametrize("start", [0, 1])
@pytest.mark.parametrize("precision", [mg.GEMM_TF32, mg.GEMM_FP32])
def test_positive_scores_alone(start, precision):
    nodes, dim, edges = 5_000, 36, 700
    ctx = mg.Context(0)
    g = inputs.erdos_renyi_graph(nodes, 2 * nodes, seed=1, device="cuda")
    ctx.load_graph(g.row_offsets, g.nbrs)
    rng = np.random.RandomState(4)
    src, dst, rel = (torch.from_numpy(rng.randint(0, n, edges).astype(np.int32)) for n in (nodes, nodes, 50))
    lp = ctx.lp_prepare(src, rel, dst, 2, 30, seed=5)
    v = lp.view()

    def rows(n, seed):
        x = torch.zeros(n * dim + 4, device="cuda")[start:start + n * dim].view(n, dim)
        return x.copy_(inputs.normal_features(n, dim, seed=seed, device="cuda"))

    h, r = inputs.normal_features(v["targets"].numel(), dim, seed=6, device="cuda"), rows(50, 7)
    pos, nd, ns = ctx.distmult_score(lp, h, r, 0, precision)
    terms = h[v["src_idx"].long()].double() * r[rel.cuda().long()].double() * h[v["dst_idx"].long()].double()
    assert nd is None and ns is None
    assert float(((pos.double() - terms.sum(1)).abs() / terms.square().sum(1).sqrt()).max()) < 1e-5
