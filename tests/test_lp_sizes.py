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
