"""Long thin grids of few values: chains of links over many tiles.

The merges between the tiles of such grids climb far, go on in their long form
and shorten the chains while others climb and displace them; grids of 64 tiles
and more are merged in scattered order. Every triplet, pair and label equals the
oracle's, in the single, wide and batched forms. All outputs are whole numbers:
there is no tolerance.
"""

import numpy as np
import pytest
import torch

import oracle
import paper_2301_10838_gb300 as mt
from paper_2301_10838_gb300.batch import Batch

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 20_011), (3, 3, 6_001), (3, 5_003, 3), (7_001, 3, 3), (8, 8, 4_100), (1, 33, 3_000), (1_024, 12, 12),
          (1_007, 1, 1), (1_009, 1, 16), (40, 700, 17)]


def make(shape, levels):
    if levels == 0:  # one plateau
        return np.zeros(shape, np.float32)
    if levels < 0:  # a falling ramp: every tile's saddles fall along the grid
        return -np.arange(np.prod(shape), dtype=np.float32).reshape(shape)
    return np.random.default_rng(levels).integers(0, levels, size=shape).astype(np.float32)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("levels", [0, -1, 2, 16, 256])
def test_thin_grids(shape, levels):
    f = np.ascontiguousarray(make(shape, levels))
    W_ref = oracle.merge_tree(f)
    p_ref, roots = oracle.pairs(W_ref)
    t = float(np.median(f))
    lab_ref = oracle.components(f, t)
    d = torch.from_numpy(f).cuda()
    n, g = d.numel(), mt.grid_of(d)
    ws, wws = mt.workspace(g), mt.wide_workspace(g)
    W = torch.empty(n, dtype=torch.int64, device="cuda")
    W2 = torch.empty((n, 2), dtype=torch.int64, device="cuda")
    labels = torch.empty(n, dtype=torch.int32, device="cuda")
    pairs = torch.empty((n, 2), dtype=torch.int32, device="cuda")
    for cfg in (0, mt.MT_CFG_LARGE_TILES):
        k, root = mt.mt_build_step(d, W, t, labels, pairs, ws, cfg=cfg)
        assert np.array_equal(W.cpu().numpy().view(np.uint64), W_ref)
        assert k == len(p_ref) and root == int(roots[0])
        assert np.array_equal(pairs[:k].cpu().numpy().view(np.uint32), p_ref)
        assert np.array_equal(labels.cpu().numpy().view(np.uint32), lab_ref)
    mt.mt_build_triplets_wide(d, W2, wws)
    mt.mt_sync_status(wws)
    w2 = W2.cpu().numpy().view(np.uint64)
    assert np.array_equal((w2[:, 0] << np.uint64(32)) | w2[:, 1], W_ref)


@pytest.mark.parametrize("levels", [0, 2, 16])
@pytest.mark.parametrize("cfg", [0, mt.MT_CFG_SMALL_TILES])
def test_thin_grids_in_a_batch(levels, cfg):
    fields = [make(s, levels) for s in SHAPES]
    b = Batch(SHAPES)
    b.load([np.ascontiguousarray(f) for f in fields])
    b.cfg = cfg
    b.launch()
    mt.mt_sync_status(b.ws)
    for i, f in enumerate(fields):
        W, p = b.results(i)
        W_ref = oracle.merge_tree(f)
        assert np.array_equal(W.cpu().numpy().view(np.uint64), W_ref), SHAPES[i]
        assert np.array_equal(p.cpu().numpy().view(np.uint32), oracle.pairs(W_ref)[0])
