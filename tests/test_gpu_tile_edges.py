"""The tile kernel where its tables and bit columns reach their ends.

Fields whose tiles keep far more edges than the list holds (isolated maxima,
each of whose six lower neighbours is a component of its own), fields whose
levels tie along whole faces, and sides around multiples of the tile's, each
equal to the oracle in every triplet, pair and label. All outputs are whole
numbers: there is no tolerance.
"""

import numpy as np
import pytest
import torch

import oracle
import paper_2301_10838_gb300 as mt

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16, 16), (15, 17, 16), (33, 16, 31), (48, 32, 34), (1, 16, 47), (16, 1, 1)]


def make(kind, shape, rng):
    z, y, x = np.indices(shape)
    if kind == "isolated_maxima":  # every other vertex is a maximum, its neighbours minima of their own
        f = rng.random(shape, dtype=np.float32)
        return np.where((x + y + z) % 2 == 0, f, f + 2).astype(np.float32)
    if kind == "flat_faces":  # constant on slabs, so that parallel edges tie across every tile face
        return ((x // 5 + 2 * (y // 7) + 3 * (z // 3)) % 4).astype(np.float32)
    if kind == "ramp":  # one minimum: columns of lower-than bits are all ones or all zeros
        return (x + 100 * y + 10000 * z).astype(np.float32)
    return -(x + 100 * y + 10000 * z).astype(np.float32)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["isolated_maxima", "flat_faces", "ramp", "falling_ramp"])
def test_tile_edges(shape, kind):
    f = np.ascontiguousarray(make(kind, shape, np.random.default_rng(5)))
    W_ref = oracle.merge_tree(f)
    p_ref, roots = oracle.pairs(W_ref)
    t = float(np.median(f))
    lab_ref = oracle.components(f, t)
    d = torch.from_numpy(f).cuda()
    n = d.numel()
    ws = mt.workspace(mt.grid_of(d))
    for cfg in (0, mt.MT_CFG_LARGE_TILES):
        W = torch.empty(n, dtype=torch.int64, device="cuda")
        labels = torch.empty(n, dtype=torch.int32, device="cuda")
        pairs = torch.empty((n, 2), dtype=torch.int32, device="cuda")
        k, root = mt.mt_build_step(d, W, t, labels, pairs, ws, cfg=cfg)
        assert np.array_equal(W.cpu().numpy().view(np.uint64), W_ref)
        assert k == len(p_ref) and root == int(roots[0])
        assert np.array_equal(pairs[:k].cpu().numpy().view(np.uint32), p_ref)
        assert np.array_equal(labels.cpu().numpy().view(np.uint32), lab_ref)
    wws = mt.wide_workspace(mt.grid_of(d))
    W2 = torch.empty((n, 2), dtype=torch.int64, device="cuda")
    mt.mt_build_triplets_wide(d, W2, wws)
    mt.mt_sync_status(wws)
    w2 = W2.cpu().numpy().view(np.uint64)
    assert np.array_equal((w2[:, 0] << np.uint64(32)) | w2[:, 1], W_ref)
