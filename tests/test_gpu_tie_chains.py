"""Climbs of the repair pass whose links tie with saddles outside their tile.

A link whose saddle has the key of the climb's level and lies outside the tile
is followed after a look at the ids, while other lanes of the warp go on by
comparing words. In the field below the lanes of two rows need such links one
after another, and each of them then a long chain of links of the same level
inside the tile, so that the warp's climb takes as many rounds as its lanes'
links add up to. All outputs are whole numbers: there is no tolerance.
"""

import numpy as np
import pytest
import torch

import oracle
import paper_2301_10838_gb300 as mt
from paper_2301_10838_gb300.batch import Batch

pytestmark = pytest.mark.gpu

NX, NY, NZ = 16, 16, 48


def tie_chains():
    """16 columns x (in rows y = 14, 15 by turns) rise to z = 46 and carry a
    vertex of value 1 at z = 47. Column x + 1 joins column x through a saddle of
    value 1 at z = 30 - x, below the tile of z = 32 .. 47, so the one with the
    later id lies nearer to column 0. From column 0 a falling path without
    chords winds through rows y = 0, 2, .. 12 of the planes z = 32, 34, .. 46;
    wherever its id exceeds that of the last saddle it has a vertex of value 1,
    which ends one basin and begins a deeper one. Everything else is a wall of
    10."""
    f = np.full((NZ, NY, NX), 10.0, np.float32)
    for x in range(NX):
        y, bottom = 14 + x % 2, 30 - x
        for z in range(bottom, 47):
            f[z, y, x] = 0.5 + 0.01 * x + 1e-4 * (z - bottom)
        f[47, y, x] = 1.0
        if x > 0:
            f[31 - x, y, x - 1] = 1.0
    path = [(30, y, 0) for y in range(13, -1, -1)] + [(31, 0, 0)]  # from column 0 to (0, 0, 32)
    for z in range(32, 48, 2):
        flip = (lambda x: x) if z % 4 == 0 else (lambda x: NX - 1 - x)  # every other plane is mirrored
        for y in range(0, 13, 2):  # rows of 14 forth and back ...
            path += [(z, y, flip(x)) for x in (range(14) if y % 4 == 0 else range(13, -1, -1))]
            if y < 12:
                path.append((z, y + 1, path[-1][2]))
        path += [(z, 12, flip(14))] + [(z, y, flip(15)) for y in range(12, -1, -1)]  # ... and back beside them
        path.append((z + 1, 0, flip(15)))
    last, since, nsad = 0, 0, 0
    for p, (z, y, x) in enumerate(path[:-1]):
        gid = x + NX * (y + NY * z)
        since += 1
        if z >= 32 and gid > last and since >= 2:
            f[z, y, x], last, since, nsad = 1.0, gid, 0, nsad + 1
        else:
            f[z, y, x] = 0.4 - 1e-4 * p
    return f, nsad


def test_tie_chains_equal_the_oracle():
    f, nsad = tie_chains()
    assert nsad > 2 * 1280 / 16  # twice the nodes of a tile, over the lanes that need the path in turn
    W_ref = oracle.merge_tree(f)
    # the links are as meant: 15 of value 1 outside the tile from the last
    # column to the first, then those of the path
    n = f.size
    s, v = (W_ref >> np.uint64(32)).astype(np.int64), (W_ref & np.uint64(0xFFFFFFFF)).astype(np.int64)
    x, links = 15 + NX * (15 + NY * 15), 0  # the bottom of column 15
    while v[x] != x:
        assert f.reshape(-1)[s[x]] == 1.0
        x, links = v[x], links + 1
    assert links >= 15 + nsad
    p_ref, roots = oracle.pairs(W_ref)
    d = torch.from_numpy(f).cuda()
    ws = mt.workspace(mt.grid_of(d))
    W = torch.empty(n, dtype=torch.int64, device="cuda")
    labels = torch.empty(n, dtype=torch.int32, device="cuda")
    pairs = torch.empty((n, 2), dtype=torch.int32, device="cuda")
    for cfg in (0, mt.MT_CFG_LARGE_TILES):
        mt.mt_build_triplets_cfg(d, W, ws, 0, cfg)
        mt.mt_sync_status(ws)
        assert np.array_equal(W.cpu().numpy().view(np.uint64), W_ref)
        for t in (0.55, 1.0, 10.0):
            k, root = mt.mt_build_step(d, W, t, labels, pairs, ws, cfg=cfg)
            assert np.array_equal(W.cpu().numpy().view(np.uint64), W_ref)
            assert np.array_equal(labels.cpu().numpy().view(np.uint32), oracle.components(f, t))
            assert k == len(p_ref) and root == int(roots[0])
            assert np.array_equal(pairs[:k].cpu().numpy().view(np.uint32), p_ref)


def test_tie_chains_wide():
    f, _ = tie_chains()
    d = torch.from_numpy(f).cuda()
    ws = mt.wide_workspace(mt.grid_of(d))
    W2 = torch.empty((f.size, 2), dtype=torch.int64, device="cuda")
    mt.mt_build_triplets_wide(d, W2, ws)
    mt.mt_sync_status(ws)
    assert np.array_equal(W2.cpu().numpy().view(np.uint64), oracle.merge_tree_wide(f))


@pytest.mark.parametrize("cfg", [0, mt.MT_CFG_SMALL_TILES])
def test_tie_chains_batch(cfg):
    f, _ = tie_chains()
    b = Batch([f.shape] * 2)
    b.load([f, f[:, ::-1].copy()])
    b.cfg = cfg
    b.launch()
    mt.mt_sync_status(b.ws)
    for i, g in enumerate([f, f[:, ::-1].copy()]):
        W, p = b.results(i)
        W_ref = oracle.merge_tree(g)
        assert np.array_equal(W.cpu().numpy().view(np.uint64), W_ref)
        assert np.array_equal(p.cpu().numpy().view(np.uint32), oracle.pairs(W_ref)[0])
