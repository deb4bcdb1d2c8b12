"""What a build that failed leaves behind: ids inside the field, in every word.

The calls report a value that is not finite in the status word. A caller that
goes on with the triplets all the same (another workspace, a cleared status)
must not be led out of the arrays by them.
"""

import numpy as np
import pytest
import torch

import paper_2301_10838_gb300 as mt
from paper_2301_10838_gb300 import fields

pytestmark = pytest.mark.gpu


def in_range(W, n, wide=False):
    w = W.cpu().numpy().view(np.uint64).reshape(-1)
    s, v = (w[0::2], w[1::2]) if wide else (w >> np.uint64(32), w & np.uint64(0xFFFFFFFF))
    return bool((s < n).all() and (v < n).all())


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, np.array(0x7FFFFFFF, np.uint32).view(np.float32)])
@pytest.mark.parametrize("shape", [(8, 8, 8), (33, 17, 48)])
def test_ids_stay_inside(shape, bad):
    f = fields.white_noise(shape, seed=3).copy()
    f[3, 4, 5] = bad
    d = torch.from_numpy(f).cuda()
    n, g = d.numel(), mt.grid_of(d)
    ws, wws = mt.workspace(g), mt.wide_workspace(g)
    labels = torch.empty(n, dtype=torch.int32, device="cuda")
    pairs = torch.empty((n, 2), dtype=torch.int32, device="cuda")
    for cfg in (0, mt.MT_CFG_LARGE_TILES):
        W = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        mt.mt_build_triplets_cfg(d, W, ws, 0, cfg)
        with pytest.raises(mt.MtError):
            mt.mt_sync_status(ws)
        assert in_range(W, n)
        mt.mt_components_at(d, W, 0.5, labels, ws)
        mt.mt_sync_status(ws)
        W.fill_(-1)
        with pytest.raises(mt.MtError):
            mt.mt_build_step(d, W, 0.5, labels, pairs, ws, cfg=cfg)
        assert in_range(W, n)
    W2 = torch.full((n, 2), -1, dtype=torch.int64, device="cuda")
    mt.mt_build_triplets_wide(d, W2, wws)
    with pytest.raises(mt.MtError):
        mt.mt_sync_status(wws)
    assert in_range(W2, n, wide=True)


def test_ids_of_a_batch_stay_inside():
    shapes = [(20, 16, 40), (5, 7, 9), (33, 17, 16)]
    flds = [fields.white_noise(s, seed=i).copy() for i, s in enumerate(shapes)]
    flds[1].flat[7] = np.nan
    grids = [mt.Grid(s[2], s[1], s[0]) for s in shapes]
    arena = torch.cat([torch.from_numpy(f).reshape(-1) for f in flds]).cuda()
    W = torch.full((arena.numel(),), -1, dtype=torch.int64, device="cuda")
    P = torch.empty((arena.numel(), 2), dtype=torch.int32, device="cuda")
    npairs = torch.zeros(len(shapes), dtype=torch.int64, device="cuda")
    ws = torch.empty(mt.mt_batch_workspace_bytes(grids), dtype=torch.uint8, device="cuda")
    mt.mt_batch_build(arena, grids, W, P, npairs, ws)
    with pytest.raises(mt.MtError):
        mt.mt_sync_status(ws)
    off = 0
    for s in shapes:
        n = int(np.prod(s))
        assert in_range(W[off:off + n], n)
        off += n
