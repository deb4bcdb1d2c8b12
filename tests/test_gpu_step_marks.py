"""The pairs that the one-call step marks inside the repair pass.

With rows that fill whole pieces of the bits the step takes its pairs from
there; they must be those of the separate calls, with and without a persistence
to keep, in both tile shapes, and where a tile has more minima than the pass
keeps nodes for. All outputs are whole numbers: there is no tolerance.
"""

import numpy as np
import pytest
import torch

import paper_2301_10838_gb300 as mt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(16, 16, 16), (9, 21, 32), (33, 17, 48), (40, 40, 64), (1, 1, 4112)])
@pytest.mark.parametrize("kind", ["noise", "ties", "checkerboard"])
def test_step_pairs_are_those_of_the_calls(shape, kind):
    rng = np.random.default_rng(11)
    f = rng.random(shape, dtype=np.float32) if kind != "ties" else rng.integers(-2, 3, size=shape).astype(np.float32)
    if kind == "checkerboard":  # half the vertices of a tile are minima
        z, y, x = np.indices(shape)
        f = np.where((x + y + z) % 2 == 0, f, f + 2).astype(np.float32)
    d = torch.from_numpy(np.ascontiguousarray(f)).cuda()
    n = d.numel()
    ws, ws2 = mt.workspace(mt.grid_of(d)), mt.workspace(mt.grid_of(d))
    t = float(np.median(f))
    for flags in (0, mt.MT_SUPERLEVEL):
        W = torch.empty(n, dtype=torch.int64, device="cuda")
        mt.mt_build_triplets_ex(d, W, ws, flags)
        for eps in (0.0, 0.4):
            want = torch.full((n, 2), -1, dtype=torch.int32, device="cuda")
            k, root = mt.mt_simplified_pairs(d, W, eps, flags, want, ws)
            for cfg in (0, mt.MT_CFG_LARGE_TILES):
                W2 = torch.empty(n, dtype=torch.int64, device="cuda")
                labels = torch.empty(n, dtype=torch.int32, device="cuda")
                pairs = torch.full((n, 2), -1, dtype=torch.int32, device="cuda")
                got = mt.mt_build_step(d, W2, t, labels, pairs, ws2, eps=eps, flags=flags, cfg=cfg)
                assert got == (k, root)
                assert torch.equal(W2, W) and torch.equal(pairs, want)
