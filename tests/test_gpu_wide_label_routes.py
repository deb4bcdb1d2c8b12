"""Labels with wide ids on both sides of the rule that chooses bricks.

Grids at the limits of the rule (2^23 vertices, four planes, three in four
columns of the bricks inside the grid), labelled from wide triplets; the labels
are those of the oracle, widened. All outputs are whole numbers: there is no
tolerance.
"""

import numpy as np
import pytest
import torch

import oracle
import paper_2301_10838_gb300 as mt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 1024, 2048), (4, 1024, 2047), (3, 1024, 2731), (62, 2823, 48), (62, 2900, 47),
                                   (1, 1, 70001), (20, 33, 31)])
def test_both_routes(shape):
    rng = np.random.default_rng(17)
    f = rng.integers(0, 40, size=shape).astype(np.float32)
    f += (rng.random(shape) < 0.5) * rng.random(shape).astype(np.float32)
    f = np.ascontiguousarray(f, dtype=np.float32)
    d = torch.from_numpy(f).cuda()
    n, g = d.numel(), mt.grid_of(d)
    ws = mt.wide_workspace(g)
    W2 = torch.empty((n, 2), dtype=torch.int64, device="cuda")
    labels = torch.empty(n, dtype=torch.int64, device="cuda")
    for flags, t, ref in ((0, 12.0, lambda: oracle.components(f, 12.0)),
                          (mt.MT_SUPERLEVEL, 30.25, lambda: oracle.components(-f, -30.25))):
        mt.mt_build_triplets_wide(d, W2, ws, flags)
        labels.fill_(-7)
        mt.mt_components_at_wide(d, W2, t, flags, labels, ws)
        mt.mt_sync_status(ws)
        want = ref().astype(np.int64)
        want[want == 0xFFFFFFFF] = -1
        assert np.array_equal(labels.cpu().numpy(), want)


@pytest.mark.parametrize("shape", [(9, 10, 11), (4, 1024, 2048)])
def test_ids_outside_the_grid_are_reported(shape):
    d = torch.rand(shape, device="cuda")
    n, g = d.numel(), mt.grid_of(d)
    ws = mt.wide_workspace(g)
    W2 = torch.empty((n, 2), dtype=torch.int64, device="cuda")
    mt.mt_build_triplets_wide(d, W2, ws)
    labels = torch.empty(n, dtype=torch.int64, device="cuda")
    for row in ((77, n), (n, 3), (n, n)):  # an inner vertex's target, a saddle, both
        bad = W2.clone()
        bad[77] = torch.tensor(row, dtype=torch.int64)
        mt.mt_components_at_wide(d, bad, 2.0, 0, labels, ws)
        with pytest.raises(mt.MtError) as e:
            mt.mt_sync_status(ws)
        assert e.value.code == -1
