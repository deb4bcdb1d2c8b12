"""Every route of the pair compaction, on both sides of the number of chunks up
to which the writer sums the counts itself (4096 chunks of 4096 vertices).

The one-call step with the pairs marked in its repair pass, the separate calls
with room for a bit per vertex in their workspace and without (a workspace of
the compaction part alone), with and without a persistence to keep, for both
trees and tile shapes: all give one list, which for one of the fields is also
the oracle's. All outputs are whole numbers: there is no tolerance.
"""

import numpy as np
import pytest
import torch

import oracle
import paper_2301_10838_gb300 as mt
from paper_2301_10838_gb300 import fields

pytestmark = pytest.mark.gpu

CHUNK = 4096


@pytest.mark.parametrize("shape", [(261, 257, 256), (128, 256, 512), (33, 40, 96)])
@pytest.mark.parametrize("flags", [0, mt.MT_SUPERLEVEL])
def test_routes_agree(shape, flags):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(23)
    f = torch.rand(shape, generator=gen, device="cuda")
    f = torch.floor(f * 512) / 512 if flags else f  # with ties in one of the trees
    n, g = f.numel(), mt.grid_of(f)
    ws = mt.workspace(g)
    part = 512 + (-(-n // CHUNK) * 4 + 255) // 256 * 256  # status, counters, a count per chunk
    small = torch.zeros(part, dtype=torch.uint8, device="cuda")
    W = torch.empty(n, dtype=torch.int64, device="cuda")
    mt.mt_build_triplets_ex(f, W, ws, flags)
    mt.mt_sync_status(ws)
    W2, labels = torch.empty_like(W), torch.empty(n, dtype=torch.int32, device="cuda")
    cap = n // 4
    a, b = (torch.empty((cap, 2), dtype=torch.int32, device="cuda") for _ in range(2))
    for eps in (0.0, 0.4):
        a.fill_(-1)
        k, root = mt.mt_simplified_pairs(f, W, eps, flags, a, small)
        assert 0 < k < cap
        b.fill_(-1)
        assert mt.mt_simplified_pairs(f, W, eps, flags, b, ws) == (k, root) and torch.equal(a, b)
        for cfg in (0, mt.MT_CFG_LARGE_TILES):
            b.fill_(-1)
            got = mt.mt_build_step(f, W2, 0.5, labels, b, ws, eps=eps, flags=flags, cfg=cfg)
            assert got == (k, root) and torch.equal(a, b) and torch.equal(W, W2)
        if flags == 0:
            want = oracle.simplified_pairs(f.cpu().numpy(), W.cpu().numpy().view(np.uint64), eps)
            assert np.array_equal(a[:k].cpu().numpy().view(np.uint32), want)


def test_step_counts_past_the_end_of_the_list():
    shape = (261, 257, 256)
    f = torch.rand(shape, device="cuda")
    n, g = f.numel(), mt.grid_of(f)
    ws = mt.workspace(g)
    W = torch.empty(n, dtype=torch.int64, device="cuda")
    labels = torch.empty(n, dtype=torch.int32, device="cuda")
    full = torch.empty((n // 4, 2), dtype=torch.int32, device="cuda")
    k, root = mt.mt_build_step(f, W, 0.5, labels, full, ws)
    part = torch.full((k // 2 + 9, 2), -1, dtype=torch.int32, device="cuda")
    assert mt.mt_build_step(f, W, 0.5, labels, part[:k // 2], ws, allow_partial=True) == (k, root)
    assert torch.equal(part[:k // 2], full[:k // 2]) and bool((part[k // 2:] == -1).all())


@pytest.mark.slow
def test_step_equals_the_calls_1024():
    """The benchmark's step on its field: the one-call form, whose pairs are
    marked in the repair pass, against the three calls (whose results the
    full-size test compares with the oracle)."""
    f = fields.named_field("lognorm1024", seed=1, device="cuda").contiguous()
    n, g = f.numel(), mt.grid_of(f)
    t = float(f.reshape(-1)[::4099].median())
    ws = mt.workspace(g)
    W, W2 = (torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(2))
    la, lb = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
    a, b = (torch.full((n // 8, 2), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    mt.mt_build_triplets(f, W, ws)
    mt.mt_components_at(f, W, t, la, ws)
    for eps in (0.0, 0.5):
        a.fill_(-1)
        b.fill_(-1)
        k, root = mt.mt_simplified_pairs(f, W, eps, 0, a, ws)
        assert mt.mt_build_step(f, W2, t, lb, b, ws, eps=eps) == (k, root)
        assert torch.equal(W, W2) and torch.equal(a, b)
        if eps > 0:
            mt.mt_simplified_components_at(f, W, t, eps, 0, la, ws)
            mt.mt_sync_status(ws)
        assert torch.equal(la, lb)
