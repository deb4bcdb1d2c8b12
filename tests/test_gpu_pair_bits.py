"""The pair compaction with and without a bit per vertex, and into lists that
are only aligned as the call asks.

The allocation-free call has room for the bits only up to about 8 million
vertices; past that both passes read the triplets. All outputs are whole
numbers: there is no tolerance.
"""

import numpy as np
import pytest
import torch

import oracle
import paper_2301_10838_gb300 as mt
from paper_2301_10838_gb300 import fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,eps", [((210, 210, 210), 0.0), ((64, 65, 63), 0.0), ((64, 65, 63), 0.3), ((1, 1, 33), 0.0)])
def test_with_and_without_bits(shape, eps):
    f = torch.from_numpy(fields.white_noise(shape, 3)).cuda()
    n = f.numel()
    ws = mt.workspace(mt.grid_of(f))
    W = torch.empty(n, dtype=torch.int64, device="cuda")
    mt.mt_build_triplets(f, W, ws)
    flat = torch.full((2 * n + 2,), -1, dtype=torch.int32, device="cuda")
    pairs = flat[1:2 * n + 1].view(n, 2)  # 4-byte aligned only
    if eps > 0:
        k, _ = mt.mt_simplified_pairs(f, W, eps, 0, pairs, ws)
        want = oracle.simplified_pairs(f.cpu().numpy(), W.cpu().numpy().view(np.uint64), eps)
        assert np.array_equal(pairs[:k].cpu().numpy().view(np.uint32), want)
    else:
        k, root = mt.mt_persistence_pairs(f, W, pairs, ws)
        again = torch.full((n, 2), -1, dtype=torch.int32, device="cuda")
        k2, root2 = mt.mt_persistence_pairs_noalloc(f, W, again)
        assert (k, root) == (k2, root2) and torch.equal(pairs, again)
        want, _ = oracle.pairs(W.cpu().numpy().view(np.uint64))
        assert np.array_equal(pairs[:k].cpu().numpy().view(np.uint32), want)
    assert int(flat[0]) == -1 and int(flat[2 * n + 1]) == -1 and bool((pairs[k:] == -1).all())


def test_wide_list_alignment():
    shape = (20, 33, 47)
    f = torch.from_numpy(fields.white_noise(shape, 4)).cuda()
    n, grid = f.numel(), mt.grid_of(f)
    ws = mt.wide_workspace(grid)
    W2 = torch.empty((n, 2), dtype=torch.int64, device="cuda")
    mt.mt_build_triplets_wide(f, W2, ws)
    flat = torch.full((2 * n + 2,), -1, dtype=torch.int64, device="cuda")
    pairs = flat[1:2 * n + 1].view(n, 2)  # 8-byte aligned only
    k, _ = mt.mt_persistence_pairs_wide(W2, grid, pairs, ws)
    want, _ = oracle.pairs(oracle.merge_tree(f.cpu().numpy()))
    assert np.array_equal(pairs[:k].cpu().numpy(), want.astype(np.int64))
    assert int(flat[0]) == -1 and bool((flat[2 * k + 1:] == -1).all())
