"""Branch decomposition over branch sizes chosen one by one.

The call sorts small branches in shared memory, large ones by radix passes and
the root's branch apart on large grids. The trees here are made up so that
branches of the sizes where that changes occur (the call reads only each
vertex's branch off the triplets), with values that tie; the expected grouping
is numpy's stable sort by (branch, value, index). All outputs are whole
numbers: there is no tolerance.
"""

import numpy as np
import pytest
import torch

import paper_2301_10838_gb300 as mt

pytestmark = pytest.mark.gpu


def made_up(n, sizes, root_size, levels, seed):
    """Branch of every vertex (heads at random ids), values, triplet words."""
    rng = np.random.default_rng(seed)
    ids = rng.permutation(n)
    branch = np.empty(n, np.int64)
    at = 0
    for c in [root_size, *sizes]:
        c = min(c, n - at)
        if c <= 0:
            break
        branch[ids[at:at + c]] = ids[at]
        at += c
    branch[ids[at:]] = ids[at:]  # the rest: branches of one vertex
    f = rng.integers(-levels, levels, size=n).astype(np.float32)
    f[branch == ids[0]] *= -0.0 if levels == 1 else 1.0
    u = np.arange(n, dtype=np.uint64)
    head = branch == np.arange(n)
    s = np.where(head, np.uint64(ids[0]), u)  # a head's saddle: any other vertex
    v = branch.astype(np.uint64)
    s[ids[0]] = v[ids[0]] = np.uint64(ids[0])  # the root
    v = np.where(head & (u != np.uint64(ids[0])), np.uint64(ids[0]), v)
    return branch, f, (s << np.uint64(32)) | v


CASES = [
    (1, [], 1, 4), (2, [], 2, 1), (33, [5], 7, 2), (1024, [511, 2], 100, 3), (1025, [512, 300], 200, 9),
    (4096, [513, 512, 511, 1], 1500, 1), (40_000, [1024, 1025, 513, 64, 33, 32, 31], 20_000, 50),
    (70_001, [600] * 100, 40, 7), (3_000_000, [8191, 8192, 8193, 70_000] + [514] * 300, 2_000_000, 5),
    (8_600_000, [513, 100_000, 512] + [700] * 20, 5_000_003, 4), (8_500_000, [], 8_500_000, 3),
    (8_400_000, [4_000_000, 1000], 512, 100_000),
]


@pytest.mark.parametrize("n,sizes,root_size,levels", CASES)
def test_branch_sizes(n, sizes, root_size, levels):
    branch, f, W = made_up(n, sizes, root_size, levels, n % 97)
    want = np.lexsort((np.arange(n), f, branch))
    starts = np.flatnonzero(np.r_[True, np.diff(branch[want]) != 0])
    fd = torch.from_numpy(f.reshape(1, 1, n)).cuda()
    Wd = torch.from_numpy(W.view(np.int64)).cuda()
    ws = mt.branches_workspace(mt.grid_of(fd))
    order = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    offsets = torch.full((n + 1,), -1, dtype=torch.int32, device="cuda")
    k = mt.mt_branch_decomposition(fd, Wd, 0, order, offsets, ws)
    assert k == len(starts)
    assert np.array_equal(offsets[:k + 1].cpu().numpy(), np.r_[starts, n])
    assert np.array_equal(order.cpu().numpy(), want)
