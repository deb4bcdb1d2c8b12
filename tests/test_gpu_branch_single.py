"""Branch decomposition where one branch is large.

Its vertices are sorted by value only, with their ids in place in the output
every other pass, so the number of passes (the 8-bit digits in which the keys
differ: none to four) decides where the sort begins. All outputs are whole
numbers: there is no tolerance.
"""

import numpy as np
import pytest
import torch

import paper_2301_10838_gb300 as mt

pytestmark = pytest.mark.gpu

# bits of the keys that differ: no pass to four, with gaps between the digits
MASKS = [0, 0x3F, 0x3F00, 0x7F0003, 0x00FFFF, 0xFFFFFF, 0x07000001, 0x07FFFFFF]


@pytest.mark.parametrize("n", [513, 5000, 300_001, 8_388_609])
@pytest.mark.parametrize("small", [[], [1, 512, 3]])
def test_one_large_branch(n, small):
    """n vertices: branches of the sizes in `small`, all others on the root's."""
    rng = np.random.default_rng(n + len(small))
    ids = rng.permutation(n + sum(small))
    n = len(ids)
    branch = np.empty(n, np.int64)
    at = 0
    for c in [n - sum(small), *small]:
        branch[ids[at:at + c]] = ids[at]
        at += c
    root, u = np.uint64(ids[0]), np.arange(n, dtype=np.uint64)
    head = branch == np.arange(n)
    s, v = np.where(head, root, u), np.where(head, root, branch.astype(np.uint64))
    Wd = torch.from_numpy(((s << np.uint64(32)) | v).view(np.int64)).cuda()
    order = torch.empty(n, dtype=torch.int32, device="cuda")
    offsets = torch.empty(n + 1, dtype=torch.int32, device="cuda")
    for mask in MASKS:
        f = (np.uint32(0x40000000) + (rng.integers(0, 1 << 27, size=n).astype(np.uint32) & np.uint32(mask))).view(np.float32)
        fd = torch.from_numpy(f.reshape(1, 1, n)).cuda()
        ws = mt.branches_workspace(mt.grid_of(fd))
        want = np.lexsort((np.arange(n), f, branch))
        starts = np.flatnonzero(np.r_[True, np.diff(branch[want]) != 0])
        order.fill_(-1)
        offsets.fill_(-1)
        k = mt.mt_branch_decomposition(fd, Wd, 0, order, offsets, ws)
        assert k == len(starts) == 1 + len(small)
        assert np.array_equal(offsets[:k + 1].cpu().numpy(), np.r_[starts, n])
        assert np.array_equal(order.cpu().numpy(), want), hex(mask)
