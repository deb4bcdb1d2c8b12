"""The wide path's workspace over all shapes of grids (host logic, no GPU): a
small part of the 20 bytes per vertex that the field and the triplets take, also
where most of every tile lies outside the grid, and room for a bit per vertex
that the pair compaction leaves in the notes' place."""

from __future__ import annotations

import pytest

import paper_2301_10838_gb300 as mt


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2301_10838_gb300 import build

    build.build()


def wide_bytes(nx, ny, nz):
    return int(mt.load().mt_wide_workspace_bytes(mt.Grid(nx, ny, nz)))


@pytest.mark.parametrize("grid", [(1, 1, 1), (1, 1, 4096), (1 << 30, 1, 1), (1, 1 << 30, 1), (1, 1, 1 << 30),
                                  (2**32 - 1, 2, 1), (2, 1, 2**32 - 1), (3, 2**30 + 1, 4), (65536, 65536, 1), (1, 65536, 65536),
                                  (17, 17, 10**6), (15, 16, 10**6), (1700, 1700, 1600)])
def test_bytes_per_vertex(grid):
    nx, ny, nz = grid
    n = nx * ny * nz
    b = wide_bytes(*grid)
    assert b <= 4 * n + 4096  # less than the field itself
    chunks = -(-n // 4096)
    assert b >= 512 + 12 * chunks + chunks * 512
    if min(grid) >= 256:
        assert b <= 0.15 * n
