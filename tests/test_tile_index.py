"""Local ids, tile sides and the order of the tiles against exact arithmetic, on the CPU.

csrc/mt_index.h finds a vertex's place in its tile by reciprocals; here it is
compiled for the host and compared with 64-bit division, with 32-bit and 64-bit
ids, over grids with sides from 1 to 2^32 - 1: thin ones, ragged ones, rows so
long that 16 of them pass 2^32. Whole numbers: there is no tolerance.
"""

from __future__ import annotations

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2301_10838_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "mt_index.h"
using namespace mt;
typedef unsigned long long u64;
static u64 s = 12345;
static u64 rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static u64 bad = 0, in_tile = 0;

template <int LX, int LY, int LZ, class Id>
void grid(u64 nx, u64 ny, u64 nz)
{
    const u64 TX = 1u << LX, TY = 1u << LY, TZ = 1u << LZ, nxy = nx * ny, n = nxy * nz;
    const float rnxy = 1.0f / (float)(Id)nxy, rnx = 1.0f / (float)(uint32_t)nx;
    for (int k = 0; k < 24; k++) {
        // a tile: the first, the last, or any
        auto at = [&](u64 m, u64 t) { const u64 c = (m + t - 1) / t; return (k == 0 ? 0 : k == 1 ? c - 1 : rnd() % c) * t; };
        const u64 x0 = at(nx, TX), y0 = at(ny, TY), z0 = at(nz, TZ), base = z0 * nxy + y0 * nx + x0;
        const u64 wx = nx - x0 < TX ? nx - x0 : TX, wy = ny - y0 < TY ? ny - y0 : TY, wz = nz - z0 < TZ ? nz - z0 : TZ;
        for (int q = 0; q < 200; q++) {
            u64 v;  // in the tile, near one of its rows' ends, or anywhere
            const u64 r = base + rnd() % wz * nxy + rnd() % wy * nx;
            if (q % 3 == 0) v = r + rnd() % wx;
            else if (q % 3 == 1) v = r + (rnd() & 1 ? nx : 0) + rnd() % 35 - 17;
            else v = rnd();
            v %= n;
            const u64 x = v % nx, y = v / nx % ny, z = v / nxy;
            const bool in = x >= x0 && x < x0 + wx && y >= y0 && y < y0 + wy && z >= z0 && z < z0 + wz;
            const uint32_t want = in ? (uint32_t)(x - x0 + TX * (y - y0 + TY * (z - z0))) : kNoLocal;
            const uint32_t got = tile_local<LX, LY, LZ, Id>((Id)v - (Id)base, (Id)nxy, (uint32_t)nx, rnxy, rnx,
                                                            (uint32_t)wx, (uint32_t)wy, (uint32_t)wz);
            in_tile += in;
            if (got != want && bad++ < 5)
                printf("%d-bit ids, %llu x %llu x %llu: vertex %llu of the tile at %llu: %u, not %u\n",
                       (int)sizeof(Id) * 8, nx, ny, nz, v, base, got, want);
        }
    }
}

void both(u64 nx, u64 ny, u64 nz)
{
    const unsigned __int128 n = (unsigned __int128)nx * ny * nz;
    if (n == 0) return;
    if (n < 0xFFFFFFFFull) {
        grid<4, 4, 4, uint32_t>(nx, ny, nz);
        grid<4, 4, 3, uint32_t>(nx, ny, nz);
        grid<5, 4, 4, uint32_t>(nx, ny, nz);
    }
    if (n < (unsigned __int128)1 << 34) grid<4, 4, 4, uint64_t>(nx, ny, nz);
}

int main()
{
    // the last tiles of axes up to 2^32 - 1 long
    const u64 axis[] = {1, 15, 16, 17, 4294967279u, 4294967280u, 4294967281u, 4294967295u};
    for (u64 n : axis)
        for (u64 o = n > 64 ? (n - 64) / 16 * 16 : 0; o < n; o += 16) {
            const u64 want = n - o < 16 ? n - o : 16;
            if (tile_side((uint32_t)o, 16, (uint32_t)n) != want && bad++ < 5)
                printf("axis of %llu: not %llu vertices in the tile at %llu\n", n, want, o);
        }
    // the scattered order of the tiles takes each tile once
    for (u64 i = 0; i < 20000; i++) {
        const u64 n = i < 10000 ? i + 1 : rnd() % 0x7FFFFFFFull + 1, k = scatter_stride((uint32_t)n);
        u64 a = n, b = k;
        while (b) { const u64 t = a % b; a = b, b = t; }
        if ((a != 1 || k == 0) && bad++ < 5) printf("%llu tiles: a stride of %llu\n", n, k);
    }
    const u64 side[] = {1, 2, 3, 15, 16, 17, 33, 509, 1024, 65535, 65536, (1u << 28) - 1, (1u << 28) + 1,
                        (1u << 29) + 16, 1431655764, 2147483648u, 3000000019u, 4294967295u};
    for (u64 a : side)
        for (u64 b : side)
            for (u64 c : side) both(a, b, c);
    for (int i = 0; i < 3000; i++) {  // random grids of up to 2^34 vertices, sides spread over their logarithms
        const u64 a = rnd() % (1ull << (1 + rnd() % 32)) + 1, b = rnd() % ((1ull << (1 + rnd() % 20))) + 1,
                  c = rnd() % ((1ull << (1 + rnd() % 12))) + 1;
        if (a <= 0xFFFFFFFFull) both(a, b, c);
    }
    printf("%llu wrong, %llu in their tile\n", bad, in_tile);
    return bad || in_tile < 100000;
}
"""


def test_local_ids(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "tile_index.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "tile_index")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
