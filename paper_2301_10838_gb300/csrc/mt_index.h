// Index arithmetic of the kernels that depends on nothing of the GPU, so that
// the tests can run it on the CPU over grids of any size.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define MT_HD __host__ __device__ __forceinline__
#else
#define MT_HD inline
#endif

namespace mt {

constexpr uint32_t kNoLocal = 0xFFFFu;  // no vertex of the tile

// Vertices of the grid, n along an axis, in a tile of T that begins at o < n.
// (o + T may wrap where n is within T of 2^32.)
MT_HD uint32_t tile_side(uint32_t o, uint32_t T, uint32_t n) { return n - o < T ? n - o : T; }

// Notes that the wide path's tile kernel leaves per 16x16x16 tile for the repair
// pass, in u32 words: the minima of every column (16 bits each), then the tile's
// highest key. A grid less than 16 wide has the columns of its own sides only, so
// that the notes of a line take 3 bytes per vertex (0.13 in a solid grid).
MT_HD uint32_t wide_note_words(uint32_t nx, uint32_t ny) { return ((nx < 16 ? nx : 16) * (ny < 16 ? ny : 16) + 1) / 2 + 1; }

// The order in which CTAs take the n tiles of a field to merge the edges between
// them: CTA i takes tile i * scatter_stride(n) mod n. Merged at the same time,
// neighbours are linked each to the next, a chain that later merges and the
// repair have to climb; a stride coprime to n, near n over the golden ratio,
// keeps the tiles that are merged together apart, which leaves chains as short
// as a random order would.
inline uint32_t scatter_stride(uint32_t n)
{
    if (n < 64) return 1;
    for (uint32_t k = (uint32_t)(0.6180339887 * n);; k++) {
        uint32_t a = n, b = k;
        while (b) {
            const uint32_t t = a % b;
            a = b, b = t;
        }
        if (a == 1) return k;
    }
}

// Whether a grid of tiles is only a few tiles thick: then neighbours in the order
// of their numbers make up whole chains, and nothing is gained from their
// sharing lines in L2.
inline bool thin_tiles(uint32_t ntx, uint32_t nty, uint32_t ntz)
{
    const uint32_t m = ntx > nty ? ntx : nty, most = m > ntz ? m : ntz;
    return (uint64_t)ntx * nty * ntz / most < 32;
}

// Local id, in a tile of (1 << LX, 1 << LY, 1 << LZ) vertices of which the
// first (wx, wy, wz) lie in the grid, of the vertex whose id is `rel` above
// that of the tile's first vertex (an Id that has wrapped for an earlier one);
// kNoLocal outside the tile. Within the tile's span the quotients by nxy and
// nx are at most 16, so a product with the reciprocal (rnxy, rnx) is off by at
// most one, which the remainder shows. With 64-bit ids the remainder by nxy
// may itself need more than 32 bits (nx above 2^28).
template <int LX, int LY, int LZ, class Id>
MT_HD uint32_t tile_local(Id rel, Id nxy, uint32_t nx, float rnxy, float rnx, uint32_t wx, uint32_t wy, uint32_t wz)
{
    constexpr uint32_t TX = 1u << LX, TY = 1u << LY, TZ = 1u << LZ;
    if ((uint64_t)rel >= (uint64_t)TZ * nxy) return kNoLocal;
    uint32_t dz = (uint32_t)((float)rel * rnxy);
    if ((Id)dz * nxy > rel) dz--;
    Id r = rel - (Id)dz * nxy;
    if (r >= nxy) dz++, r -= nxy;
    if ((uint64_t)r >= (uint64_t)TY * nx) return kNoLocal;
    uint32_t dy = (uint32_t)((float)r * rnx);
    if ((Id)dy * nx > r) dy--;
    Id dx = r - (Id)dy * nx;
    if (dx >= nx) dy++, dx -= nx;
    return dx < wx && dy < wy && dz < wz ? (uint32_t)dx + TX * (dy + TY * dz) : kNoLocal;
}

}  // namespace mt
