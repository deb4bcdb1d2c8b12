// Kernels that build the triplet merge tree (Algorithm 1 of the paper):
//   k_tile     per tile, in shared memory: initialisation seeded with a lower
//              neighbour, descent pointer jumping, Merge of the in-tile
//              edges, Repair of the tile's minima
//   k_cross    Merge (Algorithm 3) of the edges between tiles, 64-bit CAS
//   k_repair   Repair (Algorithm 5) via Representative (Algorithm 4); in
//              mt_build_components also the components of G_t
#include <cuda_runtime.h>

#include <type_traits>

#include "mt_device.cuh"
#include "mt_fields.cuh"
#include "mt_index.h"
#include "mt_internal.h"

namespace mt {

// ---------------------------------------------------------------- k_tile
//
// The initialisation loop and most of the edge loop of Algorithm 1, one
// brick ("tile") of the grid per CTA, entirely in shared memory.
//
// Algorithm 1 may merge the edges in any order. This kernel merges first the
// edges inside each tile: it loads the tile's values into shared memory
// (coalesced float4 rows), builds the triplet tree of the tile's own subgraph
// with the lock-free Merge (64-bit CAS on link words in shared memory), repairs
// its minima and writes these out as global triplets. Local ids
// l = lx + TX * (ly + TY * lz) order the tile's vertices exactly as their
// global linear indices do, so ties break identically. Values are kept as
// 32-bit keys whose unsigned order is the float order (-0 and +0 share one
// key), so a vertex comparison is an integer comparison of (key, id).
//
// Which edges. Let S be the upper end of an edge (S, a). If another lower
// neighbour c of S lies on a common grid square with a, and the square's
// fourth corner q is below S too, then a - q - c joins a and c below S: once
// one of the edges (S, a), (S, c) is merged the other adds nothing, at any
// level. (The edges of that path have levels below S; by induction over the
// levels they may have been left out for the same reason, and their ends are
// still joined at their own levels.) So among the lower neighbours of S only
// the components of "joined through a square below S" matter. One lower
// neighbour seeds S (Algorithm 1 starts at T[S] = (S, lower neighbour): a
// valid triplet of the graph of descent edges), every other component gives
// one edge. On a lognormal field 0.23 edges per vertex are left of the 1.55
// whose ends descend to different minima, for about 0.11 minima; all of them
// are merged straight away, in no order, by short climbs (4 links each).
//
// The lower-than relations are computed bit-sliced. A thread owns a column of
// TZ vertices along z and slides a window of keys up it: nine comparisons
// per vertex (with the neighbours at +x, +y, +z and six of the twelve square
// corners) give nine words of one bit per vertex. The other nine relations
// are the complements of the neighbour columns' bits, exchanged through
// shared memory, and the components are then flooded for all vertices of the
// column at once, one LOP3 per word and square.
//
// What leaves the kernel. After the merges the branch minima are repaired
// (Algorithm 5) and written as global triplets: a valid normalised triplet
// tree of the minima in the full grid minus the edges between tiles, which
// k_cross merges next. An inner vertex takes no part in those merges, so its
// word only says which minimum of the tile it descends to (kInner, local id);
// k_repair gives it its triplet, once, when the tree is whole. (Repaired here
// as well it climbed 1.6 links on average, for 3.8 ms at 1024^3.)
//
// What it costs. The kernel is bound by instruction issue (73 % of the issue
// slots, HBM 15 % busy). On the 1024^3 lognormal field it takes 11.7 ms: loads
// 1.2, relations 0.7, components 1.0, edge list 0.7, descent 1.1, merges 3.5,
// minima 0.6, faces and the words of the inner vertices 2.9. The earlier
// design, which kept every edge whose ends descend to different minima and
// settled most of them by comparing cached climbs in 8 rounds over level
// buckets, took 31.5 ms (29 warp instructions per vertex).
// The climbs and merges are loops whose lanes stay together by votes: with
// ordinary divergent loops the same algorithm took 24.0 ms against 14.5, since
// a warp whose lanes left a loop one by one ran what follows it once per
// group. The merges by 4, 3 or 2 of the 8 warps took 12.0, 11.9 and 14.1 ms,
// merges from each column's own words without the list 13.6, the faces'
// values loaded before the merges or before the minima's repair 12.5 and 12.7.
constexpr int log2i(int x) { return x <= 1 ? 0 : 1 + log2i(x / 2); }

template <int LX, int LY, int LZ>
struct Tile {
    static constexpr int TX = 1 << LX, TY = 1 << LY, TZ = 1 << LZ;
    static constexpr int TV = TX * TY * TZ;
    static constexpr int NT = TX * TY;  // a thread per column
    static_assert(TZ <= 16, "a column's bits fit half a word");
    static_assert(LX + LY + LZ + 3 <= 16, "an edge entry packs a local id and a direction into 16 bits");
    static_assert(TX % 4 == 0, "rows are loaded as float4");
    static constexpr int kList = NT * 8 / kTileListShrink;  // edges listed (the others are merged in place)
    // shared memory: a link word (8 B) per x-adjacent pair of vertices, of
    // which at most one is a minimum; keys (4 B) and seeds (2 B) per vertex;
    // then 16 B per thread that hold in turn the exchanged words, the edge
    // list and the list of face edges
    static constexpr size_t kSmem = (size_t)TV * (4 + 4 + 2) + (size_t)NT * 16;
    static constexpr int kCTAs = (int)(227 * 1024 / (kSmem + 1024)) < 1536 / NT ? (int)(227 * 1024 / (kSmem + 1024)) : 1536 / NT;
    // face record of a tile (u32 words): per group of 32 edges of the faces
    // +x, +y, +z the number of kept ones (a byte each), then the tops in this
    // tile of the kept edges' ends on the + faces and on the - faces, then the
    // levels S of the + faces' edges; 16 entries per group
    static constexpr int G = (TY * TZ + TX * TZ + TX * TY) / 32;
    static constexpr int kFaceHead = (G + 15) / 16 * 4, kFaceSide = 16 * G;
    static constexpr int kFaceWords = kFaceHead + 3 * kFaceSide;
    // after the face record, for the repair pass: the minima of every column
    // (16 bits each), the tile's highest key (the wide path has only these, see
    // wide_note_words)
    static constexpr int kNoteWords = NT / 2 + 4, kTileWords = kFaceWords + kNoteWords;
    static_assert(TY * TZ <= NT && TX * TZ <= NT, "one edge of a face per thread");
    static constexpr int FX = TY * TZ, FY = TX * TZ, FZ = TX * TY, FH = FX + FY + FZ;  // edges of the + faces
    static_assert(2 * FH * 8 <= TV * 4, "the faces' levels fit the key array");
    static_assert(2 * kFaceSide * 4 <= NT * 16, "the face edge list fits its buffer");
};

// Order-preserving 32-bit key of a float (+0 and -0 map to the same key).
__device__ __forceinline__ uint32_t order_key(float x)
{
    const uint32_t b = x == 0.0f ? 0u : __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
// (ka, a) before (kb, b)
__device__ __forceinline__ bool kbefore(uint32_t ka, uint32_t a, uint32_t kb, uint32_t b)
{
    return ka < kb || (ka == kb && a < b);
}

// The key of no vertex: above every finite key. Vertices outside the grid
// have it, and so has the link word of a root.
constexpr uint32_t kNoKey = 0xFFFFFFFFu;

// A minimum's link in the tile's tree as one 64-bit word: the saddle's key,
// its local id (16 bits), the target's local id (16 bits). Links compare as
// integers by level: a walk to level (kS, S) follows word w iff
// w <= level_word(kS, S), and a root's word (kNoKey) stops every walk.
__device__ __forceinline__ uint64_t level_word(uint32_t kS, uint32_t S)
{
    return (uint64_t)kS << 32 | S << 16 | 0xFFFFu;
}
__device__ __forceinline__ uint32_t link_s(uint64_t w) { return (uint32_t)w >> 16; }
__device__ __forceinline__ uint32_t link_v(uint64_t w) { return (uint32_t)w & 0xFFFFu; }

// Merge (Algorithm 3) on the tile's tree, lock-free with 64-bit CAS on the
// link words L (of vertex x at L[x / 2]). One try: u and v have climbed to
// their deepest vertices below the level `lim` and differ; the later one (its
// word wv) is linked under the earlier, and the link it held is re-inserted
// by going on from there (a displaced root carries none; after a failed CAS
// both climb again). Returns true when the edge is done.
__device__ __forceinline__ bool sm_link(uint64_t *L, const uint32_t *K, uint64_t &lim, uint32_t &u, uint32_t &v,
                                        uint64_t wu, uint64_t wv)
{
    const bool sw = kbefore(K[v], v, K[u], u);
    const uint32_t lo = sw ? v : u;
    v = sw ? u : v, u = lo;
    wv = sw ? wu : wv;
    const uint64_t want = (lim & ~(uint64_t)0xFFFFu) | u;
    if (atomicCAS(reinterpret_cast<unsigned long long *>(L + (v >> 1)), (unsigned long long)wv,
                  (unsigned long long)want) == wv) {
        if ((uint32_t)(wv >> 32) == kNoKey) return true;
        lim = wv | 0xFFFFu;
        v = link_v(wv);
    }
    return u == v;
}

// The minimum that vertex x descends to along the seeds D.
template <int TV>
__device__ __forceinline__ uint32_t sm_descend(const uint16_t *D, uint32_t x)
{
    const volatile uint16_t *vD = D;
    for (uint32_t h = 0; h < (uint32_t)TV; h++) {
        const uint32_t y = vD[x];
        if (y == x) break;
        x = y;
    }
    return x;
}

// A whole merge of the edge (S, w), out of line for the rare edges that find
// the list full.
template <int TV>
__device__ __noinline__ bool sm_merge_rare(uint64_t *L, const uint32_t *K, const uint16_t *D, uint32_t S, uint32_t w)
{
    uint32_t u = sm_descend<TV>(D, S), v = sm_descend<TV>(D, w);
    const volatile uint64_t *vL = L;
    uint64_t lim = level_word(K[S], S);
    for (uint32_t it = 0; it < kMergeStepLimit; it++) {
        const uint64_t wu = vL[u >> 1], wv = vL[v >> 1];
        const bool mu = wu <= lim, mv = wv <= lim;
        if (mu) u = link_v(wu);
        if (mv) v = link_v(wv);
        if (u == v || (!mu && !mv && sm_link(L, K, lim, u, v, wu, wv))) return true;
    }
    return false;
}

// WIDE: the triplets leave the tile as 128-bit words of two 64-bit ids
// (W[2u] = s, W[2u + 1] = v) for grids of 2^32 vertices and more; the work
// inside the tile, on 16-bit local ids, is the same, and no face record is
// written (the wide path merges the edges between tiles from their ends).
template <int LX, int LY, int LZ, bool WIDE = false>
__device__ __forceinline__ void tile_body(const FieldDesc &fd, uint32_t tile, uint32_t *status)
{
    using TR = Tri<WIDE>;
    using Id = typename TR::Id;
    const float *__restrict__ f = fd.f;
    const float sg = fd.sg;
    uint64_t *__restrict__ W = fd.W;
    const uint32_t nx = fd.nx, ny = fd.ny, nz = fd.nz, ntx = fd.ntx, nty = fd.nty;
    using TS = Tile<LX, LY, LZ>;
    constexpr uint32_t TX = TS::TX, TY = TS::TY, TZ = TS::TZ, TV = TS::TV, NT = TS::NT, LV = LX + LY + LZ;
    extern __shared__ __align__(16) uint64_t tile_smem[];
    uint64_t *L = tile_smem;                                  // link words of the minima
    uint32_t *K = reinterpret_cast<uint32_t *>(L + TV / 2);   // order keys
    uint16_t *D = reinterpret_cast<uint16_t *>(K + TV);       // seeds, then descent minima
    uint32_t *X = reinterpret_cast<uint32_t *>(D + TV);       // 16 B per thread, see Tile
    uint16_t *list = reinterpret_cast<uint16_t *>(X);
    volatile uint64_t *vL = L;
    volatile uint16_t *vD = D;
    __shared__ uint32_t s_nlist, s_nface, s_kmax;

    const uint32_t lane = threadIdx.x & 31;
    const uint32_t tx = tile % ntx, ty = (tile / ntx) % nty, tz = tile / (ntx * nty);
    const uint32_t x0 = tx * TX, y0 = ty * TY, z0 = tz * TZ;
    const uint32_t wx = min(TX, nx - x0), wy = min(TY, ny - y0), wz = min(TZ, nz - z0);
    const Id nxy = (Id)nx * ny;  // n < 2^32 unless WIDE, so every id fits an Id
    const Id base = (Id)z0 * nxy + (Id)y0 * nx + x0;
    auto lxo = [](uint32_t l) { return l & (TX - 1); };
    auto lyo = [](uint32_t l) { return (l >> LX) & (TY - 1); };
    auto lzo = [](uint32_t l) { return l >> (LX + LY); };
    auto gid = [&](uint32_t l) -> Id { return base + (Id)lzo(l) * nxy + (Id)lyo(l) * nx + lxo(l); };

    auto put = [&](Id u, Id sd, Id tg) {
        if constexpr (WIDE) reinterpret_cast<ulonglong2 *>(W)[u] = make_ulonglong2(sd, tg);
        else W[u] = tri_pack(sd, tg);
    };

    // 1. load the tile's values (rows of TX floats) as order keys; vertices
    //    outside the grid get kNoKey
    bool bad = false;
    if (nx % 4 == 0 && (uintptr_t)f % 16 == 0) {
#pragma unroll
        for (uint32_t i = 0; i < TV / 4 / NT; i++) {
            const uint32_t l = 4 * (i * NT + threadIdx.x);
            uint4 k = make_uint4(kNoKey, kNoKey, kNoKey, kNoKey);
            if (lxo(l) < wx && lyo(l) < wy && lzo(l) < wz) {
                float4 v = __ldg(reinterpret_cast<const float4 *>(f + gid(l)));
                v.x *= sg, v.y *= sg, v.z *= sg, v.w *= sg;
                bad |= !isfinite(v.x) | !isfinite(v.y) | !isfinite(v.z) | !isfinite(v.w);
                k = make_uint4(order_key(v.x), order_key(v.y), order_key(v.z), order_key(v.w));
            }
            *reinterpret_cast<uint4 *>(K + l) = k;
        }
    } else {
#pragma unroll 8
        for (uint32_t i = 0; i < TV / NT; i++) {
            const uint32_t l = i * NT + threadIdx.x;
            uint32_t k = kNoKey;
            if (lxo(l) < wx && lyo(l) < wy && lzo(l) < wz) {
                const float v = sg * __ldg(f + gid(l));
                bad |= !isfinite(v);
                k = order_key(v);
            }
            K[l] = k;
        }
    }
    if (threadIdx.x == 0) s_nlist = 0, s_nface = 0, s_kmax = 0;
    if (bad) raise_status(status, ST_NONFINITE);
    __syncthreads();

    // 2. lower-than words of the thread's column: bit z of p<d> says that the
    //    neighbour at d is before vertex (x, y, z). In p.. the neighbour has
    //    the later id, so it is before only with a strictly lower key; in
    //    q.. (one plane down) it has the earlier id. Reads past the tile's
    //    faces give some other word of shared memory; those bits are masked
    //    below.
    const uint32_t col = threadIdx.x, cx = lxo(col), cy = lyo(col);
    uint32_t px = 0, py = 0, pz = 0, pxy = 0, pmxy = 0, pxz = 0, pyz = 0, qxz = 0, qyz = 0, kmax = 0;
    {
        uint32_t kc = K[col], kx = K[col + 1], ky = K[col + TX], kxd = 0, kyd = 0;
#pragma unroll
        for (uint32_t z = 0; z < TZ; z++) {
            const uint32_t l = col + z * NT;
            const uint32_t kcu = z + 1 < TZ ? K[l + NT] : kNoKey, kxu = z + 1 < TZ ? K[l + NT + 1] : kNoKey,
                           kyu = z + 1 < TZ ? K[l + NT + TX] : kNoKey;
            kmax = max(kmax, kc + 1);  // kNoKey, outside the grid, gives 0
            px |= (uint32_t)(kx < kc) << z;
            py |= (uint32_t)(ky < kc) << z;
            pz |= (uint32_t)(kcu < kc) << z;
            pxy |= (uint32_t)(K[l + TX + 1] < kc) << z;
            pmxy |= (uint32_t)(K[l + TX - 1] < kc) << z;
            pxz |= (uint32_t)(kxu < kc) << z;
            pyz |= (uint32_t)(kyu < kc) << z;
            if (z > 0) {
                qxz |= (uint32_t)(kxd <= kc) << z;
                qyz |= (uint32_t)(kyd <= kc) << z;
            }
            kxd = kx, kyd = ky;
            kc = kcu, kx = kxu, ky = kyu;
        }
    }
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) atomicMax(&s_kmax, kmax);
    X[col] = px | pxz << 16;
    X[NT + col] = qxz | pxy << 16;
    X[2 * NT + col] = py | pyz << 16;
    X[3 * NT + col] = qyz | pmxy << 16;
    __syncthreads();

    // 3. the lower neighbours of every vertex, their components, the seed
    //    and the edges left to merge
    const bool inx = cx < wx && cy < wy;
    const uint32_t zm = inx ? (1u << wz) - 1u : 0u;
    uint32_t minima;       // bit z: vertex z of the column is a minimum of the tile
    uint32_t ex, ey, ez;   // edges to merge: bits z (towards -) and 16 + z (towards +)
    {
        const uint32_t cm = (col - 1) & (NT - 1);
        const uint32_t a = X[cm], b = X[NT + cm];                          // column (x - 1, y)
        const uint32_t c = X[2 * NT + ((col - TX) & (NT - 1))], d = X[3 * NT + ((col - TX) & (NT - 1))];  // (x, y - 1)
        const uint32_t e = X[NT + ((col - TX - 1) & (NT - 1))];            // (x - 1, y - 1)
        const uint32_t g = X[3 * NT + ((col - TX + 1) & (NT - 1))];        // (x + 1, y - 1)
        // lower neighbours (a relation to a neighbour with an earlier id is
        // the complement of that neighbour's relation to this vertex)
        const uint32_t lx0 = cx > 0 ? ~a & zm : 0u, lx1 = cx + 1 < wx ? px & zm : 0u;
        const uint32_t ly0 = cy > 0 ? ~c & zm : 0u, ly1 = cy + 1 < wy ? py & zm : 0u;
        const uint32_t lz0 = (~pz << 1) & zm, lz1 = pz & zm;
        minima = zm & ~(lx0 | lx1 | ly0 | ly1 | lz0 | lz1);
        // squares: both neighbours and the corner between them are lower
        const uint32_t x0y0 = lx0 & ly0 & ~(e >> 16), x1y0 = lx1 & ly0 & ~(g >> 16);
        const uint32_t x0y1 = lx0 & ly1 & pmxy, x1y1 = lx1 & ly1 & pxy;
        const uint32_t x0z0 = lx0 & lz0 & (~(a >> 16) << 1), x1z0 = lx1 & lz0 & qxz;
        const uint32_t x0z1 = lx0 & lz1 & (~(b & 0xFFFFu) >> 1), x1z1 = lx1 & lz1 & pxz;
        const uint32_t y0z0 = ly0 & lz0 & (~(c >> 16) << 1), y1z0 = ly1 & lz0 & qyz;
        const uint32_t y0z1 = ly0 & lz1 & (~(d & 0xFFFFu) >> 1), y1z1 = ly1 & lz1 & pyz;
        // the seed: the first lower neighbour
        const uint32_t sx0 = lx0, sx1 = lx1 & ~lx0, m2 = lx0 | lx1;
        const uint32_t sy0 = ly0 & ~m2, m3 = m2 | ly0, sy1 = ly1 & ~m3, m4 = m3 | ly1;
        const uint32_t sz0 = lz0 & ~m4, sz1 = lz1 & ~(m4 | lz0);
        // flood its component (three passes reach all but a few; a
        // component cut in two only costs an edge that adds nothing)
        uint32_t rx0 = sx0, rx1 = sx1, ry0 = sy0, ry1 = sy1, rz0 = sz0, rz1 = sz1;
#pragma unroll
        for (int it = 0; it < 3; it++) {
            ry0 |= (rx0 & x0y0) | (rx1 & x1y0) | (rz0 & y0z0) | (rz1 & y0z1);
            ry1 |= (rx0 & x0y1) | (rx1 & x1y1) | (rz0 & y1z0) | (rz1 & y1z1);
            rz0 |= (rx0 & x0z0) | (rx1 & x1z0) | (ry0 & y0z0) | (ry1 & y1z0);
            rz1 |= (rx0 & x0z1) | (rx1 & x1z1) | (ry0 & y0z1) | (ry1 & y1z1);
            rx0 |= (ry0 & x0y0) | (ry1 & x0y1) | (rz0 & x0z0) | (rz1 & x0z1);
            rx1 |= (ry0 & x1y0) | (ry1 & x1y1) | (rz0 & x1z0) | (rz1 & x1z1);
        }
        // of the other components, the first neighbour (a neighbour joined
        // to one earlier in the order x0 x1 y0 y1 z0 z1 is left out)
        ex = (lx0 & ~rx0) | (lx1 & ~rx1) << 16;
        ey = (ly0 & ~(ry0 | x0y0 | x1y0)) | (ly1 & ~(ry1 | x0y1 | x1y1)) << 16;
        ez = (lz0 & ~(rz0 | x0z0 | x1z0 | y0z0 | y1z0)) | (lz1 & ~(rz1 | x0z1 | x1z1 | y0z1 | y1z1)) << 16;
#pragma unroll
        for (uint32_t z = 0; z < TZ; z++) {
            const uint32_t l = col + z * NT;
            uint32_t v = l, bit = 1u << z;
            if (sx0 & bit) v = l - 1;
            if (sx1 & bit) v = l + 1;
            if (sy0 & bit) v = l - TX;
            if (sy1 & bit) v = l + TX;
            if (sz0 & bit) v = l - NT;
            if (sz1 & bit) v = l + NT;
            D[l] = (uint16_t)v;
        }
        for (uint32_t m = minima; m; m &= m - 1) {
            const uint32_t l = col + (__ffs(m) - 1) * NT;
            L[l >> 1] = (uint64_t)kNoKey << 32 | 0xFFFF0000u | l;
        }
    }
    __syncthreads();

    // 4. list the edges; pointer jumping along the seeds (concurrent jumps
    //    only shorten chains, so racing readers stay correct)
    bool ok = true;
    {
        const uint32_t cnt = __popc(ex) + __popc(ey) + __popc(ez);
        uint32_t incl = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        uint32_t pos = 0;
        if (lane == 31) pos = atomicAdd(&s_nlist, incl);
        pos = __shfl_sync(0xffffffffu, pos, 31) + incl - cnt;
#pragma unroll
        for (uint32_t axis = 0; axis < 3; axis++) {
            for (uint32_t m = axis == 0 ? ex : axis == 1 ? ey : ez; m; m &= m - 1) {
                const uint32_t i = __ffs(m) - 1, up = i >> 4, S = col + (i & 15) * NT;
                if (pos < (uint32_t)TS::kList) {
                    list[pos] = (uint16_t)(S | (2 * axis + up) << LV);
                } else {  // list full: merge in place
                    const uint32_t step = axis == 0 ? 1u : axis == 1 ? TX : NT;
                    ok &= sm_merge_rare<TV>(L, K, D, S, up ? S + step : S - step);
                }
                pos++;
            }
        }
    }
#pragma unroll 4
    for (uint32_t z = 0; z < TZ; z++) {
        const uint32_t l = col + z * NT;
        uint32_t x = vD[l];
        x = vD[x];
        x = vD[x];
        uint32_t y = vD[x];
        for (uint32_t h = 0; h < TV && __any_sync(0xffffffffu, x != y); h++) x = y, y = vD[x];
        vD[l] = (uint16_t)x;
    }
    __syncthreads();

    // 5. merge the listed edges, from the minima their ends descend to. A
    //    warp takes its share of the list in order; a lane that is done with
    //    an edge takes the share's next one, so that the lanes do not wait for
    //    the longest re-insertion of each round. The loop is uniform over the
    //    warp (votes, no divergent branches): two links of both climbs, then
    //    one try to link where both have stopped.
    {
        const uint32_t nlist = min(s_nlist, (uint32_t)TS::kList);
        const uint32_t share = (nlist + NT / 32 - 1) / (NT / 32);
        uint32_t next = (threadIdx.x >> 5) * share;
        const uint32_t end = min(next + share, nlist), below = (1u << lane) - 1u;
        uint32_t u = 0, v = 0, it = 0;
        uint64_t lim = 0;
        bool have = false;
        for (;;) {
            const uint32_t need = __ballot_sync(0xffffffffu, !have);
            if (need) {
                const uint32_t i = next + __popc(need & below);
                if (!have && i < end) {
                    const uint32_t e = list[i];
                    const uint32_t S = e & (TV - 1), d = e >> LV;
                    const uint32_t step = d < 2 ? 1u : d < 4 ? (uint32_t)TX : NT;
                    u = vD[S];
                    v = vD[(d & 1) ? S + step : S - step];
                    lim = level_word(K[S], S);
                    have = u != v;
                }
                __syncwarp();
                next += __popc(need);
                if (next >= end && !__any_sync(0xffffffffu, have)) break;
            }
            uint64_t wu = 0, wv = 0;
            bool mu = false, mv = false;
#pragma unroll
            for (int hop = 0; hop < 2; hop++) {
                if (have) {
                    wu = vL[u >> 1], wv = vL[v >> 1];
                    mu = wu <= lim, mv = wv <= lim;
                    u = mu ? link_v(wu) : u;
                    v = mv ? link_v(wv) : v;
                }
                __syncwarp();
            }
            have = have && u != v;
            if (have && !mu && !mv) have = !sm_link(L, K, lim, u, v, wu, wv);
            __syncwarp();
            if (++it > kMergeStepLimit) {
                ok = false;
                break;
            }
        }
    }
    __syncthreads();

    // 6. repair the branch minima (Algorithm 5); concurrent repairs move
    //    targets along their own chains below their own saddles, which
    //    leaves the end of every walk unchanged
    for (uint32_t m = minima; m; m &= m - 1) {
        const uint32_t l = col + (__ffs(m) - 1) * NT;
        const uint64_t w = vL[l >> 1];
        uint32_t s = l, x = l;  // a root's triplet
        if ((uint32_t)(w >> 32) != kNoKey) {
            const uint64_t lim = w | 0xFFFFu;
            s = link_s(w), x = link_v(w);
            for (uint32_t h = 0; h < TV; h++) {
                const uint64_t wx_ = vL[x >> 1];
                if (wx_ > lim) break;
                x = link_v(wx_);
            }
            if (x != link_v(w)) vL[l >> 1] = (w & ~(uint64_t)0xFFFFu) | x;
        }
        put(gid(l), gid(s), gid(x));
    }

    // 7. for k_repair: the words of the inner vertices say which tile minimum
    //    they descend to (they get their triplets once all merges are done);
    //    the tile's minima and highest key
    uint32_t *rec = fd.faces;
    if constexpr (WIDE) {
        const uint32_t mx = min(nx, TX), words = wide_note_words(nx, ny);
        rec += (size_t)tile * words;
        if (cx < mx && cy < min(ny, TY)) reinterpret_cast<uint16_t *>(rec)[cx + cy * mx] = (uint16_t)minima;
        if (threadIdx.x == 0) rec[words - 1] = s_kmax - 1;
    } else {
        rec += (size_t)tile * TS::kTileWords;
        reinterpret_cast<uint16_t *>(rec + TS::kFaceWords)[col] = (uint16_t)minima;
        if (threadIdx.x == 0) rec[TS::kFaceWords + NT / 2] = s_kmax - 1;
    }
    if (inx) {
        const Id u0 = gid(col);
#pragma unroll
        for (uint32_t z = 0; z < TZ; z++)
            if (z < wz && !((minima >> z) & 1u)) put(u0 + z * nxy, TR::kInner, (Id)vD[col + z * NT]);
    }

    // 8. for k_cross: the edges into the neighbouring tiles that can matter,
    //    with the tile-local top of their end in this tile, i.e. the deepest
    //    vertex of its tile component below the edge's level S. By the same
    //    argument as above an edge (a, b) between tiles adds nothing if a
    //    parallel edge (c, q) of the face beside it has a lower level: both
    //    its ends are before S, so with a - c and q - b inside the tiles they
    //    join a and b below S. What is left are the local minima of the
    //    level over each face (about 44 of 256 edges on a lognormal field),
    //    no two of them neighbours, so at most 16 of a group of 32 (one or
    //    two rows of a face). Both tiles of a face find the same edges in the
    //    same order. The kept edges of all faces are listed before their
    //    climbs, so that the climbs run with all lanes busy.
    if constexpr (!WIDE) {
        uint64_t *lev = reinterpret_cast<uint64_t *>(K);  // (key, id) of the levels, face after face
        const uint32_t e = threadIdx.x;
        auto face_size = [](uint32_t fc) -> uint32_t { return fc % 3 == 0 ? TS::FX : fc % 3 == 1 ? TS::FY : TS::FZ; };
        auto face_off = [](uint32_t fc) -> uint32_t {
            return (fc / 3) * TS::FH + (fc % 3 == 0 ? 0 : fc % 3 == 1 ? TS::FX : TS::FX + TS::FY);
        };
        uint64_t mine[6];
#pragma unroll
        for (uint32_t fc = 0; fc < 6; fc++) {  // faces +x, +y, +z, -x, -y, -z
            const uint32_t dir = fc % 3, side = fc / 3, lg1 = dir == 0 ? LY : LX;
            const uint32_t c1 = e & ((1u << lg1) - 1), c2 = e >> lg1;  // in-face coordinates
            const bool in = e < face_size(fc) && c1 < (dir == 0 ? wy : wx) &&
                            c2 < (dir == 2 ? wy : wz);
            const bool has = side == 0 ? (dir == 0 ? x0 + TX < nx : dir == 1 ? y0 + TY < ny : z0 + TZ < nz)
                                       : (dir == 0 ? x0 : dir == 1 ? y0 : z0) > 0;
            mine[fc] = ~0ull;
            if (has && in) {
                const uint32_t last = dir == 0 ? TX - 1 : dir == 1 ? (TY - 1) * TX : (TZ - 1) * NT;
                const uint32_t l = (dir == 0 ? c1 * TX + c2 * NT : dir == 1 ? c1 + c2 * NT : e) + (side ? 0u : last);
                const uint32_t step = dir == 0 ? 1u : dir == 1 ? nx : (uint32_t)nxy;
                const uint32_t ga = (uint32_t)gid(l), gb = side ? ga - step : ga + step;
                const uint64_t ka = (uint64_t)K[l] << 32 | ga,
                               kb = (uint64_t)order_key(sg * __ldg(f + gb)) << 32 | gb;
                mine[fc] = ka > kb ? ka : kb;
            }
        }
        __syncthreads();
#pragma unroll
        for (uint32_t fc = 0; fc < 6; fc++)
            if (e < face_size(fc)) lev[face_off(fc) + e] = mine[fc];
        __syncthreads();
        uint32_t bal[6], tot = 0;
#pragma unroll
        for (uint32_t fc = 0; fc < 6; fc++) {
            // edges outside the face have level ~0: they are not kept (no
            // level is) and put no other out
            const uint32_t dir = fc % 3, lg1 = dir == 0 ? LY : LX;
            const uint32_t m1 = 1u << lg1, m2 = dir == 2 ? TY : TZ, c1 = e & (m1 - 1), c2 = e >> lg1;
            const uint64_t *p = lev + face_off(fc) + e;
            const uint64_t v = mine[fc];
            const bool keep = v != ~0ull && !((c1 > 0 && p[-1] < v) || (c1 + 1 < m1 && p[1] < v) ||
                                              (c2 > 0 && *(p - m1) < v) || (c2 + 1 < m2 && p[m1] < v));
            bal[fc] = __ballot_sync(0xffffffffu, keep);
            tot += __popc(bal[fc]);
        }
        uint32_t pos = 0;
        if (lane == 0) pos = atomicAdd(&s_nface, tot);
        pos = __shfl_sync(0xffffffffu, pos, 0);
        const uint32_t grp = threadIdx.x >> 5, below = (1u << lane) - 1u;
#pragma unroll
        for (uint32_t fc = 0; fc < 6; fc++) {
            const uint32_t side = fc / 3, goff = face_off(fc % 3) / 32;
            if (grp < face_size(fc) / 32) {
                if (side == 0 && lane == 0) reinterpret_cast<uint8_t *>(rec)[goff + grp] = (uint8_t)__popc(bal[fc]);
                if ((bal[fc] >> lane) & 1u) {
                    const uint32_t r = __popc(bal[fc] & below);
                    // entry: place in the record's tops, edge number
                    X[pos + r] = (side * TS::kFaceSide + 16 * (goff + grp) + r) << 16 | (face_off(fc) + e);
                }
            }
            pos += __popc(bal[fc]);
        }
        __syncthreads();
        const uint32_t nface = s_nface;
        for (uint32_t i = threadIdx.x; i < nface; i += NT) {
            const uint32_t en = X[i], out = en >> 16, fe = en & 0xFFFFu;
            const uint64_t v = lev[fe];
            const uint32_t kS = (uint32_t)(v >> 32), gS = (uint32_t)v;
            const uint32_t side = fe >= TS::FH, r = fe - side * TS::FH;
            const uint32_t dir = r < TS::FX ? 0u : r < TS::FX + TS::FY ? 1u : 2u, lg1 = dir == 0 ? LY : LX;
            const uint32_t ee = r - face_off(dir), c1 = ee & ((1u << lg1) - 1), c2 = ee >> lg1;
            const uint32_t last = side ? 0u : dir == 0 ? TX - 1 : dir == 1 ? (TY - 1) * TX : (TZ - 1) * NT;
            uint32_t x = D[(dir == 0 ? c1 * TX + c2 * NT : dir == 1 ? c1 + c2 * NT : ee) + last];
            for (uint32_t h = 0; h < TV; h++) {
                const uint64_t w = vL[x >> 1];
                const uint32_t ks = (uint32_t)(w >> 32);
                if (ks > kS || (ks == kS && (uint32_t)gid(link_s(w)) > gS)) break;  // link above the level
                x = link_v(w);
            }
            rec[TS::kFaceHead + out] = (uint32_t)gid(x);
            if (!side) rec[TS::kFaceHead + 2 * TS::kFaceSide + out] = gS;
        }
    }
    if (!ok) raise_status(status, ST_TIMEOUT);
}

// One CTA per tile (queue == null), or a persistent grid that takes tiles
// from a device-side counter until none is left (the batched build).
template <int LX, int LY, int LZ, class Loc, bool WIDE = false>
__global__ void __launch_bounds__(Tile<LX, LY, LZ>::NT, Tile<LX, LY, LZ>::kCTAs)
    k_tile(Loc loc, uint32_t ntiles, uint32_t *queue, uint32_t *status)
{
    if (queue == nullptr) {
        uint32_t local;
        const FieldDesc fd = loc.tile(blockIdx.x, local);
        tile_body<LX, LY, LZ, WIDE>(fd, local, status);
        return;
    }
    __shared__ uint32_t s_next;
    for (;;) {
        if (threadIdx.x == 0) s_next = atomicAdd(queue, 1u);
        __syncthreads();
        const uint32_t t = s_next;
        __syncthreads();
        if (t >= ntiles) break;
        uint32_t local;
        const FieldDesc fd = loc.tile(t, local);
        tile_body<LX, LY, LZ, WIDE>(fd, local, status);
        __syncthreads();
    }
}

// ---------------------------------------------------------------- k_cross
//
// The rest of the edge loop of Algorithm 1: the edges between neighbouring
// tiles, merged with 64-bit CAS on the global triplets (Algorithms 2, 3).
// CTA t takes the edges from tile t to its +x, +y, +z neighbour tiles. k_tile
// left the edges that can matter (the local minima of the level over each
// face), in the same order in the records of both tiles: the level S, and for
// each end its tile-local top at S (the deepest vertex of its tile component
// below S), where the merge's climbs start. Edges with the same pair of tops
// join the same two tile components, so only the one with the earliest level
// of each pair is merged (a shared-memory hash with 64-bit atomicMin): about
// 93 of the 132 edges per tile on a lognormal field.
//
// The kernel is bound by the latency of its chains of dependent reads (38 % of
// the issue slots used, HBM 39 % busy at 512^3): 4.7 ms on the 1024^3
// lognormal field, 4.8 with the tiles in order instead of scattered (512^3 0.55
// and 0.63, 256^3 white noise 143 and 155 us, a line of 2^18 constant vertices
// 55 and 390); 6.3 ms with a merge that read a vertex's value and a
// re-inserted link's level only when it needed them, in order and without the
// hash; 5.6 ms with the new merge alone. The fields of a batch are small enough
// for L2, where the hash costs more than the merges it saves (512 uneven
// fields: 0.36 ms with it, 0.29 without), and 16 CTAs per SM run better than
// the 12 that hide most of HBM's latency (0.39 ms with 11 CTAs, 0.29 with 16;
// single field 4.8 ms with 12, 5.2 with 14).
//
// Steps before a merge goes on in the long form: 16 (8 and 32: 256^3 white noise
// 148 and 144, of 16 values 169 and 183 us); in a batch, where the call alone
// costs registers, 32 (2572 us with 16, 2570 with 32 and 64, 2560 without).
constexpr uint32_t kShortField = 16, kShortBatch = 32;  // steps before the long form

static __device__ __noinline__ bool merge_long(uint64_t *W, const Field f, uint32_t S, float fS, uint32_t u, uint32_t v)
{
    return merge_steps<true>(W, f, S, fS, u, v);
}

template <int LX, int LY, int LZ, class Loc>
__global__ void __launch_bounds__(128, std::is_same<Loc, OneField>::value ? 12 : 16)
    k_cross(Loc loc, uint32_t stride, uint32_t *status)
{
    if (block_skips(status)) return;
    using TS = Tile<LX, LY, LZ>;
    constexpr uint32_t G = TS::G, GX = TS::FX / 32, GY = TS::FY / 32, NT = 128;
    constexpr uint32_t HS = 16 * G > 512 ? 1024 : 512;  // slots for at most 16 edges per group
    static_assert(16 * G <= HS, "the hash holds every edge");
    constexpr unsigned long long EMPTY = ~0ull;
    __shared__ unsigned long long hkey[HS], hlev[HS];  // pair of tops; (key, id) of the earliest level
    __shared__ uint32_t off[65];                       // first edge of each group
    __shared__ uint16_t list[HS];
    __shared__ uint32_t s_n;
    uint32_t tile;
    constexpr bool ONE = std::is_same<Loc, OneField>::value;
    const FieldDesc fd = loc.tile(ONE ? (uint32_t)((uint64_t)blockIdx.x * stride % gridDim.x) : blockIdx.x, tile);
    const Field f{fd.f, fd.sg};
    constexpr uint32_t kWords = TS::kTileWords;
    const uint32_t *rec = fd.faces + (size_t)tile * kWords;
    if (threadIdx.x < 32) {
        static_assert(G <= 64, "two groups per lane");
        const uint8_t *cnt = reinterpret_cast<const uint8_t *>(rec);
        const uint32_t g = 2 * threadIdx.x, c0 = g < G ? cnt[g] : 0u, c1 = g + 1 < G ? cnt[g + 1] : 0u;
        uint32_t incl = c0 + c1;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (threadIdx.x >= (uint32_t)o) incl += y;
        }
        off[g] = incl - c0 - c1, off[g + 1] = incl - c1;
        if (threadIdx.x == 31) off[64] = incl, s_n = 0;
    }
    constexpr bool DEDUP = ONE;  // see above
    if (DEDUP)
        for (uint32_t i = threadIdx.x; i < HS; i += NT) hkey[i] = EMPTY, hlev[i] = EMPTY;
    __syncthreads();
    bool ok = true;
    for (uint32_t i = threadIdx.x; i < off[64]; i += NT) {
        uint32_t g = 0;  // the last group whose first edge is at or before i
#pragma unroll
        for (uint32_t w = 32; w > 0; w >>= 1)
            if (off[g + w] <= i) g += w;
        const uint32_t p = 16 * g + i - off[g];
        const uint32_t nb = g < GX ? 1u : g < GX + GY ? fd.ntx : fd.ntx * fd.nty;  // the neighbour tile
        uint32_t ta = rec[TS::kFaceHead + p], S = rec[TS::kFaceHead + 2 * TS::kFaceSide + p];
        uint32_t tb = rec[(size_t)nb * kWords + TS::kFaceHead + TS::kFaceSide + p];
        if (!DEDUP) {
            float fS = f[S];
            if (!merge_steps<false, kShortBatch>(fd.W, f, S, fS, ta, tb)) ok &= merge_long(fd.W, f, S, fS, ta, tb);
            continue;
        }
        const unsigned long long key = (unsigned long long)ta << 32 | tb,
                                 lev = (unsigned long long)order_key(f[S]) << 32 | S;
        uint32_t h = (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> 54) & (HS - 1);
        for (uint32_t q = 0; q < HS; q++) {
            const unsigned long long k0 = atomicCAS(&hkey[h], EMPTY, key);
            if (k0 == EMPTY) list[atomicAdd(&s_n, 1u)] = (uint16_t)h;
            if (k0 == EMPTY || k0 == key) {
                atomicMin(&hlev[h], lev);
                break;
            }
            h = (h + 1) & (HS - 1);
        }
    }
    if constexpr (DEDUP) {
        __syncthreads();
        // the merge in slot h: tops, level
        auto slot = [&](uint32_t h, uint32_t &S, float &fS, uint32_t &u, uint32_t &v) {
            const uint32_t kS = (uint32_t)(hlev[h] >> 32);
            fS = __uint_as_float((kS & 0x80000000u) ? kS ^ 0x80000000u : ~kS);  // the value with that order key
            S = (uint32_t)hlev[h], u = (uint32_t)(hkey[h] >> 32), v = (uint32_t)hkey[h];
        };
        // merges that are not done soon go on in the long form after the others
        // (in a loop of its own, so that its registers stay out of this one)
        uint32_t todo = 0;  // a bit for each of the thread's turns
        static_assert(HS / NT <= 32, "a bit per turn");
        for (uint32_t j = threadIdx.x, k = 0; j < s_n; j += NT, k++) {
            const uint32_t h = list[j];
            uint32_t S, u, v;
            float fS;
            slot(h, S, fS, u, v);
            if (!merge_steps<false, kShortField>(fd.W, f, S, fS, u, v)) {
                hkey[h] = (unsigned long long)u << 32 | v, hlev[h] = (unsigned long long)order_key(fS) << 32 | S;
                todo |= 1u << k;
            }
        }
        for (; todo; todo &= todo - 1) {
            uint32_t S, u, v;
            float fS;
            slot(list[threadIdx.x + NT * (__ffs(todo) - 1)], S, fS, u, v);
            ok &= merge_steps<true>(fd.W, f, S, fS, u, v);
        }
    }
    if (!ok) raise_status(status, ST_TIMEOUT);
}

// --------------------------------------------------------------- k_repair
//
// Repair (Algorithm 5) after the cross-tile merges: T[u] = (s, Rep(u, s))
// restores minimality. Level comparisons use the vertex order, not values
// alone: with tied values a saddle s' equal in value to s but after it in the
// order is not yet part of the sublevel set at s. Concurrent repairs only
// replace a target by one further along the same chain below the same level,
// so a stale copy of an entry is still a valid (longer) way to the same
// answer: every read of a triplet here is an ordinary cached load.
//
// One CTA per tile of the tile kernel, a thread per column. The chains that
// the tile's vertices climb are copied to shared memory once, as a small
// forest of link words that is closed up to the tile's highest value:
//  1. number the tile's minima densely (the tile kernel left a bit per
//     vertex, the tile's highest key, and in the word of every inner vertex
//     the local id of the minimum it descends to);
//  2. a node per minimum: its link's saddle (key, and local id if the saddle
//     lies in the tile) and the node of its target. A target outside the tile
//     is entered in a small hash, and its own link follows in the next round,
//     until the links lie above the tile's highest value. On a lognormal
//     field a tile has about 450 minima and 46 such foreign nodes, in 4 rounds;
//  3. repair the branch minima by climbing the forest (past its edge, the
//     global chain);
//  4. repair every inner vertex: from its minimum's node follow the links at
//     or below it (2.4 on average), voting so that the warp stays together.
// Tables that are full (more than kMin minima, a crowded hash) leave a link
// without a node; whoever needs it goes on along the global chain.
//
// What it costs, on the 1024^3 lognormal field: 8.5 ms, 10.8 ms with labels
// (11.7 and 14.2 ms with copies of each target's first 8 links found through
// a hash per vertex, from triplets that the tile kernel had repaired itself
// at 3.8 ms more), 11.1 ms with labels and the pairs marked, which saves 1.2 ms
// of the pair compaction. With 6 CTAs per SM: numbering 1.0, links 3.2 (chains
// of dependent reads), targets and labels 0.7 to 1.2, inner vertices 4.9 to
// 5.4 (16 to 24 bytes each way per vertex, 130 thread instructions). Issue
// slots are 60 % busy. Climbing the forest before its targets are repaired
// costs 1.4 ms more; marking the pairs in the loop over the inner vertices 1.0
// ms more than from the list of minima.
//
// With LAB the pass also labels the components of G_t (the labels of
// k_labels) where it already stands. The representative of u at level t is
// the end of the walk from u along links with f(s) <= t (Algorithm 4 with a
// value test). Any valid triplet forest gives the same end, repaired or not:
// a walk stops at the first link above t, and every link it passes joins two
// vertices of one component of G_t, the second deeper. So a node at the edge
// of the forest takes its label from a global walk, every other node by
// climbing the forest to t or to such a node, and a vertex in G_t has the
// label of its representative's node: t >= f(u), so the walk at t passes the
// representative at u. Concurrent repairs move entries along their own
// chains below their own saddles, which keeps every walk's end.

// The end of the walk from x along links at or below level (fS, S)
// (Algorithm 4 along the global chain), the next triplet read beside the
// saddle's value. ok = false if the walk ran out of steps. Out of line, like
// label_walk: few vertices need it, and inlined copies slow the common path.
template <bool WIDE>
__device__ __noinline__ typename Tri<WIDE>::Id repair_walk(const uint64_t *W, const float *f, float sg,
                                                          typename Tri<WIDE>::Id x, typename Tri<WIDE>::Id S,
                                                          float fS, bool *ok)
{
    using Id = typename Tri<WIDE>::Id;
    Id s, v;
    Tri<WIDE>::load(W, x, s, v);
    for (uint32_t h = 0; h <= kChaseLimit; h++) {
        if (s == x && v == x) return x;
        const float fs = sg * __ldg(f + s);
        Id ns, nv;
        Tri<WIDE>::load(W, v, ns, nv);
        if (s != S && !(fs < fS || (fs == fS && s < S))) return x;
        x = v, s = ns, v = nv;
    }
    *ok = false;
    return x;
}

// The label at t of the component reached from x: the end r of the walk
// along links with f(s) <= t (Algorithm 4 with a value test), or 0xFFFFFFFF
// when eps > 0 and r heads a branch of persistence below eps (its component
// lies in a filled pit). Bit 32 of the result is set if the walk ran out of
// steps.
__device__ __noinline__ uint64_t label_walk(const uint64_t *W, const Field f, uint32_t x, float t, float eps)
{
    for (uint32_t h = 0;; h++) {
        const uint64_t T = W[x];
        const uint32_t s = tri_s(T), v = tri_v(T);
        if ((s == x && v == x) || !(f[s] <= t)) break;
        x = v;
        if (h >= kChaseLimit) return (1ull << 32) | x;
    }
    if (eps > 0.0f) {
        const uint32_t s = tri_s(W[x]);
        if (s != x && !(f[s] - f[x] >= eps)) return 0xFFFFFFFFull;
    }
    return x;
}

template <int LX, int LY, int LZ, bool LAB, bool WIDE>
struct RepairShape {
    static constexpr uint32_t TV = 1u << (LX + LY + LZ), NT = 1u << (LX + LY);
    static constexpr uint32_t kMin = TV / 4 / kRepairShrink;    // minima with a node
    static constexpr uint32_t kHash = TV / 16 / kRepairShrink;  // hash slots (nodes) of foreign minima
    static constexpr uint32_t kNodes = kMin + kHash;
    // shared memory: link word and global id (with LAB also the label) of
    // every node (and of the one that stands for none), hash keys, the node of
    // each minimum by x-adjacent pair, the foreign nodes in the order they
    // were entered; with LAB the local id of each minimum, a bit per vertex
    static constexpr size_t kSmem = (size_t)(kNodes + 4) * 8 + (size_t)kNodes * (LAB || WIDE ? 8 : 4) +
                                    (size_t)kHash * (WIDE ? 8 : 4) + (size_t)TV / 2 * 2 + (size_t)kHash * 2 +
                                    (LAB ? (size_t)kMin * 2 + TV / 8 : 0);
    static_assert((kMin + kHash) % 2 == 0, "the bits after the 16-bit arrays are 4-byte aligned");
    static constexpr int kFit = (int)(227 * 1024 / (kSmem + 1024));
    // CTAs per SM the registers are limited for: 7 of 256 threads (32
    // registers, 20 bytes spilt) take 8.5 ms without labels on the 1024^3 field,
    // 6 take 9.7; with labels 6 (40 registers) take 10.8 ms and 7 take 11.0
    static constexpr int kWant = (LAB || WIDE ? 1536 : 1792) / NT, kCTAs = kFit < kWant ? kFit : kWant;
};

// A build that failed (a value is not finite, a loop ran out of steps) leaves
// valid ids behind too: the inner vertices of the tile, whose words still hold
// local ids, become roots, so that a later call on the triplets reads nothing
// out of range. The repair kernel of a single field does this where it skips;
// in batches and with wide ids the call made it spill registers (687 -> 718,
// 1406 -> 1490 us), so there a kernel of its own looks at the status word, 5 us.
template <class Loc, bool WIDE>
constexpr bool kLeaveApart = WIDE || !std::is_same<Loc, OneField>::value;

template <int LX, int LY, int LZ, bool WIDE>
__device__ __noinline__ void leave_valid(uint64_t *W, uint32_t nx, uint32_t ny, uint32_t nz, uint32_t ntx, uint32_t nty,
                                         uint32_t tile)
{
    using TR = Tri<WIDE>;
    using Id = typename TR::Id;
    constexpr uint32_t TX = 1u << LX, TY = 1u << LY, TZ = 1u << LZ;
    const uint32_t x = tile % ntx * TX + (threadIdx.x & (TX - 1)),
                   y = tile / ntx % nty * TY + (threadIdx.x >> LX), z0 = tile / (ntx * nty) * TZ;
    if (x >= nx || y >= ny) return;
    const uint32_t wz = tile_side(z0, TZ, nz);
    for (uint32_t z = 0; z < wz; z++) {
        const Id u = ((Id)(z0 + z) * ny + y) * nx + x;
        Id s, v;
        TR::load(W, u, s, v);
        if (s == TR::kInner) s = v = u;
        TR::store(W, u, s, v);  // wide: without the merges' tags
    }
}
template <int LX, int LY, int LZ, class Loc, bool WIDE>
__global__ void __launch_bounds__(1 << (LX + LY)) k_leave_valid(Loc loc, uint32_t ntiles, const uint32_t *status)
{
    if (block_skips(status))
        for (uint32_t b = blockIdx.x; b < ntiles; b += gridDim.x) {
            uint32_t t;
            const FieldDesc d = loc.tile(b, t);
            leave_valid<LX, LY, LZ, WIDE>(d.W, d.nx, d.ny, d.nz, d.ntx, d.nty, t);
        }
}

template <int LX, int LY, int LZ, class Loc, bool LAB, bool WIDE = false>
__global__ void __launch_bounds__(1 << (LX + LY), RepairShape<LX, LY, LZ, LAB, WIDE>::kCTAs)
    k_repair(Loc loc, uint32_t *status, const LabelArgs la)
{
    if (block_skips(status)) {
        if constexpr (!kLeaveApart<Loc, WIDE>) {
            uint32_t t;
            const FieldDesc d = loc.tile(blockIdx.x, t);
            leave_valid<LX, LY, LZ, WIDE>(d.W, d.nx, d.ny, d.nz, d.ntx, d.nty, t);
        }
        return;
    }
    static_assert(!(LAB && WIDE), "labels have 32-bit ids");
    using RS = RepairShape<LX, LY, LZ, LAB, WIDE>;
    using TR = Tri<WIDE>;
    using Id = typename TR::Id;
    constexpr uint32_t TX = 1u << LX, TY = 1u << LY, TZ = 1u << LZ, TV = RS::TV, NT = RS::NT, MIN = RS::kMin,
                       HS = RS::kHash, NN = RS::kNodes;
    static_assert((HS & (HS - 1)) == 0, "power of two");
    constexpr uint32_t NONE = kNoLocal;            // no node, no local id
    constexpr Id EMPTY = ~(Id)0;                   // free hash slot (no vertex id)
    constexpr uint32_t kProbes = 16;
    // word of a node whose target found no node, and of node NN, which stands
    // for a minimum without one: stops every climb, and whoever ends there
    // goes on along the global chain
    constexpr uint64_t LOST = (uint64_t)kNoKey << 32 | 0xFFFEFFFFu;
    extern __shared__ __align__(16) uint64_t rep_smem[];
    uint64_t *word = rep_smem;                     // links: saddle's key, its local id (NONE: outside), next node
    uint64_t *out = word + NN + 4;                 // LAB: label and global id of each node, else global id
    Id *ids = reinterpret_cast<Id *>(out);
    Id *hkey = reinterpret_cast<Id *>(out + (LAB || WIDE ? NN : NN / 2));
    uint16_t *node = reinterpret_cast<uint16_t *>(hkey + HS);  // of the minimum of each x-adjacent pair
    uint16_t *order = node + TV / 2;
    uint16_t *lid = order + HS;                    // LAB: local ids of the minima
    uint32_t *pbits = reinterpret_cast<uint32_t *>(lid + MIN);  // LAB: a bit per vertex that begins a pair
    __shared__ uint32_t s_nmin, s_nf;
    auto id_of = [&](uint32_t x) -> Id {
        if constexpr (LAB) return (uint32_t)out[x];
        else return ids[x];
    };

    uint32_t tile;
    const FieldDesc fd = loc.tile(blockIdx.x, tile);
    uint64_t *W = fd.W;
    const float *__restrict__ f = fd.f;
    const float sg = fd.sg;
    const uint32_t nx = fd.nx, ny = fd.ny, nz = fd.nz, ntx = fd.ntx, nty = fd.nty;
    const uint32_t tx = tile % ntx, ty = (tile / ntx) % nty, tz = tile / (ntx * nty);
    const uint32_t x0 = tx * TX, y0 = ty * TY, z0 = tz * TZ;
    const uint32_t wx = min(TX, nx - x0), wy = min(TY, ny - y0), wz = min(TZ, nz - z0);
    const Id nxy = (Id)nx * ny;
    const Id base = (Id)z0 * nxy + (Id)y0 * nx + x0;
    const uint32_t lane = threadIdx.x & 31, col = threadIdx.x, cx = col & (TX - 1), cy = col >> LX;
    const bool inx = cx < wx && cy < wy;
    const Id ucol = base + (Id)cy * nx + cx;       // vertex z of the column: ucol + z * nxy
    bool ok = true;
    auto val = [&](Id u) { return sg * __ldg(f + u); };
    // local id of vertex v, NONE outside the tile
    const float rnxy = 1.0f / (float)nxy, rnx = 1.0f / (float)nx;
    auto local_of = [&](Id v) -> uint32_t { return tile_local<LX, LY, LZ, Id>(v - base, nxy, nx, rnxy, rnx, wx, wy, wz); };
    auto id_at = [&](uint32_t l) -> Id {
        return base + (Id)(l >> (LX + LY)) * nxy + (Id)((l >> LX) & (TY - 1)) * nx + (l & (TX - 1));
    };
    // the tile's rows of values and triplets start on their way to L2: the
    // forest is built with dependent loads, each a trip to HBM otherwise
    auto prefetch_tri = [&](Id u) { asm volatile("prefetch.global.L2 [%0];" ::"l"(W + (WIDE ? 2 : 1) * (size_t)u)); };
    if (threadIdx.x < TV / 16) {
        const uint32_t l = 16 * threadIdx.x, lx = l & (TX - 1), ly = (l >> LX) & (TY - 1), lz = l >> (LX + LY);
        if (lx < wx && ly < wy && lz < wz) {
            const Id u = id_at(l);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(f + u));
            prefetch_tri(u);
            if (WIDE && lx + 8 < wx) prefetch_tri(u + 8);
        }
    }
    for (uint32_t i = threadIdx.x; i < HS; i += NT) hkey[i] = EMPTY;
    if (LAB)
        for (uint32_t i = threadIdx.x; i < TV / 32; i += NT) pbits[i] = 0;
    if (threadIdx.x == 0) s_nmin = 0, s_nf = 0, word[NN] = LOST;
    __syncthreads();

    // 1. number the tile's minima (the bits the tile kernel left per column)
    using TS = Tile<LX, LY, LZ>;
    const uint32_t *note = fd.faces;
    uint32_t minima = 0, kmax;
    if constexpr (WIDE) {
        const uint32_t mx = min(nx, TX), words = wide_note_words(nx, ny);
        note += (size_t)tile * words;
        if (cx < mx && cy < min(ny, TY)) minima = reinterpret_cast<const uint16_t *>(note)[cx + cy * mx];
        kmax = note[words - 1];
    } else {
        note += (size_t)tile * TS::kTileWords + TS::kFaceWords;
        minima = reinterpret_cast<const uint16_t *>(note)[col], kmax = note[NT / 2];
    }
    {
        const uint32_t cnt = __popc(minima);
        uint32_t incl = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        uint32_t pos = 0;
        if (lane == 31) pos = atomicAdd(&s_nmin, incl);
        pos = __shfl_sync(0xffffffffu, pos, 31) + incl - cnt;
        for (uint32_t m = minima; m; m &= m - 1, pos++) {
            const uint32_t z = __ffs(m) - 1;
            node[(col + z * NT) >> 1] = (uint16_t)(pos < MIN ? pos : NN);
            if (pos < MIN) {
                if constexpr (LAB) out[pos] = ucol + z * nxy, lid[pos] = (uint16_t)(col + z * NT);
                else ids[pos] = ucol + z * nxy;
            }
        }
    }
    __syncthreads();
    const uint32_t nmin = min(s_nmin, MIN);

    // 2. links of the nodes
    volatile Id *vhk = hkey;
    auto node_of = [&](Id v) -> uint32_t {         // the node of minimum v, entered if it is a new foreign one
        const uint32_t l = local_of(v);
        if (l != NONE) return node[l >> 1];
        uint32_t h = ((uint32_t)v * 0x9E3779B1u) >> (32 - log2i(HS));
        for (uint32_t p = 0; p < kProbes; p++) {
            Id k = vhk[h];
            if (k == EMPTY) {
                if constexpr (WIDE)
                    k = atomicCAS(reinterpret_cast<unsigned long long *>(hkey + h), (unsigned long long)EMPTY,
                                  (unsigned long long)v);
                else k = atomicCAS(hkey + h, EMPTY, v);
                if (k == EMPTY) {
                    order[atomicAdd(&s_nf, 1u)] = (uint16_t)h;
                    if constexpr (LAB) out[MIN + h] = v;
                    else ids[MIN + h] = v;
                    return MIN + h;
                }
            }
            if (k == v) return MIN + h;
            h = (h + 1) & (HS - 1);
        }
        return NN;
    };
    const uint32_t kt = order_key(la.t);
    // the label at t of the component that node x heads or leads out of the forest to
    auto label_from = [&](uint32_t x, bool walk) -> uint32_t {
        if constexpr (!LAB) return 0;
        if (!walk && !(la.eps > 0.0f)) return (uint32_t)id_of(x);
        const uint64_t r = label_walk(W, Field{f, sg}, (uint32_t)id_of(x), la.t, la.eps);
        if (r >> 32) ok = false;
        return (uint32_t)r;
    };
    auto set_label = [&](uint32_t x, uint32_t label) { reinterpret_cast<uint32_t *>(out)[2 * x + 1] = label; };
    auto enter = [&](uint32_t x, Id u, Id s, Id v, float fs) {
        uint32_t ks = kNoKey, sl = NONE, next = NONE;
        if (!(s == u && v == u)) {
            ks = order_key(fs);
            sl = local_of(s);
            if (ks <= kmax) next = node_of(v);
        }
        word[x] = next == NN ? LOST : (uint64_t)ks << 32 | sl << 16 | next;
        if (LAB && next >= NN) set_label(x, label_from(x, ks <= kt));
    };
    // the tile's minima, two per thread with their loads side by side
    for (uint32_t i = threadIdx.x; i < nmin; i += 2 * NT) {
        Id u[2], s[2], v[2];
        float fs[2];
#pragma unroll
        for (uint32_t k = 0; k < 2; k++) {
            u[k] = id_of(min(i + k * NT, nmin - 1));
            TR::load(W, u[k], s[k], v[k]);
        }
#pragma unroll
        for (uint32_t k = 0; k < 2; k++) {
            fs[k] = val(s[k]);
            prefetch_tri(v[k]);                    // read in the next round if it is a new foreign node
        }
#pragma unroll
        for (uint32_t k = 0; k < 2; k++)
            if (i + k * NT < nmin) enter(i + k * NT, u[k], s[k], v[k], fs[k]);
    }
    for (uint32_t done = 0;;) {
        __syncthreads();
        const uint32_t nf = s_nf;
        __syncthreads();
        if (done >= nf) break;
        for (uint32_t i = done + threadIdx.x; i < nf; i += NT) {
            const uint32_t x = MIN + order[i];
            const Id u = id_of(x);
            Id s, v;
            TR::load(W, u, s, v);
            prefetch_tri(v);
            enter(x, u, s, v, val(s));
        }
        done = nf;
    }

    // Climbs in the forest: from node x (its word w) follow the links at or
    // below a level, a comparison of the words as in the tile kernel. Where the
    // link's saddle or the level's lies outside the tile, its local id is NONE
    // and the comparison is by key alone; on equal keys the ids decide, read
    // from W. While a lane can go on by the words alone, lanes that need the ids
    // wait, so a warp's rounds may add up to all its lanes' links, each lane
    // passing a node at most once; a climb that is not done by then raises
    // ST_TIMEOUT.
    constexpr uint32_t kRounds = 32 * (NN + 1);
    auto link_next = [](uint64_t w) { return (uint32_t)w & 0xFFFFu; };
    auto saddle_before = [&](uint32_t x, Id S) -> bool {
        Id s, v;
        TR::load(W, id_of(x), s, v);
        return s <= S;
    };

    // 3. repair the nodes' targets, in the forest (which shortens the climbs
    //    that follow) and, for the tile's minima, in W. A node whose link has
    //    a node lies at or below the tile's highest key, and so do the links it
    //    follows; a minimum with a higher saddle goes along the global chain.
    //    With la.mask the minima that begin a pair are marked on the way: those
    //    whose saddle is not the minimum itself (the cross-tile merges make
    //    that of a minimum of the tile that is none of the grid) and, with
    //    eps, lies high enough above it.
    auto mark = [&](uint32_t l, Id u, Id sd, float fs) {
        if (sd == u || (la.eps > 0.0f && !(fs - val(u) >= la.eps))) return;
        atomicOr(pbits + (l >> 5), 1u << (l & 31));
    };
    auto mark_root = [&](Id u) {
        atomicAdd(reinterpret_cast<unsigned long long *>(la.meta + 1), 1ull);
        la.meta[2] = u;
    };
    const uint32_t nf = s_nf, nall = nmin + nf;
    volatile uint64_t *vword = word;
    for (uint32_t i0 = 0; i0 < nall; i0 += NT) {
        const uint32_t i = i0 + threadIdx.x;
        const uint32_t n = i < nmin ? i : i < nall ? MIN + order[i - nmin] : NN;
        const uint64_t w = vword[n];
        const uint32_t ks = (uint32_t)(w >> 32), sl = (uint32_t)w >> 16, x0 = link_next(w);
        const bool link = x0 != NONE;
        const uint64_t lim = sl != NONE ? w | 0xFFFFu : ((uint64_t)ks << 32) - 1;
        uint32_t x = link ? x0 : NN;
        uint64_t wx_ = vword[x];
        for (uint32_t h = 0;; h++) {
            if (h == kRounds) {
                ok = false;
                break;
            }
            const bool go = wx_ <= lim && link;
            if (!__any_sync(0xffffffffu, go)) {
                bool tie = link && (uint32_t)(wx_ >> 32) == ks && (sl == NONE || (uint32_t)wx_ >= 0xFFFF0000u);
                if (!__any_sync(0xffffffffu, tie)) break;
                if (tie) {
                    Id s, v;
                    TR::load(W, id_of(n), s, v);
                    tie = saddle_before(x, s);
                }
                if (!__any_sync(0xffffffffu, tie)) break;
                x = tie ? link_next(wx_) : x;
            } else {
                x = go ? link_next(wx_) : x;
            }
            wx_ = vword[x];
        }
        const bool left = link && (uint32_t)wx_ == (uint32_t)LOST;  // further along the global chain
        if (link && !left && x != x0) vword[n] = (w & ~(uint64_t)0xFFFFu) | x;
        if (i >= nmin) continue;                   // foreign
        const Id u = id_of(n);
        if (ks == kNoKey && w != LOST) {           // the root
            if (LAB && la.mask) mark_root(u);
            continue;
        }
        Id s, v = 0;
        if (!link || left || sl == NONE) TR::load(W, u, s, v);
        else s = id_at(sl);
        if constexpr (LAB) {
            if (la.mask) mark(lid[n], u, s, la.eps > 0.0f ? val(s) : 0.0f);
        }
        if (!link || left) TR::store(W, u, s, repair_walk<WIDE>(W, f, sg, left ? id_of(x) : v, s, val(s), &ok));
        else if (x != x0 || WIDE) TR::store(W, u, s, id_of(x));
    }
    // with LAB the labels of the nodes (those without a next node have theirs)
    if constexpr (LAB) {
        __syncthreads();
        const uint64_t limt = (uint64_t)kt << 32 | 0xFFFFFFFFu;
        for (uint32_t i0 = 0; i0 < nall; i0 += NT) {
            const uint32_t i = i0 + threadIdx.x;
            const uint32_t n = i < nmin ? i : i < nall ? MIN + order[i - nmin] : NN;
            uint32_t x = n;
            uint64_t w = word[n];
            const bool link = link_next(w) != NONE;
            for (uint32_t h = 0; h < NN; h++) {
                const bool go = w <= limt && link_next(w) != NONE;
                if (!__any_sync(0xffffffffu, go)) break;
                x = go ? link_next(w) : x;
                w = word[x];
            }
            if (link)
                set_label(n, link_next(w) == NONE ? reinterpret_cast<volatile uint32_t *>(out)[2 * x + 1]
                                                  : label_from(x, false));
        }
    }
    // minima without a node
    if (s_nmin > MIN) {
        for (uint32_t m = minima; m; m &= m - 1) {
            const uint32_t z = __ffs(m) - 1;
            if (node[(col + z * NT) >> 1] != NN) continue;
            const Id u = ucol + z * nxy;
            Id s, v;
            TR::load(W, u, s, v);
            if (!(s == u && v == u)) TR::store(W, u, s, repair_walk<WIDE>(W, f, sg, v, s, val(s), &ok));
            else if (WIDE) TR::store(W, u, s, v);
            if constexpr (LAB) {
                if (la.mask && s == u && v == u) mark_root(u);
                else if (la.mask) mark(col + z * NT, u, s, val(s));
            }
            if constexpr (LAB) {
                uint32_t lab = 0xFFFFFFFFu;
                if (val(u) <= la.t) {
                    const uint64_t r = label_walk(W, Field{f, sg}, u, la.t, la.eps);
                    if (r >> 32) ok = false;
                    lab = (uint32_t)r;
                }
                la.labels[u] = lab;
            }
        }
    }
    __syncthreads();
    if constexpr (LAB) {
        // the bits row by row: 16 or 32 vertices (build_mask sees to it that
        // they fill whole pieces)
        constexpr uint32_t ROW = TX, rows = TV / ROW;
        if (la.mask && threadIdx.x < rows) {
            static_assert(ROW == 16 || ROW == 32, "rows of 16 or 32 vertices");
            const uint32_t r = threadIdx.x, y = r & (TY - 1), z = r >> LY;
            const Id u = base + (Id)z * nxy + (Id)y * nx;
            if (y < wy && z < wz) {
                if constexpr (ROW == 16)
                    reinterpret_cast<uint16_t *>(la.mask)[u >> 4] = reinterpret_cast<const uint16_t *>(pbits)[r];
                else la.mask[u >> 5] = pbits[r];
            }
        }
    }

    // 4. inner vertices, the next row's value and word loaded ahead (rows
    //    unrolled by 4 or 8 with their loads first measured slower: the
    //    kernel then waits for instructions; two rows ahead: no faster)
    uint32_t lost = 0;                             // bit z: the climb left the forest
    auto row = [&](uint32_t z, float &fu, uint32_t &m) {
        const bool in = inx && z < wz, inner = in && !((minima >> z) & 1u);
        const Id u = ucol + z * nxy;
        fu = 0.0f, m = 0;
        if (LAB ? in : inner) fu = val(u);
        if (inner) m = (uint32_t)W[WIDE ? 2 * u + 1 : u];
    };
    float fnext;
    uint32_t mnext;
    row(0, fnext, mnext);
#pragma unroll 1
    for (uint32_t z = 0; z < wz; z++) {
        const uint32_t l = col + z * NT;
        const Id u = ucol + z * nxy;
        const bool inner = inx && !((minima >> z) & 1u);
        const float fu = fnext;
        const uint32_t m = inner ? mnext : l;      // the vertex's minimum
        row(z + 1, fnext, mnext);
        const uint32_t ku = order_key(fu);
        const uint64_t lim = inner ? level_word(ku, l) : 0u;
        uint32_t x = inner || (LAB && inx && ((minima >> z) & 1u)) ? node[m >> 1] : NN;
        uint64_t w = word[x];
        for (uint32_t h = 0;; h++) {
            if (h == kRounds) {
                ok = false;
                break;
            }
            const bool go = w <= lim;
            if (!__any_sync(0xffffffffu, go)) {
                // a link of the same key whose saddle lies outside the tile?
                bool tie = inner && (uint32_t)(w >> 32) == ku && (uint32_t)w >= 0xFFFF0000u;
                if (!__any_sync(0xffffffffu, tie)) break;
                if (tie) tie = saddle_before(x, u);
                if (!__any_sync(0xffffffffu, tie)) break;
                x = tie ? link_next(w) : x;
            } else {
                x = go ? link_next(w) : x;
            }
            w = word[x];
        }
        const bool leave = inner && (uint32_t)w == (uint32_t)LOST;
        lost |= (uint32_t)leave << z;
        if (x != NN && !leave) {
            if constexpr (LAB) {
                const uint64_t o = out[x];
                if (inner) W[u] = tri_pack(u, (uint32_t)o);
                la.labels[u] = fu <= la.t ? (uint32_t)(o >> 32) : 0xFFFFFFFFu;
            } else if constexpr (WIDE) {
                reinterpret_cast<ulonglong2 *>(W)[u] = make_ulonglong2(u, ids[x]);
            } else {
                W[u] = tri_pack(u, ids[x]);
            }
        }
    }
    // the few that left the forest follow the global chain from their minimum
    for (; lost; lost &= lost - 1) {
        const Id u = ucol + (__ffs(lost) - 1) * nxy;
        const float fu = val(u);
        const Id r = repair_walk<WIDE>(W, f, sg, id_at((uint32_t)W[WIDE ? 2 * u + 1 : u]), u, fu, &ok);
        if constexpr (WIDE) reinterpret_cast<ulonglong2 *>(W)[u] = make_ulonglong2(u, r);
        else W[u] = tri_pack(u, r);
        if constexpr (LAB) {
            const uint64_t q = label_walk(W, Field{f, sg}, (uint32_t)r, la.t, la.eps);
            if (q >> 32) ok = false;
            la.labels[u] = fu <= la.t ? (uint32_t)q : 0xFFFFFFFFu;
        }
    }
    if (!ok) raise_status(status, ST_TIMEOUT);
}

// ------------------------------------------------------------ host side

// Tile shapes. Variant 0: 16 x 16 x 16, 4096 vertices, 44 KB of shared memory,
// five CTAs of 256 threads per SM. Variant 1: 16 x 16 x 8, for batches of small
// fields that would leave most of a large tile empty. Variant 2: 32 x 16 x 16,
// which a single field may choose (MT_CFG_LARGE_TILES).
template <int V> struct Variant;
template <> struct Variant<0> { static constexpr int LX = 4, LY = 4, LZ = 4; };
template <> struct Variant<1> { static constexpr int LX = 4, LY = 4, LZ = 3; };
template <> struct Variant<2> { static constexpr int LX = 5, LY = 4, LZ = 4; };
template <int V> using TileOf = Tile<Variant<V>::LX, Variant<V>::LY, Variant<V>::LZ>;

void tile_shape(int variant, uint32_t &tx, uint32_t &ty, uint32_t &tz)
{
    if (variant == 1) {
        tx = 1u << Variant<1>::LX, ty = 1u << Variant<1>::LY, tz = 1u << Variant<1>::LZ;
    } else if (variant == 2) {
        tx = 1u << Variant<2>::LX, ty = 1u << Variant<2>::LY, tz = 1u << Variant<2>::LZ;
    } else {
        tx = 1u << Variant<0>::LX, ty = 1u << Variant<0>::LY, tz = 1u << Variant<0>::LZ;
    }
}

// Workspace words per tile: one per end of every edge of its six faces, more
// than its record takes.
uint32_t face_words(int variant)
{
    static_assert(TileOf<0>::kTileWords <= 2 * TileOf<0>::FH && TileOf<1>::kTileWords <= 2 * TileOf<1>::FH &&
                      TileOf<2>::kTileWords <= 2 * TileOf<2>::FH,
                  "the tile records fit the workspace");
    return 2 * (variant == 1 ? TileOf<1>::FH : variant == 2 ? TileOf<2>::FH : TileOf<0>::FH);
}

uint64_t tile_count(int variant, uint32_t nx, uint32_t ny, uint32_t nz)
{
    uint32_t tx, ty, tz;
    tile_shape(variant, tx, ty, tz);
    return (uint64_t)((nx + tx - 1) / tx) * ((ny + ty - 1) / ty) * ((nz + tz - 1) / tz);
}

template <int V, class Loc, bool WIDE = false>
static cudaError_t launch_tile(const Loc &loc, uint32_t ntiles, uint32_t *queue, int persistent_grid,
                               uint32_t *status, cudaStream_t st)
{
    using VV = Variant<V>;
    using TS = TileOf<V>;
    auto kern = k_tile<VV::LX, VV::LY, VV::LZ, Loc, WIDE>;
    static AttrFlags flags;  // per instantiation
    int dev;
    if (flags.pending(dev)) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TS::kSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        flags.done(dev);
    }
    kern<<<queue ? (unsigned)persistent_grid : ntiles, TS::NT, TS::kSmem, st>>>(loc, ntiles, queue, status);
    count_launch();
    return cudaGetLastError();
}

template <int V, class Loc, bool LAB = false, bool WIDE = false>
static cudaError_t launch_repair(const Loc &loc, uint32_t ntiles, uint32_t *status, cudaStream_t st,
                                 const LabelArgs &la = LabelArgs{})
{
    using VV = Variant<V>;
    using RS = RepairShape<VV::LX, VV::LY, VV::LZ, LAB, WIDE>;
    auto kern = k_repair<VV::LX, VV::LY, VV::LZ, Loc, LAB, WIDE>;
    static AttrFlags flags;  // per instantiation
    int dev;
    if (flags.pending(dev)) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RS::kSmem);
        if (e != cudaSuccess) return e;
        flags.done(dev);
    }
    kern<<<ntiles, RS::NT, RS::kSmem, st>>>(loc, status, la);
    count_launch();
    if constexpr (kLeaveApart<Loc, WIDE>) {
        const uint32_t grid = ntiles < 608u ? ntiles : 608u;
        k_leave_valid<VV::LX, VV::LY, VV::LZ, Loc, WIDE><<<grid, RS::NT, 0, st>>>(loc, ntiles, status);
        count_launch();
    }
    return cudaGetLastError();
}

// Build steps with tile variant V (of the knobs in include/mt.h the tile shapes
// alone choose anything).
template <int V, class Loc>
static cudaError_t run_build(const Loc &loc, uint32_t ntiles, uint32_t *queue, int persistent_grid, uint32_t *status,
                             cudaStream_t st, const LabelArgs *la = nullptr)
{
    using VV = Variant<V>;
    cudaError_t e;
    {
        PhaseScope ps(kTile, st);
        if ((e = launch_tile<V>(loc, ntiles, queue, persistent_grid, status, st)) != cudaSuccess) return e;
    }
    {
        PhaseScope ps(kMerge, st);
        uint32_t stride = 1;  // the scattered order costs the large tiles more in L2 than it saves (1024^3: 5.0 -> 6.8 ms)
        if constexpr (std::is_same<Loc, OneField>::value)
            if (V == 0 || thin_tiles(loc.d.ntx, loc.d.nty, ntiles / (loc.d.ntx * loc.d.nty))) stride = scatter_stride(ntiles);
        k_cross<VV::LX, VV::LY, VV::LZ, Loc><<<ntiles, 128, 0, st>>>(loc, stride, status);
        count_launch();
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    PhaseScope ps(kRepair, st);
    if constexpr (std::is_same<Loc, OneField>::value) {
        if (la) return launch_repair<V, Loc, true>(loc, ntiles, status, st, *la);
    }
    return launch_repair<V>(loc, ntiles, status, st);
}

uint32_t *build_mask(uint32_t *faces, uint32_t nx, uint32_t ny, uint32_t nz, uint32_t cfg)
{
    const int v = cfg & MT_CFG_LARGE_TILES ? 2 : 0;
    uint32_t tx, ty, tz;
    tile_shape(v, tx, ty, tz);
    if (nx % tx != 0) return nullptr;
    constexpr int w0 = TileOf<0>::kTileWords, w2 = TileOf<2>::kTileWords;
    static_assert(2 * TileOf<0>::FH - w0 >= TileOf<0>::TV / 32 && 2 * TileOf<2>::FH - w2 >= TileOf<2>::TV / 32,
                  "a bit per vertex fits behind the records");
    static_assert(w0 % 4 == 0 && w2 % 4 == 0, "16-byte aligned");
    return faces + tile_count(v, nx, ny, nz) * (v == 2 ? w2 : w0);
}

// A single field in the tile shape of variant V (0, or 2 with MT_CFG_LARGE_TILES).
template <int V>
static cudaError_t build_one(const float *f, uint64_t *W, uint32_t nx, uint32_t ny, uint32_t nz, Workspace &ws,
                             uint32_t *faces, float sg, cudaStream_t st, const LabelArgs *la)
{
    using VV = Variant<V>;
    OneField loc;
    loc.d = FieldDesc{};
    loc.d.f = f;
    loc.d.W = W;
    loc.d.faces = faces;
    loc.d.sg = sg;
    loc.d.nx = nx, loc.d.ny = ny, loc.d.nz = nz;
    loc.d.n = (uint64_t)nx * ny * nz;
    loc.d.ntx = (nx + (1u << VV::LX) - 1) >> VV::LX;
    loc.d.nty = (ny + (1u << VV::LY) - 1) >> VV::LY;
    const uint32_t ntz = (nz + (1u << VV::LZ) - 1) >> VV::LZ;
    const uint64_t ntiles = (uint64_t)loc.d.ntx * loc.d.nty * ntz;
    return run_build<V>(loc, (uint32_t)ntiles, nullptr, 0, ws.status, st, la);
}

cudaError_t launch_build(const float *f, uint64_t *W, uint32_t nx, uint32_t ny, uint32_t nz, Workspace &ws,
                         uint32_t *faces, float sg, cudaStream_t st, uint32_t cfg, const LabelArgs *la)
{
    if (cfg & MT_CFG_LARGE_TILES) return build_one<2>(f, W, nx, ny, nz, ws, faces, sg, st, la);
    return build_one<0>(f, W, nx, ny, nz, ws, faces, sg, st, la);
}

// The tile kernel and the repair pass with 64-bit ids and 128-bit words (the
// wide path), on 16x16x16 tiles.
static_assert(TileOf<0>::TX == 16 && TileOf<0>::TY == 16 && TileOf<0>::TZ == 16, "as wide_note_words has it");

static bool wide_field(const float *f, uint64_t *W2, uint32_t *notes, uint32_t nx, uint32_t ny, uint32_t nz, float sg,
                       OneField &loc, uint64_t &ntiles)
{
    using VV = Variant<0>;
    loc.d = FieldDesc{};
    loc.d.f = f;
    loc.d.W = W2;
    loc.d.faces = notes;
    loc.d.sg = sg;
    loc.d.nx = nx, loc.d.ny = ny, loc.d.nz = nz;
    loc.d.n = (uint64_t)nx * ny * nz;
    loc.d.ntx = (uint32_t)(((uint64_t)nx + (1u << VV::LX) - 1) >> VV::LX);
    loc.d.nty = (uint32_t)(((uint64_t)ny + (1u << VV::LY) - 1) >> VV::LY);
    ntiles = (uint64_t)loc.d.ntx * loc.d.nty * (((uint64_t)nz + (1u << VV::LZ) - 1) >> VV::LZ);
    return ntiles < 0x80000000ull;
}

cudaError_t launch_tile_wide(const float *f, uint64_t *W2, uint32_t *notes, uint32_t nx, uint32_t ny, uint32_t nz, float sg,
                             uint32_t *status, cudaStream_t st)
{
    OneField loc;
    uint64_t ntiles;
    if (!wide_field(f, W2, notes, nx, ny, nz, sg, loc, ntiles)) return cudaErrorInvalidValue;
    return launch_tile<0, OneField, true>(loc, (uint32_t)ntiles, nullptr, 0, status, st);
}

cudaError_t launch_repair_wide(const float *f, uint64_t *W2, uint32_t *notes, uint32_t nx, uint32_t ny, uint32_t nz, float sg,
                               uint32_t *status, cudaStream_t st)
{
    OneField loc;
    uint64_t ntiles;
    if (!wide_field(f, W2, notes, nx, ny, nz, sg, loc, ntiles)) return cudaErrorInvalidValue;
    return launch_repair<0, OneField, false, true>(loc, (uint32_t)ntiles, status, st);
}

cudaError_t launch_batch_build(const FieldDesc *d_descs, uint32_t nfields, uint32_t ntiles, uint32_t cfg,
                               uint32_t *status, uint32_t *queue, cudaStream_t st)
{
    ManyFields loc{d_descs, nfields};
    cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    // persistent grid: as many CTAs as fit on the GPU at once
    const bool small = cfg & MT_CFG_SMALL_TILES;
    const int per_sm = small ? TileOf<1>::kCTAs : TileOf<0>::kCTAs;
    const int grid = device_sms() * per_sm;
    if (small) return run_build<1>(loc, ntiles, queue, grid, status, st);
    return run_build<0>(loc, ntiles, queue, grid, status, st);
}

}  // namespace mt
