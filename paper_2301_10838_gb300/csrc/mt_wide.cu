// Triplet merge trees with wide vertex ids (grids of 2^32 vertices and more).
//
// Section 3.2 of the paper packs the two 32-bit ids of a triplet (s, v) into
// one 64-bit word because SYCL offers no double-word compare-and-swap, which
// caps a grid at 2^32 vertices; Section 5 names wider ids as future work. On
// sm_103a a 128-bit compare-and-swap exists (atom.cas.b128), so this path
// keeps the whole triplet in one 128-bit word, W[u] = (s, v) with two 64-bit
// ids. It computes the same unique triplets as the 32-bit path, in three
// steps of Algorithm 1 (which merges the edges in any order):
//   1. the tile kernel of the 32-bit path (mt_build.cu) builds the merge tree
//      of every 16x16x16 tile in shared memory on 16-bit local ids and writes
//      it with 64-bit ids (launch_tile_wide);
//   2. k_w_cross merges the edges between neighbouring tiles that can matter
//      with the lock-free Merge (Algorithms 2 and 3) on the global 128-bit
//      words, starting from the tile minima their ends descend to;
//   3. the repair pass of the 32-bit path restores minimality (Algorithms 4
//      and 5; launch_repair_wide).
//
// Torn reads. While merges run, every 64-bit half of a word carries the same
// 30-bit version tag above its 34-bit id; a compare-and-swap writes both
// halves with the next tag. A reader that loads the two halves and finds
// different tags saw a concurrent update between them and loads again, so a
// climb never follows a pair (s, v) that no Merge wrote, whatever the
// hardware's atomicity for 128-bit loads. Ids therefore have 34 bits:
// n < 2^34 vertices, more than fit in the 288 GB of one GB300 at the 20 bytes
// per vertex the field and the triplets take. The tile kernel writes tag 0;
// repair writes every word back without its tag.
//
// Pairs: k_w_pairs_count / k_w_scan / k_w_pairs_write (ordered compaction with
// 64-bit offsets). Labels: the labels kernel of the 32-bit path with 64-bit ids
// (launch_labels_wide).
#include <cuda_runtime.h>

#include <cmath>

#include "../../include/mt.h"
#include "mt_device.cuh"
#include "mt_index.h"
#include "mt_internal.h"

namespace mt {
namespace {

constexpr uint32_t kIdBits = 34;
constexpr uint64_t kIdMask = (1ull << kIdBits) - 1;
constexpr uint64_t kMaxWideVertices = 1ull << kIdBits;
constexpr uint32_t kTagMask = (1u << (64 - kIdBits)) - 1;
constexpr uint32_t kWChunk = 4096;         // vertices per pair-compaction chunk
constexpr int kWThreads = 256;

// Workspace: [0, 256) status word, [256, 512) meta (npairs, roots, root),
// then per-chunk pair counts (u32) and offsets (u64), then the notes that the
// tile kernel leaves for the repair pass, or the pair compaction's bits.
struct WideWs {
    uint32_t *status;
    uint64_t *meta;
    uint32_t *counts;
    uint64_t *offsets;
    uint32_t *notes;
    uint64_t nchunks;
};

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

constexpr uint32_t kSide = 16;  // side of a tile (of the tile kernel's, too)

struct Geo {
    uint64_t nx, ny, nz, nxy, n;
};

size_t wide_ws_bytes(const Geo &g)
{
    const uint64_t nchunks = (g.n + kWChunk - 1) / kWChunk, t = kSide;
    const uint64_t tiles = ((g.nx + t - 1) / t) * ((g.ny + t - 1) / t) * ((g.nz + t - 1) / t);
    const size_t notes = tiles * wide_note_words((uint32_t)g.nx, (uint32_t)g.ny) * 4, bits = nchunks * (kWChunk / 8);
    return 512 + al256(nchunks * 4) + al256(nchunks * 8) + al256(notes > bits ? notes : bits);
}

bool carve(void *base, size_t bytes, const Geo &g, WideWs &ws)
{
    const uint64_t n = g.n;
    if (!base || ((uintptr_t)base & 255) || bytes < wide_ws_bytes(g)) return false;
    char *p = static_cast<char *>(base);
    ws.nchunks = (n + kWChunk - 1) / kWChunk;
    ws.status = reinterpret_cast<uint32_t *>(p);
    ws.meta = reinterpret_cast<uint64_t *>(p + 256);
    ws.counts = reinterpret_cast<uint32_t *>(p + 512);
    ws.offsets = reinterpret_cast<uint64_t *>(p + 512 + al256(ws.nchunks * 4));
    ws.notes = reinterpret_cast<uint32_t *>(p + 512 + al256(ws.nchunks * 4) + al256(ws.nchunks * 8));
    return true;
}

// the values as the order sees them (sg = -1: the tree of -f)
struct FieldW {
    const float *f;
    float sg;
    __device__ __forceinline__ float operator[](uint64_t i) const { return sg * __ldg(f + i); }
};

__device__ __forceinline__ bool before_w(float fa, uint64_t a, float fb, uint64_t b)
{
    return fa < fb || (fa == fb && a < b);
}

// 128-bit compare-and-swap of the word at p (two u64: lo, hi); returns the old word.
__device__ __forceinline__ void cas128(uint64_t *p, uint64_t cmp_lo, uint64_t cmp_hi, uint64_t new_lo,
                                       uint64_t new_hi, uint64_t &old_lo, uint64_t &old_hi)
{
    asm volatile("{\n\t.reg .b128 c, w, o;\n\t"
                 "mov.b128 c, {%2, %3};\n\t"
                 "mov.b128 w, {%4, %5};\n\t"
                 "atom.relaxed.gpu.global.cas.b128 o, [%6], c, w;\n\t"
                 "mov.b128 {%0, %1}, o;\n\t}"
                 : "=l"(old_lo), "=l"(old_hi)
                 : "l"(cmp_lo), "l"(cmp_hi), "l"(new_lo), "l"(new_hi), "l"(p)
                 : "memory");
}

// Both halves of a word in one 16-byte load (one memory sector); the
// memory model guarantees each 8-byte half, not the pair.
__device__ __forceinline__ void ld_word(const uint64_t *W, uint64_t u, uint64_t &lo, uint64_t &hi)
{
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "l"(W + 2 * u) : "memory");
}

// A word read during the merges: both halves with the same tag. Returns
// false if every one of a bounded number of reads was torn.
__device__ __forceinline__ bool wload(const uint64_t *W, uint64_t u, uint64_t &lo, uint64_t &hi)
{
    for (int i = 0; i < 1024; i++) {
        ld_word(W, u, lo, hi);
        if ((lo >> kIdBits) == (hi >> kIdBits)) return true;
    }
    return false;
}

// ----------------------------------------------------------------- merge
// Merge(S, a, b): make a and b connected at level S, value fS (Algorithm 3), as
// in the 32-bit path: both climbs side by side, everything a step may need
// read with the step before it. A word read ahead may be torn; it is read
// again, until its halves carry one tag, when the climb moves to it. Returns
// false if a read stayed torn or the step budget ran out.
// 512^3 lognormal: k_w_cross 0.99 ms, 1.31 ms with one climb after the other.
// A merge that is not done soon goes on in the long form, which shortens the
// chains it climbs (merge_steps in mt_device.cuh); the call costs the short form
// 0.03 ms there, and a 65536 x 3 x 3 field of 16 values takes 0.22 ms instead of
// 2.6.
struct WideMerge {
    uint64_t *W;
    FieldW f;

    struct Node {
        uint64_t x, lo, hi;  // vertex, its word
        float fx;            // its value
    };

    __device__ __forceinline__ bool settle(Node &a) const
    {
        return (a.lo >> kIdBits) == (a.hi >> kIdBits) || wload(W, a.x, a.lo, a.hi);
    }

    // where a climb has come from, in the LONG form of a merge: the vertex, its
    // word (lo is the saddle) and its saddle's value
    struct Trail {
        uint64_t x, lo, hi;
        float fs;
    };
    static constexpr uint64_t NONE = ~0ull;

    // x -> y at the trail's saddle, y = a.x -> z at the saddle sa: if sa comes
    // first x is linked to z (see merge_steps in mt_device.cuh)
    __device__ __forceinline__ void shorten(Trail &p, const Node &a, uint64_t sa, float fsa, uint64_t z) const
    {
        if (p.x != NONE && before_w(fsa, sa, p.fs, p.lo & kIdMask)) {
            const uint64_t tag = (uint64_t)(((p.lo >> kIdBits) + 1) & kTagMask) << kIdBits;
            uint64_t olo, ohi;
            cas128(W + 2 * p.x, p.lo, p.hi, (p.lo & kIdMask) | tag, z | tag, olo, ohi);
        }
        p = Trail{a.x, a.lo, a.hi, fsa};
    }

    // 1: done, 0: out of steps, -1: a read stayed torn
    template <bool LONG, uint32_t LIMIT = kMergeStepLimit>
    __device__ __forceinline__ int run(uint64_t &S, float &fS, uint64_t &a, uint64_t &b) const
    {
        Node u{a, 0, 0, f[a]}, v{b, 0, 0, f[b]};
        Trail pu{NONE, 0, 0, 0.0f}, pv = pu;
        ld_word(W, a, u.lo, u.hi);
        ld_word(W, b, v.lo, v.hi);
        for (uint32_t steps = 0; steps < LIMIT; steps++) {
            if (u.x == v.x) return 1;
            if (!settle(u) || !settle(v)) return -1;
            const uint64_t su = u.lo & kIdMask, sv = v.lo & kIdMask;
            Node nu{u.hi & kIdMask, 0, 0, 0.0f}, nv{v.hi & kIdMask, 0, 0, 0.0f};  // behind the links
            const bool ru = su == u.x && nu.x == u.x, rv = sv == v.x && nv.x == v.x;
            const float fsu = f[su], fsv = f[sv];
            nu.fx = f[nu.x], nv.fx = f[nv.x];
            ld_word(W, nu.x, nu.lo, nu.hi);
            ld_word(W, nv.x, nv.lo, nv.hi);
            const bool mu = !ru && (su == S || before_w(fsu, su, fS, S)),
                       mv = !rv && (sv == S || before_w(fsv, sv, fS, S));
            if (LONG && mu) shorten(pu, u, su, fsu, nu.x);
            if (LONG && mv) shorten(pv, v, sv, fsv, nv.x);
            if (mu) u = nu;
            if (mv) v = nv;
            if (mu || mv) continue;
            const bool sw = before_w(v.fx, v.x, u.fx, u.x);  // v is the earlier one: link u under it
            const Node hi = sw ? u : v;
            const uint64_t tag = (uint64_t)(((hi.lo >> kIdBits) + 1) & kTagMask) << kIdBits;
            uint64_t olo, ohi;
            cas128(W + 2 * hi.x, hi.lo, hi.hi, S | tag, (sw ? v.x : u.x) | tag, olo, ohi);
            if (olo == hi.lo && ohi == hi.hi) {
                if (sw ? ru : rv) return 1;  // displaced a root: it carries no link
                S = sw ? su : sv, fS = sw ? fsu : fsv;  // re-insert the displaced link
                if (sw) u = nu, pu.x = NONE;
                else v = nv, pv.x = NONE;
            } else if (sw) {
                u.lo = olo, u.hi = ohi;
            } else {
                v.lo = olo, v.hi = ohi;
            }
        }
        a = u.x, b = v.x;
        return 0;
    }

    __device__ bool merge(uint64_t S, float fS, uint64_t a, uint64_t b) const
    {
        const int r = run<false, kShort>(S, fS, a, b);
        return r ? r > 0 : merge_long(S, fS, a, b);
    }
    __device__ __noinline__ bool merge_long(uint64_t S, float fS, uint64_t a, uint64_t b) const
    {
        return run<true>(S, fS, a, b) > 0;
    }
    static constexpr uint32_t kShort = 32;  // steps before the long form (16: no faster, 96: 65536 x 3 x 3 slower)
};

// One CTA per 16x16x16 tile: the edges from the tile to its +x, +y and +z
// neighbour tiles, merged at the level of their later end (the tile kernel
// has already merged every edge inside a tile). An edge adds nothing if a
// parallel edge of its face beside it has a lower level (both its ends are
// then before the edge's level, and inside the two tiles they are neighbours
// of the edge's ends), so only the local minima of the level over each face
// are merged: about 132 of the 768 edges on a lognormal field. They are
// listed first, so that all lanes have one to merge.
__global__ void __launch_bounds__(256, 4) k_w_cross(FieldW f, Geo g, uint32_t ntx, uint32_t nty, uint64_t *W,
                                                 uint32_t stride, uint32_t *status)
{
    if (block_skips(status)) return;
    constexpr uint32_t F = kSide * kSide;
    constexpr uint64_t kInner = kIdMask;  // saddle id of an inner vertex's word; its target is then a local id
    __shared__ uint64_t lev[3][F];        // (order key, order of the id within the face) of each edge's level
    __shared__ uint16_t list[3 * F];
    __shared__ uint32_t s_n;
    const WideMerge M{W, f};
    const uint32_t tile = stride == 1 ? blockIdx.x : (uint32_t)((uint64_t)blockIdx.x * stride % gridDim.x);
    const uint32_t tx = tile % ntx, ty = (tile / ntx) % nty, tz = tile / (ntx * nty);
    const uint64_t x0 = (uint64_t)tx * kSide, y0 = (uint64_t)ty * kSide, z0 = (uint64_t)tz * kSide;
    const uint32_t wx = (uint32_t)min((uint64_t)kSide, g.nx - x0), wy = (uint32_t)min((uint64_t)kSide, g.ny - y0),
                   wz = (uint32_t)min((uint64_t)kSide, g.nz - z0);
    const uint64_t base = z0 * g.nxy + y0 * g.nx + x0;
    const uint32_t e = threadIdx.x, c1 = e % kSide, c2 = e / kSide, lane = threadIdx.x & 31;
    // the ends of edge (c1, c2) of face dir (0, 1, 2: +x, +y, +z)
    auto ends = [&](uint32_t dir, uint32_t p, uint32_t q, uint64_t &a, uint64_t &b) {
        if (dir == 0) a = base + q * g.nxy + p * g.nx + (kSide - 1), b = a + 1;
        else if (dir == 1) a = base + q * g.nxy + (kSide - 1) * g.nx + p, b = a + g.nx;
        else a = base + (kSide - 1) * g.nxy + q * g.nx + p, b = a + g.nxy;
    };
    if (threadIdx.x == 0) s_n = 0;
    uint64_t mine[3];
#pragma unroll
    for (uint32_t dir = 0; dir < 3; dir++) {
        const bool has = dir == 0 ? x0 + kSide < g.nx : dir == 1 ? y0 + kSide < g.ny : z0 + kSide < g.nz;
        mine[dir] = ~0ull;
        if (has && c1 < (dir == 0 ? wy : wx) && c2 < (dir == 2 ? wy : wz)) {
            uint64_t a, b;
            ends(dir, c1, c2, a, b);
            const float fa = f[a], fb = f[b];
            const uint32_t side = before_w(fa, a, fb, b);  // 1: b is the later end
            const float fs = side ? fb : fa;
            const uint32_t bits = fs == 0.0f ? 0u : __float_as_uint(fs);
            const uint32_t key = (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
            const uint32_t pos = dir == 0 ? 2 * e + side : dir == 1 ? c2 * 2 * kSide + side * kSide + c1 : side * F + e;
            mine[dir] = (uint64_t)key << 32 | pos;
        }
        lev[dir][e] = mine[dir];
    }
    __syncthreads();
#pragma unroll
    for (uint32_t dir = 0; dir < 3; dir++) {
        const uint64_t v = mine[dir], *p = &lev[dir][e];
        const bool keep = v != ~0ull && !((c1 > 0 && p[-1] < v) || (c1 + 1 < kSide && p[1] < v) ||
                                          (c2 > 0 && *(p - kSide) < v) || (c2 + 1 < kSide && p[kSide] < v));
        const uint32_t bal = __ballot_sync(0xffffffffu, keep);
        uint32_t pos = 0;
        if (lane == 0) pos = atomicAdd(&s_n, __popc(bal));
        pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(bal & ((1u << lane) - 1u));
        if (keep) list[pos] = (uint16_t)(dir * F + e);
    }
    __syncthreads();
    bool ok = true;
    for (uint32_t i = threadIdx.x; i < s_n; i += blockDim.x) {
        const uint32_t en = list[i], dir = en / F, ee = en % F;
        uint64_t a, b;
        ends(dir, ee % kSide, ee / kSide, a, b);
        const float fa = f[a], fb = f[b];
        const bool up = before_w(fa, a, fb, b);
        // climbs start at the tile minima the ends descend to
        auto start = [&](uint64_t u, uint64_t tbase) -> uint64_t {
            uint64_t lo, hi;
            ld_word(W, u, lo, hi);
            if ((lo & kIdMask) != kInner) return u;
            const uint32_t l = (uint32_t)hi;
            return tbase + (uint64_t)(l / F) * g.nxy + (uint64_t)(l / kSide % kSide) * g.nx + l % kSide;
        };
        const uint64_t step = dir == 0 ? kSide : dir == 1 ? kSide * g.nx : kSide * g.nxy;
        ok &= M.merge(up ? b : a, up ? fb : fa, start(a, base), start(b, base + step));
    }
    if (!ok) raise_status(status, ST_TIMEOUT);
}

// ----------------------------------------------------------------- pairs
// One CTA per chunk; warp w owns 512 consecutive vertices, read in 16 rows of
// 32 (one 16-byte load each, eight rows loaded before any is used). The count
// leaves a bit per vertex, so that the write reads the words of pairs only.
constexpr int kWRows = kWChunk / kWThreads;  // rows of 32 per warp

__global__ void __launch_bounds__(kWThreads) k_w_pairs_count(const uint64_t *W, uint64_t n, uint32_t *counts,
                                                             uint32_t *mask, uint64_t *meta, const uint32_t *status)
{
    if (block_skips(status)) return;
    __shared__ uint32_t s_cnt;
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t a = blockIdx.x * (uint64_t)kWChunk + warp * (kWRows * 32);
    uint32_t mine = 0;  // lane r: the flags of row r
    constexpr int RB = 8;
#pragma unroll
    for (int q = 0; q < kWRows; q += RB) {
        ulonglong2 T[RB];
#pragma unroll
        for (int r = 0; r < RB; r++) {
            const uint64_t u = a + (q + r) * 32 + lane;
            T[r] = u < n ? reinterpret_cast<const ulonglong2 *>(W)[u] : make_ulonglong2(u, ~u);
        }
#pragma unroll
        for (int r = 0; r < RB; r++) {
            const uint64_t u = a + (q + r) * 32 + lane;
            if (T[r].x == u && T[r].y == u) {
                atomicAdd(reinterpret_cast<unsigned long long *>(meta + 1), 1ull);
                meta[2] = u;
            }
            const uint32_t bal = __ballot_sync(0xffffffffu, T[r].x != u);
            mine = lane == (uint32_t)(q + r) ? bal : mine;
        }
    }
    if (lane < (uint32_t)kWRows) mask[blockIdx.x * (uint64_t)(kWChunk / 32) + warp * kWRows + lane] = mine;
    const uint32_t c = __reduce_add_sync(0xffffffffu, __popc(mine));
    if (lane == 0 && c) atomicAdd(&s_cnt, c);
    __syncthreads();
    if (threadIdx.x == 0) counts[blockIdx.x] = s_cnt;
}

// exclusive scan of the chunk counts into 64-bit offsets (one CTA): warp w
// owns a contiguous range read in coalesced rows of 32; a pass sums the
// ranges, one warp scans the sums, and a second pass scans row by row with
// shuffles on top of the carry
__global__ void __launch_bounds__(1024) k_w_scan(const uint32_t *counts, uint64_t *offsets, uint64_t m,
                                                 uint64_t *meta, const uint32_t *status)
{
    if (block_skips(status)) return;
    __shared__ uint64_t wsum[32];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t per = ((m + 31) / 32 + 31) / 32 * 32;
    const uint64_t a = warp * per, b = a + per < m ? a + per : m;
    uint64_t s = 0;
    for (uint64_t i = a + lane; i < b; i += 32) s += counts[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) wsum[warp] = s;
    __syncthreads();
    if (warp == 0) {
        const uint64_t v = wsum[lane];
        uint64_t incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        wsum[lane] = incl - v;
        if (lane == 31) meta[0] = incl;
    }
    __syncthreads();
    uint64_t carry = wsum[warp];
    for (uint64_t r = a; r < b; r += 32) {
        const uint64_t i = r + lane;
        const uint32_t c = i < b ? counts[i] : 0u;
        uint32_t incl = c;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        if (i < b) offsets[i] = carry + incl - c;
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
}

// ordered write: the chunk's pairs at its offset, by ascending u (one warp
// after another, the flags' ranks within a row)
__global__ void __launch_bounds__(kWThreads, 4) k_w_pairs_write(const uint64_t *W, const uint64_t *offsets,
                                                             const uint32_t *__restrict__ mask, uint64_t *pairs,
                                                             uint64_t cap, const uint32_t *status)
{
    if (block_skips(status)) return;
    constexpr int kWarps = kWThreads / 32;
    __shared__ uint32_t s_wc[kWarps];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t a = blockIdx.x * (uint64_t)kWChunk + warp * (kWRows * 32);
    uint32_t mine = 0;
    if (lane < (uint32_t)kWRows) mine = mask[blockIdx.x * (uint64_t)(kWChunk / 32) + warp * kWRows + lane];
    const uint32_t c = __reduce_add_sync(0xffffffffu, __popc(mine));
    if (lane == 0) s_wc[warp] = c;
    uint64_t s[kWRows];
#pragma unroll
    for (int r = 0; r < kWRows; r++) {
        const uint32_t q = __shfl_sync(0xffffffffu, mine, r);
        s[r] = (q >> lane) & 1u ? W[2 * (a + r * 32 + lane)] : 0;
    }
    __syncthreads();
    uint64_t run = offsets[blockIdx.x];
    for (uint32_t w = 0; w < warp; w++) run += s_wc[w];
    const bool one = ((uintptr_t)pairs & 15) == 0;  // the list is only 8-byte aligned
#pragma unroll
    for (int r = 0; r < kWRows; r++) {
        const uint64_t u = a + r * 32 + lane;
        const uint32_t q = __shfl_sync(0xffffffffu, mine, r);
        if ((q >> lane) & 1u) {
            const uint64_t pos = run + __popc(q & ((1u << lane) - 1u));
            if (pos < cap) {
                if (one) reinterpret_cast<ulonglong2 *>(pairs)[pos] = make_ulonglong2(u, s[r]);
                else pairs[2 * pos] = u, pairs[2 * pos + 1] = s[r];
            }
        }
        run += __popc(q);
    }
}

mt_status wide_grid(mt_grid g, Geo &geo)
{
    if (g.nx == 0 || g.ny == 0 || g.nz == 0) return MT_ERR_INVALID;
    geo.nx = g.nx, geo.ny = g.ny, geo.nz = g.nz;
    geo.nxy = geo.nx * geo.ny;
    geo.n = geo.nxy * geo.nz;
    if (geo.n >= kMaxWideVertices) return MT_ERR_TOO_LARGE;
    return MT_OK;
}

}  // namespace
}  // namespace mt

using namespace mt;

extern "C" {

size_t mt_wide_workspace_bytes(mt_grid g)
{
    Geo geo;
    if (wide_grid(g, geo) != MT_OK) return 0;
    return wide_ws_bytes(geo);
}

mt_status mt_build_triplets_wide(const float *d_f, mt_grid g, uint64_t *d_W, void *d_ws, size_t ws_bytes,
                                 uint32_t flags, void *stream)
{
    Geo geo;
    mt_status st = wide_grid(g, geo);
    if (st != MT_OK) return st;
    if (!d_f || !d_W || ((uintptr_t)d_f & 3) || ((uintptr_t)d_W & 15) || (flags & ~MT_SUPERLEVEL))
        return MT_ERR_INVALID;
    WideWs ws;
    if (!carve(d_ws, ws_bytes, geo, ws)) return MT_ERR_INVALID;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const float sg = (flags & MT_SUPERLEVEL) ? -1.0f : 1.0f;
    const FieldW f{d_f, sg};
    if (cudaMemsetAsync(ws.status, 0, 512, s) != cudaSuccess) return MT_ERR_CUDA;
    {
        PhaseScope ps(kTile, s);
        if (launch_tile_wide(d_f, d_W, ws.notes, g.nx, g.ny, g.nz, sg, ws.status, s) != cudaSuccess) return MT_ERR_CUDA;
    }
    const uint32_t ntx = (uint32_t)((geo.nx + kSide - 1) / kSide), nty = (uint32_t)((geo.ny + kSide - 1) / kSide),
                   ntz = (uint32_t)((geo.nz + kSide - 1) / kSide);
    {
        PhaseScope ps(kMerge, s);
        // Thin grids are merged in scattered order: a line of 2^18 constant
        // vertices 0.10 ms instead of 0.20. With 16-byte words others lose more to
        // L2 than shorter chains give back: 512^3 lognormal 1.00 ms, in order 0.96.
        const uint32_t tiles = ntx * nty * ntz, stride = thin_tiles(ntx, nty, ntz) ? scatter_stride(tiles) : 1u;
        k_w_cross<<<tiles, 256, 0, s>>>(f, geo, ntx, nty, d_W, stride, ws.status);
        count_launch();
    }
    {
        PhaseScope ps(kRepair, s);
        if (launch_repair_wide(d_f, d_W, ws.notes, g.nx, g.ny, g.nz, sg, ws.status, s) != cudaSuccess) return MT_ERR_CUDA;
    }
    return cudaGetLastError() == cudaSuccess ? MT_OK : MT_ERR_CUDA;
}

mt_status mt_persistence_pairs_wide(const uint64_t *d_W, mt_grid g, uint64_t *d_pairs, uint64_t cap,
                                    uint64_t *h_npairs, uint64_t *h_root, void *d_ws, size_t ws_bytes, void *stream)
{
    Geo geo;
    mt_status st = wide_grid(g, geo);
    if (st != MT_OK) return st;
    if (!d_W || !h_npairs || ((uintptr_t)d_W & 15) || (cap && (!d_pairs || ((uintptr_t)d_pairs & 7))))
        return MT_ERR_INVALID;
    WideWs ws;
    if (!carve(d_ws, ws_bytes, geo, ws)) return MT_ERR_INVALID;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(ws.meta, 0, 3 * sizeof(uint64_t), s) != cudaSuccess) return MT_ERR_CUDA;
    {
        PhaseScope ps(kPairs, s);
        // the bits take the place of the build's notes, which are done with
        uint32_t *mask = ws.notes;
        k_w_pairs_count<<<(unsigned)ws.nchunks, kWThreads, 0, s>>>(d_W, geo.n, ws.counts, mask, ws.meta, ws.status);
        k_w_scan<<<1, 1024, 0, s>>>(ws.counts, ws.offsets, ws.nchunks, ws.meta, ws.status);
        k_w_pairs_write<<<(unsigned)ws.nchunks, kWThreads, 0, s>>>(d_W, ws.offsets, mask, d_pairs, cap, ws.status);
        count_launch(3);
        if (cudaGetLastError() != cudaSuccess) return MT_ERR_CUDA;
    }
    uint64_t meta[4];
    if (readback(ws.meta, ws.status, s, meta) != cudaSuccess) return MT_ERR_CUDA;
    const uint32_t bits = (uint32_t)meta[3];
    if (bits) return status_from_bits(bits);
    *h_npairs = meta[0];
    if (h_root) *h_root = meta[1] == 1 ? meta[2] : ~0ull;
    if (meta[1] != 1) return MT_ERR_INVALID;
    return meta[0] > cap ? MT_ERR_CAPACITY : MT_OK;
}

mt_status mt_components_at_wide(const float *d_f, const uint64_t *d_W, mt_grid g, float t, uint32_t flags,
                                uint64_t *d_labels, void *d_ws, size_t ws_bytes, void *stream)
{
    Geo geo;
    mt_status st = wide_grid(g, geo);
    if (st != MT_OK) return st;
    if (!d_f || !d_W || !d_labels || std::isnan(t) || ((uintptr_t)d_f & 3) || ((uintptr_t)d_W & 15) ||
        ((uintptr_t)d_labels & 7) || (flags & ~MT_SUPERLEVEL))
        return MT_ERR_INVALID;
    WideWs ws;
    if (!carve(d_ws, ws_bytes, geo, ws)) return MT_ERR_INVALID;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const float sg = (flags & MT_SUPERLEVEL) ? -1.0f : 1.0f;
    return launch_labels_wide(d_f, d_W, g.nx, g.ny, g.nz, sg * t, sg, d_labels, ws.status, s) == cudaSuccess
               ? MT_OK
               : MT_ERR_CUDA;
}

}  // extern "C"
