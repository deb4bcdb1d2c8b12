// Device-side building blocks of the triplet merge tree (sm_103a).
//
// Triplet word:  W[u] = (s << 32) | v  encodes the triplet (u, s, v)
// (Section 2.1; one 64-bit word per vertex as in Section 3.2, so that a single
// 64-bit compare-and-swap updates the pair).
// Order:         a < b  <=>  f[a] < f[b] || (f[a] == f[b] && a < b).
#pragma once
#include <cstdint>
#include <type_traits>

namespace mt {

// Status bits kept in the first word of the workspace.
enum : uint32_t {
    ST_NONFINITE = 1u,
    ST_TIMEOUT = 2u,
    ST_CAPACITY = 4u,
    ST_CORRUPT = 8u,  // a triplet array given by the caller holds an id >= n
};

// Table sizes of the shared-memory hashes and lists. Each table has a path
// for when it is full (merge an edge in place, climb the global chain); the
// defaults keep those paths rare. A library built with MT_STRESS_TABLES shrinks
// the tables so that the tests reach every such path, and takes wide labels
// through bricks for small fields, too; its results are the same.
#ifdef MT_STRESS_TABLES
constexpr int kTileListShrink = 64;       // k_tile: edge list
constexpr uint32_t kRepairShrink = 64;    // k_repair: nodes of the tile's minima and of foreign ones
constexpr uint32_t kLabelShrink = 64;     // k_labels: hash of chain starts
#else
constexpr int kTileListShrink = 1;
constexpr uint32_t kRepairShrink = 1;
constexpr uint32_t kLabelShrink = 1;
#endif

// Limits of the bounded device loops. A merge that needs more steps than this
// gives up and raises ST_TIMEOUT instead of spinning.
constexpr uint32_t kMergeStepLimit = 1u << 24;
constexpr uint32_t kChaseLimit = 1u << 24;

__device__ __forceinline__ uint32_t tri_s(uint64_t w) { return (uint32_t)(w >> 32); }
__device__ __forceinline__ uint32_t tri_v(uint64_t w) { return (uint32_t)w; }
__device__ __forceinline__ uint64_t tri_pack(uint32_t s, uint32_t v) { return ((uint64_t)s << 32) | v; }

// a before b in the total order (value, index)
__device__ __forceinline__ bool before(float fa, uint32_t a, float fb, uint32_t b)
{
    return fa < fb || (fa == fb && a < b);
}

// Loads of triplet words that other threads may be updating concurrently:
// relaxed, device scope, so that they are not served from a stale L1 line.
__device__ __forceinline__ uint64_t ld_tri(const uint64_t *p)
{
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_tri(uint64_t *p, uint64_t v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t cas_tri(uint64_t *p, uint64_t expect, uint64_t want)
{
    return atomicCAS(reinterpret_cast<unsigned long long *>(p), (unsigned long long)expect,
                     (unsigned long long)want);
}

__device__ __forceinline__ void raise_status(uint32_t *status, uint32_t bit) { atomicOr(status, bit); }

// Whether a CTA skips its work because an earlier error is recorded. The
// status word may be raised by another CTA at any moment, so one thread reads
// it and every thread gets that one answer: kernels with barriers must leave
// (or stay) as a whole block.
__device__ __forceinline__ bool block_skips(const uint32_t *status)
{
    return __syncthreads_or(threadIdx.x == 0 && *(const volatile uint32_t *)status != 0) != 0;
}

// A triplet in global memory: one 64-bit word of two 32-bit ids, or (WIDE) two
// 64-bit words whose ids carry the merges' tags in their upper 30 bits.
template <bool WIDE>
struct Tri {
    using Id = typename std::conditional<WIDE, uint64_t, uint32_t>::type;
    static constexpr uint64_t kMask = (1ull << 34) - 1;
    // saddle id of the word of a tile's inner vertex between the tile kernel
    // and the repair pass; the word's other id is then the local id of
    // the tile minimum the vertex descends to (no merge reads such words:
    // every target of a link is a minimum of its tile)
    static constexpr Id kInner = WIDE ? (Id)kMask : (Id)0xFFFFFFFFu;
    static __device__ __forceinline__ void load(const uint64_t *W, Id u, Id &s, Id &v)
    {
        if constexpr (WIDE) {
            const ulonglong2 w = reinterpret_cast<const ulonglong2 *>(W)[u];
            s = w.x & kMask, v = w.y & kMask;
        } else {
            const uint64_t w = W[u];
            s = tri_s(w), v = tri_v(w);
        }
    }
    static __device__ __forceinline__ void store(uint64_t *W, Id u, Id s, Id v)
    {
        if constexpr (WIDE)
            asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(W + 2 * u), "l"(s), "l"(v) : "memory");
        else st_tri(W + u, tri_pack(s, v));
    }
};

// The values as the order sees them: f itself (sublevel sets), or -f (sg =
// -1) for the tree of the superlevel sets, the split tree. Multiplying by -1
// is exact, and -0 still equals +0.
struct Field {
    const float *f;
    float sg;
    __device__ __forceinline__ float operator[](uint32_t i) const { return sg * __ldg(f + i); }
};

// Algorithm 3 (Merge), lock-free: make a and b connected at level S (value fS)
// in the triplet forest, given that they are connected below S in the graph.
//   1. climb a and b to their deepest vertices u, v below S: follow links
//      while their saddle is at or below S in the vertex order (a root word
//      (x, x) always stops a walk; the paper's pseudocode has no guard for it);
//   2. if they coincide the edge adds nothing;
//   3. otherwise order them so that u comes first and swing v's link to
//      (S, u) with one 64-bit CAS (Algorithm 2);
//   4. the link that v held before, (sv, tv), is not lost: if v was not a
//      root, continue by merging u and tv at level sv. (A displaced root
//      carries no link, so the merge ends there.)
//   5. if the CAS fails another thread moved v first: climb again.
// A merge is a chain of dependent reads, so everything a step may need is
// read with the step before it: both climbs advance side by side, a vertex's
// own value (to order u and v) is read beside its word, a link's saddle
// value beside the next vertex's word and value, and the displaced link's
// saddle value is the one its level test has read.
//
// A merge that is not done after LIMIT steps goes on in the LONG form, which
// shortens the chains that it climbs: where the link of x leads to y and the
// link of y has an earlier saddle than that of x, x is linked to the target z of
// y, at its own saddle. That is what Repair does later, and as sound now: y and z
// are joined below the saddle of x, by the link of y or by the merge that has
// displaced it. Chains of links whose saddles fall, as over the tiles of long
// thin grids and on plateaus, are otherwise climbed to their end by every merge:
// a 65536 x 3 x 3 field of 16 values took 2130 us here and 460 in the repair,
// with this 166 and 154; 128^3 of 16 values 66 + 103, now 48 + 68 us.
// Returns true when the merge is done; (S, u, v) is what is left to merge if not.
template <bool LONG, uint32_t LIMIT = kMergeStepLimit>
__device__ __forceinline__ bool merge_steps(uint64_t *W, const Field f, uint32_t &S, float &fS, uint32_t &u,
                                            uint32_t &v)
{
    uint64_t Tu = ld_tri(W + u), Tv = ld_tri(W + v);
    float fu = f[u], fv = f[v];
    // LONG: the vertex that each climb has come from, its word, its saddle's value
    constexpr uint32_t NONE = 0xFFFFFFFFu;
    uint32_t pu = NONE, pv = NONE;
    uint64_t pTu = 0, pTv = 0;
    float pfu = 0.0f, pfv = 0.0f;
    for (uint32_t steps = 0; steps < LIMIT; steps++) {
        if (u == v) return true;
        const uint32_t su = tri_s(Tu), tu = tri_v(Tu), sv = tri_s(Tv), tv = tri_v(Tv);
        const bool ru = su == u && tu == u, rv = sv == v && tv == v;
        // saddle values, and the words and values behind the links (a root's
        // lead to itself)
        const float fsu = f[su], fsv = f[sv], ftu = f[tu], ftv = f[tv];
        const uint64_t Tnu = ld_tri(W + tu), Tnv = ld_tri(W + tv);
        const bool mu = !ru && (su == S || before(fsu, su, fS, S)), mv = !rv && (sv == S || before(fsv, sv, fS, S));
        if (mu || mv) {
            if (LONG && mu) {
                if (pu != NONE && before(fsu, su, pfu, tri_s(pTu))) cas_tri(W + pu, pTu, tri_pack(tri_s(pTu), tu));
                pu = u, pTu = Tu, pfu = fsu;
            }
            if (LONG && mv) {
                if (pv != NONE && before(fsv, sv, pfv, tri_s(pTv))) cas_tri(W + pv, pTv, tri_pack(tri_s(pTv), tv));
                pv = v, pTv = Tv, pfv = fsv;
            }
            if (mu) u = tu, Tu = Tnu, fu = ftu;
            if (mv) v = tv, Tv = Tnv, fv = ftv;
            continue;
        }
        const bool sw = before(fv, v, fu, u);  // v is the earlier one: link u under it
        const uint32_t lo = sw ? v : u, hi = sw ? u : v;
        const uint64_t Thi = sw ? Tu : Tv;
        const uint64_t old = cas_tri(W + hi, Thi, tri_pack(S, lo));
        if (old == Thi) {
            if (sw ? ru : rv) return true;  // displaced a root
            // go on with the link that hi held: merge lo and its target there
            S = sw ? su : sv, fS = sw ? fsu : fsv;
            if (sw) u = tu, Tu = Tnu, fu = ftu, pu = NONE;
            else v = tv, Tv = Tnv, fv = ftv, pv = NONE;
        } else if (sw) {
            Tu = old;
        } else {
            Tv = old;
        }
    }
    return false;
}

}  // namespace mt
