// Branch decomposition of a finished triplet merge tree.
//
// Every vertex belongs to one branch of the tree (Section 2.1): a minimum u
// (W[u].s != u, or the root W[u] = (u, u)) heads its own branch, and an inner
// vertex u (W[u] = (u, v), v != u) lies on the branch of v, the deepest
// vertex of its component at level f(u), whose minimum the arc through u
// descends to. The call lists all vertices grouped by branch -- branches by
// ascending id of their minimum, each group in the vertex order (value, then
// index), so that it starts with its minimum -- and the offset of every group:
// the per-branch vertex lists that the CPU implementation keeps beside its
// triplets (Section 3.1), as one array.
//
// Most vertices lie on the root's branch (72 % on a lognormal field: above the
// percolation level nearly everything does), most others on branches of a few
// vertices, and a few branches lie between. So a sort of the whole (branch,
// value, index) is split by branch size:
//   1. count the vertices of every branch, and scan the counts into the
//      groups' starts (which are the offsets);
//   2. a vertex of a small branch (at most kSmall vertices) takes a place
//      in its group, in any order, and each small group is then sorted in
//      shared memory by counting, for every member, the members before it;
//   3. the vertices of the root's branch are compacted in index order and
//      sorted by value: a stable radix sort of (32-bit key, id), 8 bits per
//      pass, passes whose digit is the same in every key skipped;
//   4. the other large branches are compacted and sorted by value the same
//      way, then stably by branch if there is more than one. On small grids the
//      root's branch goes this way, too, since launches are what counts there
//      (a constant field of 200^3, where it is the only one: 199 us, 317 with
//      the sort by branch).
// A radix pass is a digit histogram per block, an exclusive scan of the
// histograms (digit major, block minor), and a scatter that ranks each block's
// keys stably: a warp owns a contiguous run of the block's keys, finds the
// lanes sharing a digit, and adds the counts of earlier warps and earlier
// rounds.
//
// What it costs on a 512^3 lognormal field: 5.5 ms (11.3 ms as one sort of
// (branch, value) in eight passes of 12-byte elements): counting 0.5, starts
// 0.4, places 0.9 (atomics with their answers, waited for), small groups 0.4,
// compaction 0.25, four passes over the root's branch 2.6 (a pass over 98 M
// elements: 0.09 histogram, 0.53 scatter, which shared memory bounds with
// 65 % of its bandwidth), the other large branches 0.4. 128^3: 0.31 ms (0.41).
#include <cuda_runtime.h>

#include "../../include/mt.h"
#include "mt_device.cuh"
#include "mt_internal.h"

namespace mt {

// Vertices of the largest branch sorted in shared memory: counting costs a
// branch of k vertices k reads per member, and up to 512 that stays below the
// nine launches and passes another member of the large ones costs.
constexpr uint32_t kSmall = 512;
constexpr uint32_t kWindow = 1024;          // positions whose groups one CTA sorts
constexpr uint32_t kChunkV = kCompactChunk; // vertices per chunk of the ordered compaction
// Vertices up to which the root's branch is sorted among the large ones: that
// costs one more pass over it and a gather, less than the launches saved up to
// about 200^3 (128^3: 26 launches instead of 41).
constexpr uint64_t kTogether = 1u << 23;
constexpr uint32_t kSortThreads = 512, kSortWarps = kSortThreads / 32;
// Rows of 32 keys per warp: blocks of 8192 keys write long runs (98 M keys:
// 0.53 ms a scatter; blocks of 4096 0.56, 2048 0.62), blocks of 2048 keep the
// SMs busy when there are few keys (1.7 M keys: 17 us, 8192 20 us).
constexpr uint32_t kSortRows = 16, kSortRowsFew = 4;
constexpr uint64_t kSortFew = 1u << 21;

// Counters in the workspace.
struct BranchMeta {
    uint32_t root, rstart;              // the root's branch and where its group starts
    uint32_t nlarge, lstart0;           // large branches other than one sorted apart, where the first starts
    uint32_t nbranch, nl[2];            // branches; vertices of the root's branch and of the large ones
    uint32_t kor[2], kand[2];           // OR and AND of their keys
};

// order key of a float: unsigned order = float order, -0 and +0 equal
__device__ __forceinline__ uint32_t okey(float x)
{
    const uint32_t b = x == 0.0f ? 0u : __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// The branch of vertex u; u itself (and bad = true) if the word holds an id
// outside the grid.
__device__ __forceinline__ uint32_t branch_of(uint64_t T, uint32_t u, uint32_t n, bool &bad)
{
    const uint32_t s = tri_s(T), v = tri_v(T);
    if (s >= n || v >= n) {
        bad = true;
        return u;
    }
    return (s == u && v != u) ? v : u;
}

// One thread: the root, found from vertex 0 along the links (whose targets lie
// ever deeper); where the walk ends in a forest that is no tree only decides
// which branch is counted apart. Clears the counters.
__global__ void k_br_root(const uint64_t *W, uint32_t n, BranchMeta *meta)
{
    uint32_t x = 0;
    for (uint32_t h = 0; h < 256; h++) {
        const uint32_t v = tri_v(W[x]);
        if (v >= n || v == x) break;
        x = v;
    }
    *meta = BranchMeta{};
    meta->root = x;
    meta->kand[0] = meta->kand[1] = ~0u;
}

// The lanes of a row that hold the same branch side by side form a run, whose
// first lane speaks for all: `first` is that lane's number, the result the
// number of lanes in it. Lanes with part = false are in no run.
__device__ __forceinline__ uint32_t run_of(uint32_t b, bool part, uint32_t &first)
{
    const uint32_t lane = threadIdx.x & 31, below = (2u << lane) - 1u;
    const uint32_t left = __shfl_up_sync(0xffffffffu, part ? b : ~0u, 1);  // (no branch has id ~0)
    const uint32_t heads = __ballot_sync(0xffffffffu, !part || lane == 0 || left != b);
    first = 31 - __clz(heads & below);
    const uint32_t after = heads & ~below;
    return (after ? __ffs(after) - 1 : 32) - first;
}

// Vertices per branch without the branch's own minimum: cnt[b]; a bit per
// vertex that is one (hmask). A CTA counts `per` vertices, the
// root's branch in registers and the others in a shared-memory hash, one
// atomic per run: the larger of the other branches (a percent of a grid's
// vertices each) would have every run of the grid add to one address.
constexpr uint32_t kCountV = 8192, kCountVFew = 2048, kCountHash = 4096;

__global__ void __launch_bounds__(256) k_br_count(const uint64_t *__restrict__ W, uint32_t n, uint32_t per, uint32_t *cnt,
                                                  uint32_t *hmask, const BranchMeta *meta, uint32_t *status)
{
    __shared__ uint32_t hkey[kCountHash], hcnt[kCountHash], s_root;
    const uint32_t root = meta->root, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    volatile uint32_t *vhk = hkey;
    constexpr uint32_t R = 8, NO = 0xFFFFFFFFu;
    uint32_t mine = 0;
    bool bad = false;
    for (uint32_t i = threadIdx.x; i < kCountHash; i += 256) hkey[i] = NO, hcnt[i] = 0;
    if (threadIdx.x == 0) s_root = 0;
    __syncthreads();
    const uint64_t c0 = (uint64_t)blockIdx.x * per;
    for (uint64_t b0 = c0 + w * (R * 32); b0 < c0 + per; b0 += 8 * R * 32) {
        uint64_t T[R];
#pragma unroll
        for (uint32_t r = 0; r < R; r++) T[r] = b0 + r * 32 + lane < n ? W[b0 + r * 32 + lane] : 0;
        uint32_t hm = 0;
#pragma unroll
        for (uint32_t r = 0; r < R; r++) {
            const uint64_t u64 = b0 + r * 32 + lane;
            const uint32_t u = (uint32_t)u64;
            const bool in = u64 < n;
            const uint32_t b = in ? branch_of(T[r], u, n, bad) : 0u;
            const bool head = in && b == u, part = in && !head && b != root;
            mine += in && !head && b == root;
            const uint32_t bal = __ballot_sync(0xffffffffu, head);
            hm = lane == r ? bal : hm;
            uint32_t first;
            const uint32_t len = run_of(b, part, first);
            if (part && lane == first) {
                uint32_t h = (b * 0x9E3779B1u) >> 20;
                bool done = false;
                for (uint32_t q = 0; q < 8 && !done; q++) {
                    uint32_t k = vhk[h];
                    if (k == NO) k = atomicCAS(hkey + h, NO, b);
                    if (k == NO || k == b) {
                        atomicAdd(hcnt + h, len);
                        done = true;
                    }
                    h = (h + 1) & (kCountHash - 1);
                }
                if (!done) atomicAdd(cnt + b, len);
            }
        }
        if (lane < R && b0 + lane * 32 < n) hmask[b0 / 32 + lane] = hm;
    }
    static_assert(kCountHash == 1u << 12, "the hash takes 12 bits");
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0 && mine) atomicAdd(&s_root, mine);
    if (bad) raise_status(status, ST_CORRUPT);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < kCountHash; i += 256)
        if (hcnt[i]) atomicAdd(cnt + hkey[i], hcnt[i]);
    if (threadIdx.x == 0 && s_root) atomicAdd(cnt + root, s_root);
}

// per chunk of branch ids: heads and vertices
__global__ void __launch_bounds__(256) k_br_sums(const uint32_t *__restrict__ cnt,
                                                 const uint32_t *__restrict__ hmask, uint32_t n, uint32_t *heads,
                                                 uint32_t *sizes)
{
    __shared__ uint32_t sh[2];
    if (threadIdx.x < 2) sh[threadIdx.x] = 0;
    __syncthreads();
    uint32_t h = 0, z = 0;
#pragma unroll
    for (uint32_t r = 0; r < kChunkV / 256; r++) {
        const uint64_t u = (uint64_t)blockIdx.x * kChunkV + r * 256 + threadIdx.x;
        const uint32_t c = u < n ? cnt[u] + ((hmask[u >> 5] >> (u & 31)) & 1u) : 0u;
        h += c != 0;
        z += c;
    }
    h = __reduce_add_sync(0xffffffffu, h);
    z = __reduce_add_sync(0xffffffffu, z);
    if ((threadIdx.x & 31) == 0) atomicAdd(&sh[0], h), atomicAdd(&sh[1], z);
    __syncthreads();
    if (threadIdx.x == 0) heads[blockIdx.x] = sh[0], sizes[blockIdx.x] = sh[1];
}

// Exclusive scans in place of two arrays of m entries, one per CTA, their
// totals to tot[0], tot[1] (warp w owns a contiguous range, read in rows).
__global__ void __launch_bounds__(1024) k_br_scan2(uint32_t *a0, uint32_t *a1, uint32_t m, uint32_t *tot0,
                                                   uint32_t *tot1)
{
    __shared__ uint32_t wsum[32];
    uint32_t *a = blockIdx.x ? a1 : a0;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t per = ((m + 31) / 32 + 31) / 32 * 32;
    const uint64_t lo = (uint64_t)warp * per, hi = lo + per < m ? lo + per : m;
    uint32_t s = 0;
    for (uint64_t i = lo + lane; i < hi; i += 32) s += a[i];
    s = __reduce_add_sync(0xffffffffu, s);
    if (lane == 0) wsum[warp] = s;
    __syncthreads();
    if (warp == 0) {
        const uint32_t v = wsum[lane];
        uint32_t incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        wsum[lane] = incl - v;
        if (lane == 31) {
            uint32_t *tot = blockIdx.x ? tot1 : tot0;
            if (tot) *tot = incl;
        }
    }
    __syncthreads();
    uint32_t carry = wsum[warp];
    for (uint64_t r = lo; r < hi; r += 32) {
        const uint64_t i = r + lane;
        const uint32_t c = i < hi ? a[i] : 0u;
        uint32_t incl = c;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        if (i < hi) a[i] = carry + incl - c;
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
}

// Group starts: the offsets, a bit per position where a group starts, and in
// cnt[b] what the vertices of b need: the next free place of a small group,
// the number of a large branch (marked in lbits) among the large ones.
__global__ void __launch_bounds__(256) k_br_starts(uint32_t *cnt, const uint32_t *__restrict__ hmask,
                                                   uint32_t n, const uint32_t *__restrict__ heads,
                                                   const uint32_t *__restrict__ sizes, uint32_t *offsets, uint64_t cap,
                                                   uint32_t *hbits, uint32_t *lbits, uint32_t *lstart, uint32_t *lsize, bool apart, BranchMeta *meta)
{
    __shared__ uint32_t wh[8], wz[8];
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5, root = meta->root;
    constexpr uint32_t R = kChunkV / 256;   // rows of 32 per warp
    const uint64_t b0 = (uint64_t)blockIdx.x * kChunkV + w * (R * 32);
    uint32_t c[R], h = 0, z = 0;
    const uint32_t hm = lane < R && b0 + lane * 32 < n ? hmask[b0 / 32 + lane] : 0u;  // lane r: the heads of row r
#pragma unroll
    for (uint32_t r = 0; r < R; r++) {
        const uint64_t u = b0 + r * 32 + lane;
        const uint32_t is_head = (__shfl_sync(0xffffffffu, hm, r) >> lane) & 1u;
        c[r] = (u < n ? cnt[u] : 0u) + is_head;
    }
#pragma unroll
    for (uint32_t r = 0; r < R; r++) {
        h += c[r] != 0;
        z += c[r];
    }
    h = __reduce_add_sync(0xffffffffu, h);
    z = __reduce_add_sync(0xffffffffu, z);
    if (lane == 0) wh[w] = h, wz[w] = z;
    __syncthreads();
    uint32_t hrun = heads[blockIdx.x], zrun = sizes[blockIdx.x];
    for (uint32_t q = 0; q < w; q++) hrun += wh[q], zrun += wz[q];
#pragma unroll
    for (uint32_t r = 0; r < R; r++) {
        const uint32_t u = (uint32_t)(b0 + r * 32 + lane);
        const uint32_t bal = __ballot_sync(0xffffffffu, c[r] != 0);
        if (!bal) continue;
        uint32_t incl = c[r];
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        if (c[r]) {
            const uint32_t start = zrun + incl - c[r], rank = hrun + __popc(bal & ((1u << lane) - 1u));
            if (rank < cap) offsets[rank] = start;
            atomicOr(hbits + (start >> 5), 1u << (start & 31));
            if (apart && u == root) {
                meta->rstart = start;
            } else if (c[r] > kSmall) {
                const uint32_t k = atomicAdd(&meta->nlarge, 1u);
                lstart[k] = start, lsize[k] = c[r];
                if (k == 0) meta->lstart0 = start;
                atomicOr(lbits + (u >> 5), 1u << (u & 31));
                cnt[u] = k;
            } else {
                cnt[u] = start;
            }
        }
        hrun += __popc(bal);
        zrun += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const uint32_t nb = meta->nbranch;
        if (nb < cap) offsets[nb] = n;
    }
}

// Vertices of small branches take places in their groups; the others are
// marked (mask[0]: the root's branch when it is sorted apart, mask[1]: the
// large branches) and counted per chunk for the ordered compaction.
__global__ void __launch_bounds__(256, 5) k_br_place(const Field f, const uint64_t *__restrict__ W, uint32_t n,
                                                  uint32_t *cnt, const uint32_t *__restrict__ lbits, uint32_t *order,
                                                  uint32_t *pkey, uint32_t *mask0, uint32_t *mask1, uint32_t *counts0,
                                                  uint32_t *counts1, bool apart, BranchMeta *meta)
{
    __shared__ uint32_t sc[2], so[2], sa[2];
    if (threadIdx.x < 2) sc[threadIdx.x] = 0, so[threadIdx.x] = 0, sa[threadIdx.x] = ~0u;
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5, root = meta->root;
    constexpr uint32_t R = kChunkV / 256, RB = 2;
    const uint64_t b0 = (uint64_t)blockIdx.x * kChunkV + w * (R * 32);
    uint32_t c0 = 0, c1 = 0, o0 = 0, a0 = ~0u, o1 = 0, a1 = ~0u;
    bool bad = false;
    for (uint32_t q = 0; q < R; q += RB) {
        // each step for all rows before the next, so that their latencies overlap
        uint64_t T[RB];
        float fv[RB];
        uint32_t br[RB], lb[RB], pos[RB];
#pragma unroll
        for (uint32_t r = 0; r < RB; r++) {
            const uint64_t u = b0 + (q + r) * 32 + lane;
            T[r] = u < n ? W[u] : 0;
            fv[r] = u < n ? f[(uint32_t)u] : 0.0f;
        }
#pragma unroll
        for (uint32_t r = 0; r < RB; r++) {
            const uint64_t u = b0 + (q + r) * 32 + lane;
            br[r] = u < n ? branch_of(T[r], (uint32_t)u, n, bad) : 0u;
            lb[r] = lbits[br[r] >> 5];
        }
        uint32_t put = 0;  // bit r: this lane takes a place in row r
#pragma unroll
        for (uint32_t r = 0; r < RB; r++) {
            const uint64_t u64 = b0 + (q + r) * 32 + lane;
            const bool in = u64 < n;
            const uint32_t b = br[r], k = okey(fv[r]);
            const bool isroot = in && apart && b == root;
            const bool large = in && !isroot && ((lb[r] >> (b & 31)) & 1u);
            if (isroot) o0 |= k, a0 &= k;
            if (large) o1 |= k, a1 &= k;
            const bool place = in && !isroot && !large;
            put |= (uint32_t)place << r;
            uint32_t first;
            const uint32_t len = run_of(b, place, first);
            lb[r] = first;
            pos[r] = place && lane == first ? atomicAdd(cnt + b, len) : 0u;
            const uint32_t m0 = __ballot_sync(0xffffffffu, isroot), m1 = __ballot_sync(0xffffffffu, large);
            if (lane == 0 && in) mask0[u64 >> 5] = m0, mask1[u64 >> 5] = m1;
            c0 += __popc(m0), c1 += __popc(m1);
        }
#pragma unroll
        for (uint32_t r = 0; r < RB; r++) {
            const uint32_t p = __shfl_sync(0xffffffffu, pos[r], lb[r]) + lane - lb[r];
            if ((put >> r) & 1u) order[p] = (uint32_t)(b0 + (q + r) * 32 + lane), pkey[p] = okey(fv[r]);
        }
    }
    o0 = __reduce_or_sync(0xffffffffu, o0), a0 = __reduce_and_sync(0xffffffffu, a0);
    o1 = __reduce_or_sync(0xffffffffu, o1), a1 = __reduce_and_sync(0xffffffffu, a1);
    if (lane == 0) {
        atomicAdd(&sc[0], c0), atomicAdd(&sc[1], c1);
        atomicOr(&so[0], o0), atomicOr(&so[1], o1);
        atomicAnd(&sa[0], a0), atomicAnd(&sa[1], a1);
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        const uint32_t t = threadIdx.x;
        (t ? counts1 : counts0)[blockIdx.x] = sc[t];
        // most CTAs find the bits there already
        if (so[t] & ~*(volatile uint32_t *)&meta->kor[t]) atomicOr(&meta->kor[t], so[t]);
        if (*(volatile uint32_t *)&meta->kand[t] & ~sa[t]) atomicAnd(&meta->kand[t], sa[t]);
    }
}

// Sorts the small groups that start in this CTA's window of positions, in
// place: a member's place is the number of members before it in (key, id). A
// group's end is the next group's start; one with no end within kSmall
// positions is large and left alone.
__global__ void __launch_bounds__(256) k_br_small(uint32_t *order, const uint32_t *__restrict__ pkey,
                                                  const uint32_t *__restrict__ hbits, uint32_t n)
{
    constexpr uint32_t SPAN = kWindow + kSmall, WORDS = SPAN / 32 + 1;
    static_assert(kWindow % 32 == 0 && kSmall % 32 == 0 && WORDS <= 256, "whole words, one per thread");
    __shared__ uint64_t el[SPAN];           // (key, id)
    __shared__ uint32_t bits[WORDS];
    __shared__ uint16_t prev[WORDS], next[WORDS];  // last head in the words before, first head in the words after
    const uint64_t w0 = (uint64_t)blockIdx.x * kWindow;
    const uint32_t t = threadIdx.x;
    uint32_t mine = 0;
    if (t < WORDS) {
        const uint64_t wd = w0 / 32 + t;
        mine = wd <= (n - 1) / 32 ? hbits[wd] : 0u;
        if (wd == n / 32) mine |= 1u << (n & 31);  // the end of the last group
        bits[t] = mine;
    }
    if (!__syncthreads_or(t < kWindow / 32 && mine != 0)) return;
    constexpr uint32_t NO = 0xFFFFu;
    if (t < WORDS) {
        uint32_t q = NO;
        for (int j = (int)t - 1; j >= 0 && q == NO; j--)
            if (bits[j]) q = 32 * j + 31 - __clz(bits[j]);
        prev[t] = (uint16_t)q;
        q = NO;
        for (uint32_t j = t + 1; j < WORDS && q == NO; j++)
            if (bits[j]) q = 32 * j + __ffs(bits[j]) - 1;
        next[t] = (uint16_t)q;
    }
    __syncthreads();
    // start and end of the group of position p (relative to the window)
    auto group = [&](uint32_t p, uint32_t &s, uint32_t &e) -> bool {
        const uint32_t j = p >> 5, upto = bits[j] & (0xFFFFFFFFu >> (31 - (p & 31))), after = bits[j] & ~(0xFFFFFFFFu >> (31 - (p & 31)));
        s = upto ? 32 * j + 31 - __clz(upto) : prev[j];
        e = after ? 32 * j + __ffs(after) - 1 : next[j];
        return s < kWindow && e != NO && e - s <= kSmall && e - s > 1;  // (s == NO is above every position)
    };
    constexpr uint32_t PER = SPAN / 256;
    uint32_t s[PER], e[PER];
#pragma unroll
    for (uint32_t k = 0; k < PER; k++) {
        const uint32_t p = k * 256 + t;
        if (w0 + p >= n || !group(p, s[k], e[k])) e[k] = 0;
        else el[p] = (uint64_t)pkey[w0 + p] << 32 | order[w0 + p];
    }
    __syncthreads();
#pragma unroll
    for (uint32_t k = 0; k < PER; k++) {
        if (!e[k]) continue;
        const uint64_t x = el[k * 256 + t];
        uint32_t r = 0;
#pragma unroll 4
        for (uint32_t q = s[k]; q < e[k]; q++) r += el[q] < x;
        order[w0 + s[k] + r] = (uint32_t)x;
    }
}

// Ordered compaction of the marked vertices (two classes).
__global__ void __launch_bounds__(256) k_br_compact(const Field f, const uint32_t *__restrict__ mask0,
                                                    const uint32_t *__restrict__ mask1,
                                                    const uint32_t *__restrict__ starts0,
                                                    const uint32_t *__restrict__ starts1, uint32_t n, uint32_t *key0,
                                                    uint32_t *id0, uint32_t *key1, uint32_t *id1)
{
    __shared__ uint32_t wc[2][8];
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr uint32_t R = kChunkV / 256;
    const uint64_t b0 = (uint64_t)blockIdx.x * kChunkV + w * (R * 32);
    // lane r holds the masks of row r
    uint32_t m0 = 0, m1 = 0;
    if (lane < R && b0 + lane * 32 < n) m0 = mask0[b0 / 32 + lane], m1 = mask1[b0 / 32 + lane];
    const uint32_t c0 = __reduce_add_sync(0xffffffffu, __popc(m0)), c1 = __reduce_add_sync(0xffffffffu, __popc(m1));
    if (lane == 0) wc[0][w] = c0, wc[1][w] = c1;
    __syncthreads();
    if (c0 + c1 == 0) return;
    uint32_t r0 = starts0[blockIdx.x], r1 = starts1[blockIdx.x];
    for (uint32_t q = 0; q < w; q++) r0 += wc[0][q], r1 += wc[1][q];
    const uint32_t below = (1u << lane) - 1u;
    float fv[R];
#pragma unroll
    for (uint32_t r = 0; r < R; r++) {
        const uint32_t any = __shfl_sync(0xffffffffu, m0 | m1, r);
        fv[r] = (any >> lane) & 1u ? f[(uint32_t)(b0 + r * 32 + lane)] : 0.0f;
    }
#pragma unroll
    for (uint32_t r = 0; r < R; r++) {
        const uint32_t u = (uint32_t)(b0 + r * 32 + lane);
        const uint32_t q0 = __shfl_sync(0xffffffffu, m0, r), q1 = __shfl_sync(0xffffffffu, m1, r);
        const bool a = (q0 >> lane) & 1u, b = (q1 >> lane) & 1u;
        if (a || b) {
            const uint32_t k = okey(fv[r]);
            if (a) key0[r0 + __popc(q0 & below)] = k, id0[r0 + __popc(q0 & below)] = u;
            else key1[r1 + __popc(q1 & below)] = k, id1[r1 + __popc(q1 & below)] = u;
        }
        r0 += __popc(q0), r1 += __popc(q1);
    }
}

// key[i] = the large branch of vertex id[i]
__global__ void __launch_bounds__(256) k_br_rank(const uint64_t *__restrict__ W, uint32_t n,
                                                 const uint32_t *__restrict__ cnt, const uint32_t *__restrict__ id,
                                                 uint32_t m, uint32_t *key)
{
    bool bad = false;
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < m; i += (uint64_t)gridDim.x * 256) {
        const uint32_t u = id[i];
        key[i] = cnt[branch_of(W[u], u, n, bad)];
    }
}

// ------------------------------------------------------------- radix sort

// hist[d * nblocks + b] = keys of block b with digit d
template <uint32_t ROWS>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint32_t *__restrict__ keys, uint32_t n,
                                                             uint32_t shift, uint32_t nblocks,
                                                             uint32_t *__restrict__ hist)
{
    constexpr uint32_t C = 4;  // copies, so that fewer warps meet on a counter
    __shared__ uint32_t h[C][256];
    for (uint32_t i = threadIdx.x; i < C * 256; i += kSortThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    const uint64_t b0 = (uint64_t)blockIdx.x * (kSortThreads * ROWS);
    const uint32_t lane = threadIdx.x & 31;
    uint32_t *mine = h[(threadIdx.x >> 5) % C];
    uint32_t k[ROWS];
#pragma unroll
    for (uint32_t r = 0; r < ROWS; r++) {
        const uint64_t i = b0 + r * kSortThreads + threadIdx.x;
        k[r] = i < n ? keys[i] : 0u;
    }
#pragma unroll
    for (uint32_t r = 0; r < ROWS; r++) {
        const bool in = b0 + r * kSortThreads + threadIdx.x < n;
        const uint32_t d = (k[r] >> shift) & 255u;
        // a row of one digit, as high digits often are, takes one atomic
        const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0), bal = __ballot_sync(0xffffffffu, in && d == d0);
        if (bal == 0xffffffffu) {
            if (lane == 0) atomicAdd(mine + d, 32u);
        } else if (in) {
            atomicAdd(mine + d, 1u);
        }
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        uint32_t t = 0;
        for (uint32_t c = 0; c < C; c++) t += h[c][threadIdx.x];
        hist[(uint64_t)threadIdx.x * nblocks + blockIdx.x] = t;
    }
}

// CTA d: the exclusive scan over the blocks of digit d's counts, in place, and
// their total.
__global__ void __launch_bounds__(512) k_radix_scan(uint32_t *hist, uint32_t nblocks, uint32_t *total)
{
    __shared__ uint32_t part[16], s_carry;
    uint32_t *a = hist + (uint64_t)blockIdx.x * nblocks;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr uint32_t PER = 8;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (uint64_t b0 = 0; b0 < nblocks; b0 += 512 * PER) {
        // a warp owns a contiguous range, read in rows of 32
        uint32_t v[PER], s = 0;
        const uint64_t w0 = b0 + (uint64_t)w * (32 * PER);
#pragma unroll
        for (uint32_t r = 0; r < PER; r++) {
            const uint64_t i = w0 + r * 32 + lane;
            v[r] = i < nblocks ? a[i] : 0u;
            s += v[r];
        }
        s = __reduce_add_sync(0xffffffffu, s);
        if (lane == 0) part[w] = s;
        __syncthreads();
        uint32_t run = s_carry;
        for (uint32_t q = 0; q < w; q++) run += part[q];
#pragma unroll
        for (uint32_t r = 0; r < PER; r++) {
            const uint64_t i = w0 + r * 32 + lane;
            uint32_t incl = v[r];
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= (uint32_t)o) incl += y;
            }
            if (i < nblocks) a[i] = run + incl - v[r];
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        __syncthreads();
        if (threadIdx.x == 511) s_carry = run;
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = s_carry;
}

// Stable scatter of block b's keys and values to the scanned offsets (the digit
// starts are scanned from the totals by every block itself). Warp w owns keys [w * 512, (w + 1) * 512) of the block, read in kSortRows rounds of
// 32; a key's place within the block's run of its digit is the number of keys
// with that digit in earlier warps, in earlier rounds of its warp and on lower
// lanes of its round (the lanes with its digit find each other by setting their
// bits in a word per digit: 0.53 ms for 98 M keys, 0.72 with eight ballots).
// The keys are first placed in shared memory in that
// order (digit by digit), then written out in order, so that consecutive
// threads write consecutive addresses of a digit's run (32 keys long on
// average). LAST: the keys are not needed any more and stay where they are.
// With lstart the keys are branch numbers and this pass ends the sort: the
// value at place i of branch k goes to lstart[k] + i - lbase[k].
// Shared memory: the keys and values of the block (where the values go later
// are the lane words, 256 per warp, at first), counts, digit starts.
template <uint32_t ROWS>
struct ScatterShape {
    static constexpr uint32_t kBlock = kSortThreads * ROWS;
    static constexpr uint32_t kVals = kBlock > kSortWarps * 256 ? kBlock : kSortWarps * 256;
    static constexpr size_t kSmem = ((size_t)kBlock + kVals) * 4 + (size_t)kSortWarps * 256 * 2 + 512 * 4;
};

template <bool LAST, uint32_t ROWS>
__global__ void __launch_bounds__(kSortThreads, 2) k_radix_scatter(const uint32_t *__restrict__ kin,
                                                                   const uint32_t *__restrict__ vin, uint32_t *kout,
                                                                   uint32_t *vout, uint32_t n, uint32_t shift,
                                                                   uint32_t nblocks, const uint32_t *__restrict__ offs,
                                                                   const uint32_t *__restrict__ total,
                                                                   const uint32_t *__restrict__ lstart,
                                                                   const uint32_t *__restrict__ lbase)
{
    extern __shared__ __align__(16) uint32_t sort_smem[];
    using SS = ScatterShape<ROWS>;
    uint32_t *skey = sort_smem, *sval = skey + SS::kBlock;
    uint32_t *base = sval + SS::kVals;             // 256: where the block's run of each digit goes
    uint32_t *lst = base + 256;                    // 256: where it starts in shared memory
    uint16_t (*cnt)[256] = reinterpret_cast<uint16_t(*)[256]>(lst + 256);  // per warp: counts, then running places
    __shared__ uint32_t wtot[8], wall[8];
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    volatile uint32_t *bits = sval + w * 256;      // this warp's lanes by digit, before the values are placed
    for (uint32_t i = threadIdx.x; i < kSortWarps * 128; i += kSortThreads) reinterpret_cast<uint32_t *>(cnt)[i] = 0;
    for (uint32_t i = lane; i < 256; i += 32) bits[i] = 0;
    uint32_t dbase = 0;                            // thread = digit: keys with lower digits
    if (threadIdx.x < 256) {
        const uint32_t c = total[threadIdx.x];
        uint32_t incl = c;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        if (lane == 31) wall[w] = incl;
        dbase = incl - c + offs[(uint64_t)threadIdx.x * nblocks + blockIdx.x];
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        for (uint32_t q = 0; q < w; q++) dbase += wall[q];
        base[threadIdx.x] = dbase;
    }
    const uint64_t blk0 = (uint64_t)blockIdx.x * SS::kBlock, b0 = blk0 + (uint64_t)w * (ROWS * 32);
    uint32_t k[ROWS];
    uint32_t place[ROWS / 2];                 // ranks among the warp's keys of the digit, two rows in one
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (uint32_t r = 0; r < ROWS; r++) {
        const uint64_t i = b0 + r * 32 + lane;
        k[r] = i < n ? kin[i] : ~0u;
    }
    volatile uint16_t *vc = cnt[w];
#pragma unroll
    for (uint32_t r = 0; r < ROWS; r++) {
        const bool in = b0 + r * 32 + lane < n;
        const uint32_t d = (k[r] >> shift) & 255u;
        if (in) atomicOr(const_cast<uint32_t *>(bits) + d, 1u << lane);
        __syncwarp();
        const uint32_t p = bits[d], c = vc[d], q = c + __popc(p & lt);
        __syncwarp();
        place[r / 2] = r & 1 ? place[r / 2] | q << 16 : q;
        if (in && (p & lt) == 0) bits[d] = 0, vc[d] = (uint16_t)(c + __popc(p));  // the digit's first lane
        __syncwarp();
    }
    __syncthreads();
    // thread = digit: the block's count of the digit, its local start
    // (exclusive scan over digits), and the places where the warps begin
    uint32_t tot = 0, incl = 0;
    if (threadIdx.x < 256) {
        const uint32_t d = threadIdx.x;
#pragma unroll
        for (uint32_t q = 0; q < kSortWarps; q++) tot += cnt[q][d];
        incl = tot;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        if (lane == 31) wtot[w] = incl;
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        const uint32_t d = threadIdx.x;
        uint32_t run = incl - tot;
        for (uint32_t q = 0; q < w; q++) run += wtot[q];
        lst[d] = run;
#pragma unroll
        for (uint32_t q = 0; q < kSortWarps; q++) {
            const uint32_t c = cnt[q][d];
            cnt[q][d] = (uint16_t)run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (uint32_t r = 0; r < ROWS; r++) {
        if (b0 + r * 32 + lane < n) {
            const uint32_t pos = cnt[w][(k[r] >> shift) & 255u] + (place[r / 2] >> (16 * (r & 1)) & 0xFFFFu);
            skey[pos] = k[r];
            sval[pos] = vin[b0 + r * 32 + lane];
        }
    }
    __syncthreads();
    const uint32_t valid = n - blk0 < SS::kBlock ? (uint32_t)(n - blk0) : SS::kBlock;
    for (uint32_t j = threadIdx.x; j < valid; j += kSortThreads) {
        const uint32_t key = skey[j], d = (key >> shift) & 255u;
        uint32_t pos = base[d] + (j - lst[d]);
        if (!LAST) kout[pos] = key;
        else if (lstart) pos = lstart[key] + (pos - lbase[key]);
        vout[pos] = sval[j];
    }
}

// Workspace of the branch decomposition: the common part, then the counts per
// branch id, the arrays of the sorts (16 bytes per vertex), masks and flags (a
// bit per vertex each), the digit histograms and scan sums, the table of
// large branches and the counters.
struct BranchWs {
    uint32_t *cnt, *pool, *mask0, *mask1, *hbits, *lbits, *hmask, *heads, *sizes, *hist, *total, *lstart, *lsize;
    BranchMeta *meta;
    size_t zero_bytes;                             // from hbits on: cleared before use
};

static size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

static size_t branch_ws(uint64_t n, BranchWs *bw, char *base)
{
    const uint64_t few = n < kSortFew ? n : kSortFew, nchunks = (n + kChunkV - 1) / kChunkV;
    const uint64_t nb0 = (n + kSortThreads * kSortRows - 1) / (kSortThreads * kSortRows);
    const uint64_t nb1 = (few + kSortThreads * kSortRowsFew - 1) / (kSortThreads * kSortRowsFew);
    const uint64_t nhist = 256 * (nb0 > nb1 ? nb0 : nb1), nlarge = n / (kSmall + 1) + 1;
    size_t off = a256(workspace_bytes(n));
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off += a256(bytes);
        return base ? reinterpret_cast<uint32_t *>(base + o) : nullptr;
    };
    BranchWs b;
    b.pool = take(16 * n + 4096);
    b.mask0 = take(n / 8 + 8);
    b.mask1 = take(n / 8 + 8);
    b.hmask = b.mask1;  // done with when mask1 is written
    b.heads = take(nchunks * 4);
    b.sizes = take(nchunks * 4);
    b.hist = take(nhist * 4);
    b.total = take(256 * 4);
    b.lstart = take(nlarge * 4);
    b.lsize = take(nlarge * 4);
    b.meta = reinterpret_cast<BranchMeta *>(take(sizeof(BranchMeta)));
    const size_t z0 = off;
    b.hbits = take(n / 8 + 8);
    b.lbits = take(n / 8 + 8);
    b.cnt = take(n * 4);
    b.zero_bytes = off - z0;
    if (bw) *bw = b;
    return off;
}

// One pass by the digit at `shift`.
template <bool LAST, uint32_t ROWS>
static cudaError_t radix_pass_rows(const uint32_t *kin, const uint32_t *vin, uint32_t *kout, uint32_t *vout, uint32_t m,
                                   uint32_t shift, const BranchWs &bw, cudaStream_t st, const uint32_t *lstart,
                                   const uint32_t *lbase)
{
    using SS = ScatterShape<ROWS>;
    static AttrFlags flags;  // per instantiation
    int dev;
    if (flags.pending(dev)) {
        const cudaError_t e = cudaFuncSetAttribute(k_radix_scatter<LAST, ROWS>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SS::kSmem);
        if (e != cudaSuccess) return e;
        flags.done(dev);
    }
    const uint32_t nb = (uint32_t)(((uint64_t)m + SS::kBlock - 1) / SS::kBlock);
    k_radix_hist<ROWS><<<nb, kSortThreads, 0, st>>>(kin, m, shift, nb, bw.hist);
    k_radix_scan<<<256, 512, 0, st>>>(bw.hist, nb, bw.total);
    k_radix_scatter<LAST, ROWS><<<nb, kSortThreads, SS::kSmem, st>>>(kin, vin, kout, vout, m, shift, nb, bw.hist,
                                                                     bw.total, lstart, lbase);
    count_launch(3);
    return cudaGetLastError();
}

template <bool LAST>
static cudaError_t radix_pass(const uint32_t *kin, const uint32_t *vin, uint32_t *kout, uint32_t *vout, uint32_t m,
                              uint32_t shift, const BranchWs &bw, cudaStream_t st, const uint32_t *lstart = nullptr,
                              const uint32_t *lbase = nullptr)
{
    return m <= kSortFew
               ? radix_pass_rows<LAST, kSortRowsFew>(kin, vin, kout, vout, m, shift, bw, st, lstart, lbase)
               : radix_pass_rows<LAST, kSortRows>(kin, vin, kout, vout, m, shift, bw, st, lstart, lbase);
}

// The shifts of the 8-bit digits in which the keys differ.
static int digits(uint32_t vary, uint32_t shift[4])
{
    int k = 0;
    for (uint32_t s = 0; s < 32; s += 8)
        if ((vary >> s) & 255u) shift[k++] = s;
    return k;
}

}  // namespace mt

using namespace mt;

extern "C" {

size_t mt_branches_workspace_bytes(mt_grid g)
{
    const uint64_t n = (uint64_t)g.nx * g.ny * g.nz;
    if (!g.nx || !g.ny || !g.nz || n >= 0xFFFFFFFFull) return 0;
    return branch_ws(n, nullptr, nullptr);
}

mt_status mt_branch_decomposition(const float *d_f, const uint64_t *d_W, mt_grid g, uint32_t flags, uint32_t *d_order,
                                  uint32_t *d_offsets, uint64_t offsets_cap, uint64_t *h_nbranches, void *d_ws,
                                  size_t ws_bytes, void *stream)
{
    const uint64_t n64 = (uint64_t)g.nx * g.ny * g.nz;
    if (!g.nx || !g.ny || !g.nz) return MT_ERR_INVALID;
    if (n64 >= 0xFFFFFFFFull) return MT_ERR_TOO_LARGE;
    if (!d_f || !d_W || !d_order || !h_nbranches || (offsets_cap && !d_offsets) || ((uintptr_t)d_f & 3) ||
        ((uintptr_t)d_W & 7) || ((uintptr_t)d_order & 3) || ((uintptr_t)d_offsets & 3) || (flags & ~MT_SUPERLEVEL))
        return MT_ERR_INVALID;
    Workspace ws;
    if (ws_bytes < branch_ws(n64, nullptr, nullptr) || !carve_workspace(d_ws, ws_bytes, n64, ws)) return MT_ERR_INVALID;
    BranchWs bw;
    branch_ws(n64, &bw, static_cast<char *>(d_ws));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint32_t n = (uint32_t)n64;
    const Field f{d_f, (flags & MT_SUPERLEVEL) ? -1.0f : 1.0f};
    const bool apart = n64 > kTogether;
    const uint32_t nchunks = (uint32_t)((n64 + kChunkV - 1) / kChunkV);
    PhaseScope ps(kBranches, st);
    if (cudaMemsetAsync(bw.hbits, 0, bw.zero_bytes, st) != cudaSuccess) return MT_ERR_CUDA;
    k_br_root<<<1, 1, 0, st>>>(d_W, n, bw.meta);
    const uint32_t per = n64 <= kTogether ? kCountVFew : kCountV;
    k_br_count<<<(unsigned)((n64 + per - 1) / per), 256, 0, st>>>(d_W, n, per, bw.cnt, bw.hmask, bw.meta, ws.status);
    k_br_sums<<<nchunks, 256, 0, st>>>(bw.cnt, bw.hmask, n, bw.heads, bw.sizes);
    k_br_scan2<<<2, 1024, 0, st>>>(bw.heads, bw.sizes, nchunks, &bw.meta->nbranch, nullptr);
    k_br_starts<<<nchunks, 256, 0, st>>>(bw.cnt, bw.hmask, n, bw.heads, bw.sizes, d_offsets, offsets_cap, bw.hbits,
                                         bw.lbits, bw.lstart, bw.lsize, apart, bw.meta);
    k_br_place<<<nchunks, 256, 0, st>>>(f, d_W, n, bw.cnt, bw.lbits, d_order, bw.pool, bw.mask0, bw.mask1, bw.heads,
                                        bw.sizes, apart, bw.meta);
    k_br_scan2<<<2, 1024, 0, st>>>(bw.heads, bw.sizes, nchunks, &bw.meta->nl[0], &bw.meta->nl[1]);
    k_br_small<<<(unsigned)((n64 + kWindow - 1) / kWindow), 256, 0, st>>>(d_order, bw.pool, bw.hbits, n);
    count_launch(8);
    if (cudaGetLastError() != cudaSuccess) return MT_ERR_CUDA;
    BranchMeta m;
    uint32_t bits = 0;
    if (cudaMemcpyAsync(&m, bw.meta, sizeof(m), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(&bits, ws.status, sizeof(bits), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return MT_ERR_CUDA;
    if (bits) return status_from_bits(bits);
    const uint64_t n0 = m.nl[0], n1 = m.nl[1];
    // arrays of the sorts, carved from the pool (at most 16 bytes per vertex;
    // 64 words of slack for alignment). The root's branch, and a single large
    // one, keep their ids in their own place in d_order every other pass, so
    // that they end there.
    uint32_t *p = bw.pool;
    auto carve = [&](uint64_t words) {
        uint32_t *q = p;
        p += (words + 31) & ~31ull;
        return q;
    };
    const bool one = m.nlarge == 1;
    uint32_t *ka = carve(n0), *kb = carve(n0), *ia = carve(n0), *ib = d_order + m.rstart;
    uint32_t *ka1 = carve(n1), *kb1 = carve(n1), *ia1 = carve(n1), *ib1 = one ? d_order + m.lstart0 : carve(n1);
    uint32_t sh0[4], sh1[4];
    const int p0 = n0 ? digits(m.kor[0] ^ m.kand[0], sh0) : 0, p1 = n1 ? digits(m.kor[1] ^ m.kand[1], sh1) : 0;
    auto swap = [](uint32_t *&a, uint32_t *&b) {
        uint32_t *t = a;
        a = b, b = t;
    };
    if (p0 % 2 == 0) swap(ka, kb), swap(ia, ib);  // an even number of passes starts in place
    if (one && p1 % 2 == 0) swap(ka1, kb1), swap(ia1, ib1);
    if (n0 + n1) {
        k_br_compact<<<nchunks, 256, 0, st>>>(f, bw.mask0, bw.mask1, bw.heads, bw.sizes, n, ka, ia, ka1, ia1);
        count_launch();
    }
    cudaError_t e = cudaGetLastError();
    for (int i = 0; i < p0 && e == cudaSuccess; i++) {
        e = i + 1 < p0 ? radix_pass<false>(ka, ia, kb, ib, (uint32_t)n0, sh0[i], bw, st)
                       : radix_pass<true>(ka, ia, kb, ib, (uint32_t)n0, sh0[i], bw, st);
        swap(ka, kb), swap(ia, ib);
    }
    for (int i = 0; i < p1 && e == cudaSuccess; i++) {
        e = i + 1 < p1 ? radix_pass<false>(ka1, ia1, kb1, ib1, (uint32_t)n1, sh1[i], bw, st)
                       : radix_pass<true>(ka1, ia1, kb1, ib1, (uint32_t)n1, sh1[i], bw, st);
        swap(ka1, kb1), swap(ia1, ib1);
    }
    if (m.nlarge > 1 && e == cudaSuccess) {
        // then by branch: the keys become branch numbers; lsize becomes the
        // first place of each branch in the sorted array
        const uint64_t wantr = (n1 + 255) / 256, mostr = (uint64_t)device_sms() * 8;
        k_br_rank<<<(unsigned)(wantr < mostr ? wantr : mostr), 256, 0, st>>>(d_W, n, bw.cnt, ia1, (uint32_t)n1, ka1);
        k_br_scan2<<<1, 1024, 0, st>>>(bw.lsize, bw.lsize, m.nlarge, nullptr, nullptr);
        count_launch(2);
        e = cudaGetLastError();
        uint32_t last = 0;  // the highest digit of the branch numbers
        while (last < 24 && ((m.nlarge - 1) >> (last + 8))) last += 8;
        for (uint32_t s = 0; s <= last && e == cudaSuccess; s += 8) {
            e = s < last ? radix_pass<false>(ka1, ia1, kb1, ib1, (uint32_t)n1, s, bw, st)
                         : radix_pass<true>(ka1, ia1, kb1, d_order, (uint32_t)n1, s, bw, st, bw.lstart, bw.lsize);
            swap(ka1, kb1), swap(ia1, ib1);
        }
    }
    if (e != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return MT_ERR_CUDA;
    *h_nbranches = m.nbranch;
    return (uint64_t)m.nbranch + 1 > offsets_cap ? MT_ERR_CAPACITY : MT_OK;
}

}  // extern "C"
