// Queries on a finished triplet merge tree:
//   k_pairs_count / k_scan_counts / k_pairs_write
//       0-dimensional persistence pairs (minimum u, saddle s) for every u with
//       W[u].s != u, in ascending u (ordered stream compaction);
//   k_labels
//       representatives at a threshold t (components of G_t).
#include <cuda_runtime.h>

#include "mt_device.cuh"
#include "mt_fields.cuh"
#include "mt_internal.h"

namespace mt {

// ------------------------------------------------------------------ pairs
//
// One CTA per chunk of kCompactChunk consecutive vertices of a field; warp w
// owns the contiguous slice [w * 512, (w + 1) * 512) of the chunk and reads it
// in 16 coalesced rows of 32. A pass counts the pairs of each chunk (and finds
// the roots), a scan per field turns the counts into offsets, and a second
// pass writes each chunk's pairs at its offset in order: every warp ranks its
// flags with ballots, and one barrier combines the 8 warp totals, which keeps
// the ascending order.
//
// Both passes are bound by HBM, so the first one leaves a bit per vertex
// (`mask`, 1/64 of the triplets' size, where the caller has the room) and the
// second reads the triplets of pairs only, one vertex in ten on a lognormal
// field: 2.8 -> 2.7 ms at 1024^3, 68 -> 61 us at 256^3. With a persistence to
// keep (eps > 0) it also saves reading f at the saddles a second time, and
// those reads are issued for eight rows at a time: 585 -> 256 us at 400^3. A
// batch's fields mostly stay in L2 between the passes, where the bits cost
// more than they save (512 uneven fields: 345 us with them, 325 without).
constexpr int kCompactThreads = 256;
constexpr int kCompactWarps = kCompactThreads / 32;
constexpr int kCompactRows = kCompactChunk / kCompactThreads;  // rows of 32 per warp
static_assert(kCompactRows * 32 * kCompactWarps == kCompactChunk, "chunk = warps x rows x 32");
static_assert(kCompactRows <= 32, "a lane per row holds the row's mask");

// Which of the vertices u0 + 32 r + lane with triplets T[r] begin a pair: bit
// r of the result. Persistence simplification (SIMP): the pair (u, s) of a
// branch minimum u is kept when its persistence f(s) - f(u), computed in
// float32 on the values the order sees (sg * f), is at least eps; the values
// of a few rows are read together, without a branch between them. Without SIMP
// every pair is kept and f is not read.
template <bool SIMP>
__device__ __forceinline__ uint32_t keep_rows(const FieldDesc &fd, const uint64_t *T, uint64_t u0, float eps)
{
    const uint32_t lane = threadIdx.x & 31;
    uint32_t keep = 0;
    constexpr int RB = SIMP ? 8 : kCompactRows;
#pragma unroll
    for (int q = 0; q < kCompactRows; q += RB) {
        float fu[RB], fs[RB];
        if (SIMP) {
#pragma unroll
            for (int r = 0; r < RB; r++) {
                const uint32_t u = (uint32_t)(u0 + (q + r) * 32 + lane), s = tri_s(T[q + r]);
                fu[r] = s != u ? __ldg(fd.f + u) : 0.0f;
                fs[r] = s != u ? __ldg(fd.f + s) : 0.0f;
            }
        }
#pragma unroll
        for (int r = 0; r < RB; r++) {
            const uint32_t u = (uint32_t)(u0 + (q + r) * 32 + lane);
            bool k = tri_s(T[q + r]) != u;
            if (SIMP) k = k && fd.sg * fs[r] - fd.sg * fu[r] >= eps;
            keep |= (uint32_t)k << (q + r);
        }
    }
    return keep;
}

template <class Loc, bool SIMP>
__global__ void __launch_bounds__(kCompactThreads, std::is_same<Loc, OneField>::value ? 4 : 3) k_pairs_count(Loc loc, uint32_t *counts, uint32_t *mask, float eps,
                                                                 const uint32_t *status)
{
    if (block_skips(status)) return;
    __shared__ uint32_t warp_sum[kCompactWarps];
    uint64_t local;
    uint32_t fi;
    const FieldDesc fd = loc.chunk(blockIdx.x, local, fi);
    const uint64_t *__restrict__ W = fd.W;
    const uint64_t n = fd.n;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t b0 = local * kCompactChunk + (uint64_t)warp * (kCompactRows * 32);
    // all rows are loaded before any is used, so that their loads overlap
    uint64_t Tr[kCompactRows];
#pragma unroll
    for (int r = 0; r < kCompactRows; r++) {
        const uint64_t u = b0 + (uint64_t)r * 32 + lane;
        Tr[r] = u < n ? W[u] : (uint64_t)(uint32_t)u << 32 | (uint32_t)~u;  // past the end: neither pair nor root
    }
    const uint32_t keep = keep_rows<SIMP>(fd, Tr, b0, eps);
    uint32_t mine = 0;
#pragma unroll
    for (int r = 0; r < kCompactRows; r++) {
        const uint32_t u = (uint32_t)(b0 + (uint64_t)r * 32 + lane);
        if (Tr[r] == tri_pack(u, u)) {
            atomicAdd(reinterpret_cast<unsigned long long *>(fd.meta + 1), 1ull);
            fd.meta[2] = u;
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, (keep >> r) & 1u);
        mine = lane == (uint32_t)r ? bal : mine;
    }
    if (mask && lane < (uint32_t)kCompactRows)
        mask[(uint64_t)blockIdx.x * (kCompactChunk / 32) + warp * kCompactRows + lane] = mine;
    const uint32_t c = __reduce_add_sync(0xffffffffu, __popc(mine));
    if (lane == 0) warp_sum[warp] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t tot = 0;
        for (int w = 0; w < kCompactWarps; w++) tot += warp_sum[w];
        counts[blockIdx.x] = tot;
    }
}

// Counts of the chunks whose bits the build has left (a warp per chunk); the
// bits past the field's end are cleared.
__global__ void __launch_bounds__(kCompactThreads) k_mask_count(uint32_t *mask, uint64_t n, uint64_t nchunks,
                                                                uint32_t *counts, const uint32_t *status)
{
    if (block_skips(status)) return;
    const uint64_t c = (uint64_t)blockIdx.x * kCompactWarps + (threadIdx.x >> 5);
    if (c >= nchunks) return;
    const uint32_t lane = threadIdx.x & 31;
    uint32_t *m = mask + c * (kCompactChunk / 32), sum = 0;
#pragma unroll
    for (uint32_t k = 0; k < kCompactChunk / 32; k += 32) {
        const uint64_t u = c * kCompactChunk + (k + lane) * 32;  // the word's first vertex
        uint32_t w = 0;
        if (u < n) w = m[k + lane];
        if (u + 32 > n) {
            if (u < n) w &= (1u << (n - u)) - 1u;
            m[k + lane] = w;
        }
        sum += __popc(w);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) counts[c] = sum;
}

// Exclusive scan of one field's chunk counts in place (one CTA of 1024
// threads per field); the field's total goes to its meta[0] and, in a batch,
// to npairs[field]. Warp w owns a contiguous range of chunks and reads it in
// coalesced rows of 32: a first pass sums the range, one warp scans the 32
// sums, and a second pass scans each row with shuffles on top of the carry.
template <class Loc>
__global__ void __launch_bounds__(1024) k_scan_counts(Loc loc, uint32_t *counts, uint64_t *npairs,
                                                      const uint32_t *status)
{
    if (block_skips(status)) return;
    __shared__ uint64_t wsum[32];
    const FieldDesc fd = loc.field(blockIdx.x);
    uint32_t *cnt = counts + fd.chunk0;
    const uint64_t m = (fd.n + kCompactChunk - 1) / kCompactChunk;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t per = ((m + 31) / 32 + 31) / 32 * 32;  // chunks per warp, whole rows
    const uint64_t a = warp * per, b = a + per < m ? a + per : m;
    uint64_t s = 0;
    for (uint64_t i = a + lane; i < b; i += 32) s += cnt[i];
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
        wsum[lane] = incl - v;  // exclusive
        if (lane == 31) {
            fd.meta[0] = incl;
            if (npairs) npairs[blockIdx.x] = incl;
        }
    }
    __syncthreads();
    uint64_t carry = wsum[warp];
    for (uint64_t r = a; r < b; r += 32) {
        const uint64_t i = r + lane;
        const uint32_t c = i < b ? cnt[i] : 0u;
        uint32_t incl = c;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        if (i < b) cnt[i] = (uint32_t)(carry + incl - c);
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
}

// SUM: `offsets` still holds the chunks' counts, and every CTA adds up those
// before its own. For a single field of up to kSumChunks chunks that costs less
// than the scan's launch. The last CTA of a single field also leaves the
// counters and the status word at `out` (mapped host memory, or null).
constexpr uint64_t kSumChunks = 4096;

template <class Loc, bool SIMP, bool MASK, bool SUM>
__global__ void __launch_bounds__(kCompactThreads) k_pairs_write(Loc loc, const uint32_t *offsets,
                                                                 const uint32_t *__restrict__ mask, float eps,
                                                                 const uint32_t *status, volatile uint64_t *out)
{
    if (block_skips(status)) {
        if (out && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[3] = *status;
        return;
    }
    __shared__ uint32_t warp_cnt[kCompactWarps], warp_sum[kCompactWarps];
    uint64_t local;
    uint32_t fi;
    const FieldDesc fd = loc.chunk(blockIdx.x, local, fi);
    const uint64_t *__restrict__ W = fd.W;
    const uint64_t n = fd.n, cap = fd.cap;
    uint32_t *pairs = fd.pairs;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t b0 = local * kCompactChunk + (uint64_t)warp * (kCompactRows * 32);
    uint64_t Tr[kCompactRows];
    uint32_t mine = 0;  // lane r: the flags of row r
    if (MASK) {
        if (lane < (uint32_t)kCompactRows)
            mine = mask[(uint64_t)blockIdx.x * (kCompactChunk / 32) + warp * kCompactRows + lane];
    } else {
#pragma unroll
        for (int r = 0; r < kCompactRows; r++) {
            const uint64_t u = b0 + (uint64_t)r * 32 + lane;
            Tr[r] = u < n ? W[u] : tri_pack((uint32_t)u, (uint32_t)u);  // past the end: no pair
        }
        const uint32_t keep = keep_rows<SIMP>(fd, Tr, b0, eps);
#pragma unroll
        for (int r = 0; r < kCompactRows; r++) {
            const uint32_t bal = __ballot_sync(0xffffffffu, (keep >> r) & 1u);
            mine = lane == (uint32_t)r ? bal : mine;
        }
    }
    const uint32_t c = __reduce_add_sync(0xffffffffu, __popc(mine));
    if (lane == 0) warp_cnt[warp] = c;
    if (MASK) {
#pragma unroll
        for (int r = 0; r < kCompactRows; r++) {
            const uint32_t q = __shfl_sync(0xffffffffu, mine, r);
            Tr[r] = (q >> lane) & 1u ? W[b0 + (uint64_t)r * 32 + lane] : 0;
        }
    }
    if (SUM) {
        uint32_t s = 0;
        for (uint32_t i = threadIdx.x; i < blockIdx.x; i += kCompactThreads) s += offsets[i];
        s = __reduce_add_sync(0xffffffffu, s);
        if (lane == 0) warp_sum[warp] = s;
    }
    __syncthreads();
    uint64_t run = SUM ? 0 : offsets[blockIdx.x];
    if (SUM)
        for (int w = 0; w < kCompactWarps; w++) run += warp_sum[w];
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0 && (SUM || out)) {
        uint64_t total = run;
        for (int w = 0; w < kCompactWarps; w++) total += warp_cnt[w];
        if (SUM) fd.meta[0] = total;
        if (out) out[0] = total, out[1] = fd.meta[1], out[2] = fd.meta[2], out[3] = *status;
    }
    for (uint32_t w = 0; w < warp; w++) run += warp_cnt[w];
    const uint32_t below = (1u << lane) - 1u;
    const bool wide = ((uintptr_t)pairs & 7) == 0;  // the list is only 4-byte aligned
#pragma unroll
    for (int r = 0; r < kCompactRows; r++) {
        const uint32_t u = (uint32_t)(b0 + (uint64_t)r * 32 + lane);
        const uint32_t q = __shfl_sync(0xffffffffu, mine, r);
        if ((q >> lane) & 1u) {
            const uint64_t pos = run + __popc(q & below);
            if (pos < cap) {
                if (wide) {
                    reinterpret_cast<uint2 *>(pairs)[pos] = make_uint2(u, tri_s(Tr[r]));
                } else {
                    pairs[2 * pos] = u;
                    pairs[2 * pos + 1] = tri_s(Tr[r]);
                }
            }
        }
        run += __popc(q);
    }
}

template <class Loc>
static cudaError_t run_pairs(const Loc &loc, uint32_t nfields, uint64_t nchunks, uint32_t *counts, uint32_t *mask,
                             uint64_t *npairs, const uint32_t *status, cudaStream_t st, float eps = 0.0f,
                             uint64_t *out = nullptr, uint64_t marked = 0)
{
    PhaseScope ps(kPairs, st);
    const unsigned grid = (unsigned)nchunks;
    constexpr bool ONE = std::is_same<Loc, OneField>::value;  // a batch has no eps, bits or mapped counters
    bool simp = false;
    if constexpr (ONE) {
        simp = eps > 0.0f;
        if (marked)  // the number of vertices
            k_mask_count<<<(unsigned)((nchunks + kCompactWarps - 1) / kCompactWarps), kCompactThreads, 0, st>>>(
                mask, marked, nchunks, counts, status);
        else if (simp) k_pairs_count<Loc, true><<<grid, kCompactThreads, 0, st>>>(loc, counts, mask, eps, status);
    }
    if (!marked && !simp) k_pairs_count<Loc, false><<<grid, kCompactThreads, 0, st>>>(loc, counts, mask, eps, status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if constexpr (ONE) {
        if (mask && nchunks <= kSumChunks) {
            k_pairs_write<Loc, false, true, true><<<grid, kCompactThreads, 0, st>>>(loc, counts, mask, eps, status, out);
            count_launch(2);
            return cudaGetLastError();
        }
    }
    k_scan_counts<Loc><<<nfields, 1024, 0, st>>>(loc, counts, npairs, status);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if constexpr (ONE) {
        if (mask)
            k_pairs_write<Loc, false, true, false><<<grid, kCompactThreads, 0, st>>>(loc, counts, mask, eps, status, out);
        else if (simp)
            k_pairs_write<Loc, true, false, false><<<grid, kCompactThreads, 0, st>>>(loc, counts, mask, eps, status, out);
    }
    if (!mask && !simp)
        k_pairs_write<Loc, false, false, false><<<grid, kCompactThreads, 0, st>>>(loc, counts, mask, eps, status, out);
    count_launch(3);
    return cudaGetLastError();
}

cudaError_t launch_pairs(const uint64_t *W, uint64_t n, uint32_t *pairs, uint64_t cap, Workspace &ws,
                         cudaStream_t st, const float *f, float sg, float eps, uint64_t *out, bool clear, bool marked)
{
    if (clear) {
        const cudaError_t e = cudaMemsetAsync(ws.meta, 0, 3 * sizeof(uint64_t), st);
        if (e != cudaSuccess) return e;
    }
    OneField loc;
    loc.d = FieldDesc{};
    loc.d.W = const_cast<uint64_t *>(W);
    loc.d.pairs = pairs;
    loc.d.meta = ws.meta;
    loc.d.n = n;
    loc.d.cap = cap;
    loc.d.f = f;
    loc.d.sg = sg;
    return run_pairs(loc, 1, ws.nchunks, ws.counts, ws.mask, nullptr, ws.status, st, eps, out, marked ? n : 0);
}

cudaError_t launch_batch_pairs(const FieldDesc *d_descs, uint32_t nfields, uint64_t nchunks, uint32_t *counts,
                               uint64_t *npairs, const uint32_t *status, cudaStream_t st)
{
    ManyFields loc{d_descs, nfields};
    return run_pairs(loc, nfields, nchunks, counts, nullptr, npairs, status, st);
}

// ----------------------------------------------------------------- labels
//
// Components of G_t = {u : f[u] <= t} (Section 2.1): the label of u is its
// representative at level t (Algorithm 4 with the value test f(s) <= t that
// the paper's Representative uses), the deepest vertex of u's component, or
// 0xFFFFFFFF when f[u] > t. An inner vertex u with f[u] <= t hops to its
// deepest vertex v first (its link's saddle is u itself); the chain of branch
// links is then followed while their saddles lie in G_t.
//
// One CTA per brick of 32 x 16 x 16 vertices, in three steps: every vertex in
// G_t enters the start of its chain (its target v, or u itself for a minimum
// or a root) in a shared-memory hash and keeps the slot; the chain of every
// hashed start is followed once; every vertex then takes its label from its
// slot. The vertices of a brick share a few hundred starts, so each vertex
// costs one read of f and W and one write, and the chases run once per start.
// A vertex whose start finds no room in the hash follows its chain itself.
// 356 us for 400^3 vertices, of which HBM needs 150: the dependent reads of
// the chases and the probes' instructions (389 us with a division into rows
// per vertex and without the start's triplet being fetched when it is
// entered; loops kept together by votes, which serve the build's kernels,
// 406: nearly every probe succeeds at once). 3 CTAs per SM: 406.
//
// WIDE: 64-bit ids (the wide path's triplets and labels). Grids of which a
// brick holds too little take k_labels_each instead (see bricks_pay).
//
// With eps > 0 the labels are those of the simplified field in which every
// branch of persistence below eps is filled up to its saddle: a component of
// G_t whose representative r heads such a branch (r not the root, f(s) - f(r)
// < eps in float32 for r's saddle s) lies inside a filled pit and leaves G_t,
// its vertices labelled 0xFFFFFFFF. No other component changes: by the elder
// rule a branch is never less persistent than one that merges into it, so a
// long branch never lies inside a short one's pit.
constexpr uint32_t kLabLX = 5, kLabLY = 4, kLabLZ = 4;
constexpr uint32_t kLabThreads = 1u << (kLabLX + kLabLY);  // a thread per column of the brick
template <bool WIDE>
struct LabelShape {
    static constexpr uint32_t kSlots = (WIDE ? 2048 : 4096) / kLabelShrink;
    static constexpr size_t kSmem =
        (size_t)kSlots * 2 * sizeof(typename Tri<WIDE>::Id) + ((size_t)2 << (kLabLX + kLabLY + kLabLZ));
};

template <bool WIDE>
__global__ void __launch_bounds__(kLabThreads, 4) k_labels(const float *__restrict__ f, float sg,
                                                           const uint64_t *__restrict__ W, uint32_t nx, uint32_t ny,
                                                           uint32_t nz, uint32_t ntx, uint32_t nty, float t, float eps,
                                                           typename Tri<WIDE>::Id *__restrict__ labels,
                                                           uint32_t *status)
{
    using Id = typename Tri<WIDE>::Id;
    if (block_skips(status)) return;
    const Id nxy = (Id)nx * ny, n = nxy * nz;
    const uint32_t limit = n < kChaseLimit ? (uint32_t)n : kChaseLimit;
    constexpr uint32_t TX = 1u << kLabLX, TY = 1u << kLabLY, TZ = 1u << kLabLZ, NT = kLabThreads;
    constexpr uint32_t HS = LabelShape<WIDE>::kSlots, kProbes = 16, NB = WIDE ? 2 : 4;  // rows loaded together
    constexpr Id EMPTY = ~(Id)0, NOLABEL = ~(Id)0;
    constexpr uint16_t OUT = 0xFFFFu, SELF = 0xFFFEu;  // slot codes: not in G_t; no room in the hash
    static_assert(HS <= SELF && (HS & (HS - 1)) == 0 && TZ % NB == 0, "slot codes, power of two, whole batches");
    extern __shared__ __align__(16) uint64_t lab_smem[];
    Id *hkey = reinterpret_cast<Id *>(lab_smem);       // chain starts
    Id *hval = hkey + HS;                              // their representatives at t
    uint16_t *vslot = reinterpret_cast<uint16_t *>(hval + HS);  // per vertex: slot or code

    const uint32_t tile = blockIdx.x;
    const uint32_t tx = tile % ntx, ty = (tile / ntx) % nty, tz = tile / (ntx * nty);
    const uint32_t x0 = tx * TX, y0 = ty * TY, z0 = tz * TZ;
    const uint32_t wx = min(TX, nx - x0), wy = min(TY, ny - y0), wz = min(TZ, nz - z0);
    const uint32_t cx = threadIdx.x & (TX - 1), cy = threadIdx.x >> kLabLX;
    const bool inx = cx < wx && cy < wy;
    const Id u0 = (Id)z0 * nxy + (Id)(y0 + cy) * nx + x0 + cx;  // vertex z of the column: u0 + z * nxy
    auto val = [&](Id u) { return sg * __ldg(f + u); };
    // a triplet as the caller gave it (all bits of its ids)
    auto load = [&](Id u, Id &s, Id &v) {
        if constexpr (WIDE) {
            const ulonglong2 w = reinterpret_cast<const ulonglong2 *>(W)[u];
            s = w.x, v = w.y;
        } else {
            const uint64_t w = __ldg(reinterpret_cast<const unsigned long long *>(W) + u);
            s = tri_s(w), v = tri_v(w);
        }
    };
    // representative at t of the chain from x: the caller's triplets are
    // followed only through ids < n, and for at most `limit` links (a chain
    // of a valid tree is shorter than n, so a longer one means a cycle)
    bool ok = true, bad = false;
    auto chase = [&](Id x) -> Id {
        for (uint32_t h = 0;; h++) {
            Id s, v;
            load(x, s, v);
            if (s == x && v == x) return x;
            if (s >= n || v >= n) {
                bad = true;
                return x;
            }
            if (!(val(s) <= t)) return x;
            x = v;
            if (h >= limit) {
                ok = false;
                return x;
            }
        }
    };
    // the representative, or NOLABEL if it heads a branch shorter than eps
    auto simplified = [&](Id r) -> Id {
        if (WIDE || !(eps > 0.0f)) return r;
        Id s, v;
        load(r, s, v);
        if (s == r || s >= n) return r;  // the root (or an inner vertex of a corrupt tree)
        return val(s) - val(r) >= eps ? r : NOLABEL;
    };

    for (uint32_t i = threadIdx.x; i < HS; i += NT) hkey[i] = EMPTY;
    __syncthreads();

    // 1. chain starts into the hash
    volatile Id *vhk = hkey;
    for (uint32_t zb = 0; zb < wz; zb += NB) {
        Id sb[NB], vb[NB];
        float fb[NB];
#pragma unroll
        for (uint32_t k = 0; k < NB; k++) {
            const bool in = inx && zb + k < wz;
            const Id u = u0 + (zb + k) * nxy;
            fb[k] = in ? val(u) : 0.0f;
            sb[k] = vb[k] = 0;
            if (in) load(u, sb[k], vb[k]);
        }
#pragma unroll
        for (uint32_t k = 0; k < NB; k++) {
            const uint32_t z = zb + k;
            if (!inx || z >= wz) continue;
            const Id u = u0 + z * nxy;
            uint16_t slot = OUT;
            if (fb[k] <= t) {
                slot = SELF;
                // (an id >= n is left to the vertex's own chase, which reports it)
                if (sb[k] < n && vb[k] < n) {
                    const Id st = (sb[k] == u && vb[k] != u) ? vb[k] : u;
                    uint32_t h = (((uint32_t)st * 0x9E3779B1u) >> 16) & (HS - 1);
                    for (uint32_t p = 0; p < kProbes; p++) {
                        Id q = vhk[h];
                        if (q == EMPTY) {
                            if constexpr (WIDE)
                                q = atomicCAS(reinterpret_cast<unsigned long long *>(hkey + h),
                                              (unsigned long long)EMPTY, (unsigned long long)st);
                            else q = atomicCAS(hkey + h, EMPTY, st);
                            // its chase begins with this read
                            if (q == EMPTY)
                                asm volatile("prefetch.global.L2 [%0];" ::"l"(W + (WIDE ? 2 : 1) * (size_t)st));
                        }
                        if (q == EMPTY || q == st) {
                            slot = (uint16_t)h;
                            break;
                        }
                        h = (h + 1) & (HS - 1);
                    }
                }
            }
            vslot[threadIdx.x + z * NT] = slot;
        }
    }
    __syncthreads();

    // 2. one chase per hashed start. Each warp takes the occupied slots of
    //    its own HS / warps slots and deals them out to its lanes in order
    //    (ballot masks in registers), so that every lane has a chase instead
    //    of one lane per fixed group of mostly empty slots.
    constexpr uint32_t PER = HS / (NT / 32);  // slots per warp
    if constexpr (PER >= 32 && PER % 32 == 0) {
        constexpr uint32_t G = PER >= 32 ? PER / 32 : 1;  // (1 only in the branch not taken)
        const uint32_t lane = threadIdx.x & 31, wbase = (threadIdx.x >> 5) * PER;
        uint32_t mask[G], tot = 0;
#pragma unroll
        for (uint32_t g = 0; g < G; g++) {
            mask[g] = __ballot_sync(0xffffffffu, hkey[wbase + g * 32 + lane] != EMPTY);
            tot += __popc(mask[g]);
        }
        for (uint32_t r = lane; r < tot; r += 32) {
            // the slot of rank r among the warp's occupied slots
            uint32_t rr = r, i = 0;
#pragma unroll
            for (uint32_t g = 0; g < G; g++) {
                const uint32_t c = __popc(mask[g]);
                if (rr < c && i == 0) {
                    uint32_t m = mask[g];
                    for (uint32_t k = 0; k < rr; k++) m &= m - 1;
                    i = wbase + g * 32 + __ffs(m);  // 1 + the slot
                }
                rr = rr < c ? rr : rr - c;
            }
            hval[i - 1] = simplified(chase(hkey[i - 1]));
        }
    } else {
        for (uint32_t i = threadIdx.x; i < HS; i += NT) {
            const Id st = hkey[i];
            if (st != EMPTY) hval[i] = simplified(chase(st));
        }
    }
    __syncthreads();

    // 3. labels
    if (inx) {
        uint32_t self = 0;  // bit z: the vertex follows its chain itself
#pragma unroll 4
        for (uint32_t z = 0; z < wz; z++) {
            const uint16_t c = vslot[threadIdx.x + z * NT];
            self |= (uint32_t)(c == SELF) << z;
            if (c != SELF) labels[u0 + z * nxy] = c == OUT ? NOLABEL : hval[c];
        }
        for (; self; self &= self - 1) {
            const Id u = u0 + (__ffs(self) - 1) * nxy;
            labels[u] = simplified(chase(u));
        }
    }
    if (!ok) raise_status(status, ST_TIMEOUT);
    if (bad) raise_status(status, ST_CORRUPT);
}

// The labels of a wide field, each vertex following its own chain. Where many
// vertices of a neighbourhood share their chains the bricks of k_labels read
// them less often, but a brick with few vertices in it, or a field whose
// triplets stay in L2, costs less this way.
__global__ void __launch_bounds__(256) k_labels_each(const float *f, float sg, const uint64_t *W, uint64_t n, float t,
                                                     uint64_t *labels, uint32_t *status)
{
    if (*status) return;
    bool ok = true, bad = false;
    for (uint64_t u = blockIdx.x * 256ull + threadIdx.x; u < n; u += gridDim.x * 256ull) {
        if (!(sg * __ldg(f + u) <= t)) {
            labels[u] = ~0ull;
            continue;
        }
        const ulonglong2 wu = reinterpret_cast<const ulonglong2 *>(W)[u];
        uint64_t x = wu.x == u && wu.y != u && wu.y < n ? wu.y : u;
        for (uint64_t h = 0;; h++) {
            const ulonglong2 w = reinterpret_cast<const ulonglong2 *>(W)[x];
            if (w.x == x && w.y == x) break;
            if (w.x >= n || w.y >= n) {
                bad = true;
                break;
            }
            if (!(sg * __ldg(f + w.x) <= t)) break;
            x = w.y;
            if (h >= kChaseLimit || h >= n) {
                ok = false;
                break;
            }
        }
        labels[u] = x;
    }
    if (!ok) raise_status(status, ST_TIMEOUT);
    if (bad) raise_status(status, ST_CORRUPT);
}

// Whether wide labels take the bricks: from 2^23 vertices, four planes and
// columns of which three in four lie in the grid. Measured in us, each vertex
// by itself against bricks, white noise at its median: 160^3 83 and 114, 256^3
// 252 and 201, 512^3 2516 and 1424; planes of 8192^2 741 and 1294, 4 of them
// 7044 and 2952; 1024 x 1024 rows of 8 132 and 184, of 24 426 and 292, of 33
// 612 and 477 (16 levels: 382 and 432). Smooth fields, where every chain is
// short, lose up to 9 % to the bricks (320^3 148 and 161), fields of which
// half the vertices are minima up to a factor of two (512^3 829 and 1672).
static bool bricks_pay(uint32_t nx, uint32_t ny, uint32_t nz, uint32_t ntx, uint32_t nty)
{
    if (kLabelShrink > 1) return true;  // the tests' small tables are meant to be reached by small fields
    const uint64_t n = (uint64_t)nx * ny * nz;
    return n >= 1u << 23 && nz >= 4 && 4 * (uint64_t)nx * ny >= 3 * (uint64_t)ntx * nty * kLabThreads;
}

template <bool WIDE>
static cudaError_t run_labels(const float *f, const uint64_t *W, uint32_t nx, uint32_t ny, uint32_t nz, float t,
                              float sg, typename Tri<WIDE>::Id *labels, uint32_t *status, cudaStream_t st, float eps)
{
    PhaseScope ps(kLabels, st);
    const uint32_t ntx = (uint32_t)(((uint64_t)nx + 31) >> kLabLX), nty = (uint32_t)(((uint64_t)ny + 15) >> kLabLY),
                   ntz = (uint32_t)(((uint64_t)nz + 15) >> kLabLZ);
    if constexpr (WIDE) {
        if (!bricks_pay(nx, ny, nz, ntx, nty)) {
            const uint64_t n = (uint64_t)nx * ny * nz, want = (n + 2047) / 2048, most = (uint64_t)device_sms() * 16;
            k_labels_each<<<(unsigned)(want < most ? want : most), 256, 0, st>>>(f, sg, W, n, t, labels, status);
            count_launch();
            return cudaGetLastError();
        }
    }
    static AttrFlags attr;  // per instantiation
    int dev;
    if (attr.pending(dev)) {
        const cudaError_t e = cudaFuncSetAttribute(k_labels<WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)LabelShape<WIDE>::kSmem);
        if (e != cudaSuccess) return e;
        attr.done(dev);
    }
    const uint64_t bricks = (uint64_t)ntx * nty * ntz;
    if (bricks >= 0x80000000ull) return cudaErrorInvalidValue;
    k_labels<WIDE><<<(unsigned)bricks, kLabThreads, LabelShape<WIDE>::kSmem, st>>>(f, sg, W, nx, ny, nz, ntx, nty, t,
                                                                                  eps, labels, status);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_labels(const float *f, const uint64_t *W, uint32_t nx, uint32_t ny, uint32_t nz, float t,
                          float sg, uint32_t *labels, Workspace &ws, cudaStream_t st, float eps)
{
    return run_labels<false>(f, W, nx, ny, nz, t, sg, labels, ws.status, st, eps);
}

cudaError_t launch_labels_wide(const float *f, const uint64_t *W2, uint32_t nx, uint32_t ny, uint32_t nz, float t,
                               float sg, uint64_t *labels, uint32_t *status, cudaStream_t st)
{
    return run_labels<true>(f, W2, nx, ny, nz, t, sg, labels, status, st, 0.0f);
}

}  // namespace mt
