// Where a CTA's work lives: one field (the descriptor travels by value in the
// kernel parameters) or a packed batch of fields (a descriptor table in the
// workspace, searched by the first tile / first compaction chunk of each
// field). Every kernel of the path is written once against this interface.
#pragma once
#include <cstdint>

#include "mt_internal.h"

namespace mt {

struct OneField {
    FieldDesc d;
    __device__ __forceinline__ FieldDesc tile(uint32_t g, uint32_t &local) const
    {
        local = g;
        return d;
    }
    __device__ __forceinline__ FieldDesc chunk(uint64_t g, uint64_t &local, uint32_t &fi) const
    {
        local = g;
        fi = 0;
        return d;
    }
    __device__ __forceinline__ FieldDesc field(uint32_t) const { return d; }
};

// A field is found by whole warps: 32 lanes read the first tiles (chunks) of 32
// evenly spaced fields at a time, so that a batch of 512 fields takes two
// dependent reads instead of the nine of a binary search.
struct ManyFields {
    const FieldDesc *d;
    uint32_t nfields;
    // last field whose first(field) is <= g (fields with no tiles cannot occur)
    template <class First>
    __device__ __forceinline__ uint32_t find(uint64_t g, First first) const
    {
        const uint32_t lane = threadIdx.x & 31;
        uint32_t lo = 0, len = nfields;  // the answer is in [lo, lo + len)
        while (len > 1) {
            const uint32_t step = (len + 31) / 32, i = lo + lane * step;
            const bool le = lane * step < len && first(d[i]) <= g;
            const uint32_t k = __popc(__ballot_sync(0xffffffffu, le)) - 1;  // (field lo is always one)
            lo += k * step;
            len = len - k * step < step ? len - k * step : step;
        }
        return lo;
    }
    __device__ __forceinline__ FieldDesc tile(uint32_t g, uint32_t &local) const
    {
        const uint32_t i = find(g, [](const FieldDesc &f) -> uint64_t { return f.tile0; });
        local = g - d[i].tile0;
        return d[i];
    }
    __device__ __forceinline__ FieldDesc chunk(uint64_t g, uint64_t &local, uint32_t &fi) const
    {
        fi = find(g, [](const FieldDesc &f) -> uint64_t { return f.chunk0; });
        local = g - d[fi].chunk0;
        return d[fi];
    }
    __device__ __forceinline__ FieldDesc field(uint32_t i) const { return d[i]; }
};

}  // namespace mt
