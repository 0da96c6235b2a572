// rgroup.cuh -- lookups in a relation grouped by one column (RGroup, cyclic.h).
#pragma once

#include "cyclic.h"
#include "tables.h"

namespace mwj {

// Entries of the grouping: the direct-address layout (key b at b - min) or
// the hashed key table's slot (slot mask + 1 holds key -1).
__device__ __forceinline__ uint32_t rg_entries(const uint32_t *meta) {
    return meta[kMetaDense] ? meta[kMetaSpan] : meta[kMetaMask] + 2u;
}

__device__ __forceinline__ int rg_find(const RGroup &r, const uint32_t *meta, uint32_t b) {
    if (meta[kMetaDense]) {
        const uint32_t k = b - meta[kMetaMin];
        return k < meta[kMetaSpan] ? (int)k : -1;
    }
    return tbl_find(r.keys, meta[kMetaMask], b, r.seed);
}

}  // namespace mwj
