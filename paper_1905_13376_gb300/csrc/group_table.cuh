// group_table.cuh -- open addressing over groups of four keys.
//
// keys[] holds 2^k uint32 slots (k >= 4), kEmptyKey when free, in groups of
// four: one 16-byte load shows a whole group, so a search is one load unless
// the group is full.  A key is put into the first free slot at or after its
// home group and never moves, so a group fills in order and a search may stop
// at a group with a free slot.  kEmptyKey itself cannot be a key: callers keep
// its value apart.
#pragma once

#include "common.cuh"

namespace mwj {

// The group of four keys at which the search for key k starts.
__device__ __forceinline__ uint32_t w_home(uint32_t k, uint32_t seed, uint32_t mask) {
    return slot_of(k, seed, mask) & ~3u;
}

// Slot of key k (not -1) from its home group (slot s, keys v); kEmptyKey when a
// free slot comes first.
__device__ __forceinline__ uint32_t w_find(const uint32_t *__restrict__ keys, uint32_t mask, uint32_t k, uint32_t s,
                                           uint4 v) {
    for (uint32_t it = 0; it <= mask; it += 4) {
        if (v.x == k) return s;
        if (v.y == k) return s + 1;
        if (v.z == k) return s + 2;
        if (v.w == k) return s + 3;
        if (v.w == kEmptyKey) break;   // (a group fills in order: v.w free says that it is not full)
        s = (s + 4) & mask;
        v = __ldg((const uint4 *)(keys + s));
    }
    return kEmptyKey;
}

// Slot of key k (not -1), claimed if it is new, from its home group (possibly
// read before other threads claimed slots of it); kEmptyKey: the table is full.
__device__ __forceinline__ uint32_t w_claim(uint32_t *keys, uint32_t mask, uint32_t k, uint32_t s, uint4 v) {
    for (uint32_t it = 0; it <= mask; it += 4) {
        if (v.x == k) return s;
        if (v.y == k) return s + 1;
        if (v.z == k) return s + 2;
        if (v.w == k) return s + 3;
        if (v.w == kEmptyKey) {
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) {
                uint32_t u = q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w;
                if (u == kEmptyKey) {
                    u = atomicCAS(keys + s + q, kEmptyKey, k);
                    if (u == kEmptyKey || u == k) return s + q;
                }
            }
        }
        s = (s + 4) & mask;
        v = __ldcg((const uint4 *)(keys + s));
    }
    return kEmptyKey;
}

}  // namespace mwj
