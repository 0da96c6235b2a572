// skew.h -- heavy join keys: detection, partition routing, and the
// aggregate kernels of the heavy bucket.
#pragma once

#include "tables.h"

namespace mwj {

// Heavy-key table: kHeavySlots keys (open addressing, home slot
// slot_of(key, kHeavySeed, kHeavySlots - 1), kEmptyKey = empty) followed by
// the number of keys; at most kHeavyMax keys.
constexpr uint32_t kHeavySlots = 512;
constexpr uint32_t kHeavyMax = 256;
constexpr uint32_t kHeavySeed = 0x2545F491u;
constexpr size_t kHeavyTableWords = kHeavySlots + 4;

// Slot of key k in the heavy table (a copy in shared memory), -1 if absent.
// Not inlined: the partition kernels call it only when the table holds keys,
// and an inlined probe loop at every bucket computation of their unrolled
// loops would crowd the instruction cache of the common, heavy-free case.
static __device__ __noinline__ int heavy_slot(const uint32_t *hs, uint32_t k) {
    if (k == kEmptyKey) return -1;
    uint32_t s = slot_of(k, kHeavySeed, kHeavySlots - 1);
    for (uint32_t it = 0; it < kHeavySlots; ++it) {
        const uint32_t q = hs[s];
        if (q == k) return (int)s;
        if (q == kEmptyKey) return -1;
        s = (s + 1) & (kHeavySlots - 1);
    }
    return -1;
}

// Copy a heavy table into shared memory (every thread of the CTA calls this;
// ends with a barrier when it copies).  Returns null when there is no table
// or it holds no key, so that callers skip the per-tuple check.
__device__ __forceinline__ const uint32_t *heavy_to_smem(const uint32_t *heavy, uint32_t *buf) {
    if (!heavy || __ldg(heavy + kHeavySlots) == 0) return nullptr;
    for (uint32_t i = threadIdx.x; i < kHeavySlots; i += blockDim.x) buf[i] = __ldg(heavy + i);
    __syncthreads();
    return buf;
}

// The heavy keys of one column from a strided sample of SAMPLED of its tuples,
// by one CTA of NT threads (sm: its shared memory): those whose sampled share
// reaches 1 / (2 buckets), and at least kHeavyMinCount sampled tuples.
constexpr uint32_t kHeavyMinCount = 8;
template <uint32_t SAMPLED>
struct HeavySample {
    static constexpr uint32_t slots = 2 * SAMPLED;   // count table, at most half full
    uint32_t key[slots], cnt[slots], ht[kHeavySlots], nh;
};

template <int NT, uint32_t SAMPLED>
__device__ __forceinline__ void heavy_sample_cta(const int32_t *__restrict__ col, uint32_t n, uint32_t buckets,
                                                 uint32_t *__restrict__ heavy, HeavySample<SAMPLED> &sm) {
    constexpr uint32_t kHeavyCountSlots = HeavySample<SAMPLED>::slots;
    const uint32_t m = n < SAMPLED ? n : SAMPLED;
    constexpr uint32_t PER = SAMPLED / NT;
    static_assert(PER * NT == SAMPLED, "a whole number of samples per thread");
    uint32_t ks[PER];
#pragma unroll
    for (uint32_t q = 0; q < PER; ++q) {
        const uint32_t j = threadIdx.x + q * NT;
        ks[q] = j < m ? (uint32_t)__ldg(col + (uint32_t)(((uint64_t)j * n) / m)) : kEmptyKey;
    }
    for (uint32_t i = threadIdx.x; i < kHeavyCountSlots; i += NT) {
        sm.key[i] = kEmptyKey;
        sm.cnt[i] = 0;
    }
    for (uint32_t i = threadIdx.x; i < kHeavySlots; i += NT) sm.ht[i] = kEmptyKey;
    if (threadIdx.x == 0) sm.nh = 0;
    __syncthreads();
#pragma unroll
    for (uint32_t q = 0; q < PER; ++q) {
        const uint32_t k = ks[q];
        if (k == kEmptyKey) continue;   // the table's empty marker is never heavy
        uint32_t s = slot_of(k, kHeavySeed, kHeavyCountSlots - 1);
        for (uint32_t it = 0; it < kHeavyCountSlots; ++it) {   // at most half full: ends early
            uint32_t held = sm.key[s];
            if (held == kEmptyKey) {
                held = atomicCAS(&sm.key[s], kEmptyKey, k);
                if (held == kEmptyKey) held = k;
            }
            if (held == k) {
                atomicAdd(&sm.cnt[s], 1u);
                break;
            }
            s = (s + 1) & (kHeavyCountSlots - 1);
        }
    }
    __syncthreads();
    const uint32_t t = max(kHeavyMinCount, m / (2u * buckets));
    for (uint32_t i = threadIdx.x; i < kHeavyCountSlots; i += NT) {
        const uint32_t k = sm.key[i];
        if (k == kEmptyKey || sm.cnt[i] < t) continue;
        if (atomicAdd(&sm.nh, 1u) >= kHeavyMax) continue;
        // at most kHeavyMax = kHeavySlots / 2 keys: a free slot is always found
        uint32_t s = slot_of(k, kHeavySeed, kHeavySlots - 1);
        for (uint32_t it = 0; it < kHeavySlots && atomicCAS(&sm.ht[s], kEmptyKey, k) != kEmptyKey; ++it)
            s = (s + 1) & (kHeavySlots - 1);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < kHeavySlots; i += NT) heavy[i] = sm.ht[i];
    if (threadIdx.x == 0) heavy[kHeavySlots] = sm.nh < kHeavyMax ? sm.nh : kHeavyMax;
}

// Heavy keys of the join column B from samples of R's and S's B columns: a
// key is heavy when its sampled share in either relation reaches half of an
// average H(B) bucket (1 / (2 I)).  Also zeroes hw (kHeavySlots u64).
cudaError_t heavy_detect(const int32_t *rb, int64_t nR, const int32_t *sb, int64_t nS, uint32_t I,
                         uint32_t *heavy, unsigned long long *hw, cudaStream_t st);

// The heavy bucket (index hb of the partitions) of the linear aggregates:
// hw[h] = sum of deg_T(c) over S tuples (h, c), then for R tuples (a, h):
// total += hw[h] and (GROUP BY A) cnt[a] += hw[h].
cudaError_t heavy_linear(const uint2 *Sp, const uint32_t *offS, uint32_t hbS, const uint2 *Rp,
                         const uint32_t *offR, uint32_t hbR, const uint32_t *heavy, const TImg &T,
                         unsigned long long *hw, int32_t a_domain, unsigned long long *cnt,
                         unsigned long long *total, int num_sms, cudaStream_t st);

}  // namespace mwj
