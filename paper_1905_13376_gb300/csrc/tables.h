// tables.h -- T's tables (one L2-resident table, or per-bucket images) and their lookup.
#pragma once

#include "common.cuh"

namespace mwj {

// Words of a single table's meta array: mask of the hashed slots, distinct
// estimate, and, when the sizing pass chose the direct-address layout
// (kMetaDense = 1), the smallest key, the span of the keys and a shift: the entry
// of key k is then at (k - min) << shift (0 for all but a star join's weights),
// nothing is hashed and no key is stored.
// kMetaTry: that layout is left to the distinct estimate.  kMetaPacked: hashed
// weights in packed slots (bit 0; bit 1: some sum has an upper word, linear_l2.h).
constexpr int kMetaMask = 0, kMetaEst = 1, kMetaShift = 2, kMetaDense = 3, kMetaMin = 4, kMetaSpan = 5, kMetaTry = 6,
              kMetaPacked = 7;
constexpr int kMetaWords = 8;

// J == 0: one table of (meta[0] + 1) packed (deg << 32 | c) slots, home slot
//         slot_of(c, seed_slot, meta[0]) (the one-bucket plan of linear_l2.cu
//         has tables of its own).
// J >= 1: bucket j = bucket_of(c, seed_bucket, J) lives at
//         img[2*off[j] .. 2*off[j] + cap[j]); with row output start[2*off[j] + slot]
//         is the first position of c's D values in dlist.
struct TImg {
    const uint64_t *img;
    const uint32_t *off;
    const uint32_t *cap;
    const uint32_t *start;
    const int32_t *dlist;
    const uint32_t *meta;
    uint32_t J;
    uint32_t seed_bucket;
    uint32_t seed_slot;
};

__device__ __forceinline__ uint32_t timg_deg(const TImg &t, int32_t c) {
    if (t.J == 0) {
        const uint32_t mask = __ldg(t.meta);
        uint32_t s = slot_of((uint32_t)c, t.seed_slot, mask);
        for (uint32_t it = 0; it <= mask; ++it) {
            uint64_t v = __ldg((const unsigned long long *)(t.img + s));
            if (v == kEmpty64) return 0;
            if ((uint32_t)v == (uint32_t)c) return (uint32_t)(v >> 32);
            s = (s + 1) & mask;
        }
        return 0;
    }
    uint32_t j = (t.J == 1) ? 0u : bucket_of(c, t.seed_bucket, t.J);
    uint64_t base = 2ull * __ldg(t.off + j);
    return img_lookup(t.img + base, __ldg(t.cap + j), (uint32_t)c, t.seed_slot);
}

// deg and start of c (deg 0 when absent); bucket images only
__device__ __forceinline__ uint32_t timg_deg_start(const TImg &t, int32_t c, uint32_t *start) {
    uint32_t j = (t.J == 1) ? 0u : bucket_of(c, t.seed_bucket, t.J);
    uint64_t base = 2ull * __ldg(t.off + j);
    int64_t s = img_slot(t.img + base, __ldg(t.cap + j), (uint32_t)c, t.seed_slot);
    if (s < 0) return 0;
    uint64_t v = __ldg((const unsigned long long *)(t.img + base + s));
    *start = __ldg(t.start + base + s);
    return (uint32_t)(v >> 32);
}

cudaError_t tables_build(const uint32_t *keys, const uint2 *pairs, const uint32_t *off, uint32_t J,
                         uint32_t seed, uint64_t *img, uint32_t *capv, uint32_t *startv,
                         int32_t *dlist, DevStatus *status, int num_sms, cudaStream_t st);

// slots to reserve for the single table of nT tuples (worst case)
size_t single_table_slots(int64_t nT);
// ekey/ecnt: nT entries each; ecount: J; meta: at least 4 words (the layout
// flag, kMetaDense, is written too).
cudaError_t single_table_build(const uint32_t *keys, const uint32_t *off, uint32_t J, uint32_t seed,
                               uint32_t *ekey, uint32_t *ecnt, uint32_t *ecount, uint32_t *meta,
                               uint64_t *tbl, DevStatus *status, int num_sms, cudaStream_t st);

// One table without partitioning T: a HyperLogLog pass over the keys sizes
// the table (2^k >= 4 x the estimate, 2 x for large ones, at most
// reserve_slots), then the keys are inserted directly.  hll_regs:
// hll_scratch_registers(num_sms) u32; meta: kMetaWords.
cudaError_t single_table_direct(const int32_t *keys, int64_t n, uint32_t seed, unsigned int *hll_regs,
                                uint32_t *meta, uint64_t *tbl, uint64_t reserve_slots,
                                DevStatus *status, int num_sms, cudaStream_t st);
// Only its sizing step; with allow_dense a compact key range gets the
// direct-address layout.  hll_name, size_name: the launches' names in the
// per-kernel profile.
cudaError_t single_table_size(const int32_t *keys, int64_t n, uint32_t seed, unsigned int *hll_regs,
                              uint32_t *meta, uint64_t reserve_slots, int num_sms, cudaStream_t st,
                              const char *hll_name = "t_hll", const char *size_name = "t_size",
                              bool allow_dense = false);

// Several key columns sized in the same launches, a column for up to
// kSizeCols tables of its keys (meta[q], at most reserve[q] hashed slots and
// range[q] direct-address entries each).
constexpr uint32_t kSizeCols = 3;
struct SizeCol {
    const int32_t *keys;
    uint32_t n, seed;
    unsigned int *scratch;   // hll_scratch_registers(num_sms) u32 of its own
    uint32_t *meta[kSizeCols];
    uint64_t reserve[kSizeCols], range[kSizeCols];
    uint32_t ntargets;
    // > 0: the direct-address entries of the (one) table are spread out over this
    // many at most, so that adds to neighbouring keys meet in no L2 sector
    uint64_t spread = 0;
    bool weights = false;   // the table may take packed slots (linear_l2.h)
    // a range of at most `sure` entries is direct-address whatever the number of
    // distinct keys, a larger one when it is at most `per_key` times the estimate
    // or the keys are few (k_hll)
    uint64_t sure = 1ull << 24;
    uint64_t near = 3ull << 23;   // the same for up to 2^18 keys
    double per_key = 8.0;
};
// A column whose heavy keys (sampled share at least 1 / (2 x buckets)) are
// named by the first of these launches (allow_dense only) in `heavy`
// (kHeavyTableWords, skew.h).
struct HeavyCol {
    const int32_t *keys;
    uint32_t n, buckets;
    uint32_t *heavy;
    bool coarse = false;   // from half as large a sample
};
cudaError_t size_columns(const SizeCol *cols, uint32_t ncols, const HeavyCol *heavy, uint32_t nheavy, bool allow_dense,
                         int num_sms, cudaStream_t st, const char *hll_name = "t_hll",
                         const char *size_name = "t_size");
// Tables to empty, in the layout meta describes: degrees (keys null; u32
// entries, or hashed packed slots) or weights (u64 sums; hashed: keys[] too).
struct ClearTable {
    unsigned long long *tbl;
    uint32_t *keys;
    const uint32_t *meta;
};
// One launch for all of them (at most kSizeCols) and the call's outputs:
// zero[0, nzero) and *total (both may be null).
cudaError_t tables_clear(const ClearTable *t, uint32_t n, unsigned long long *zero, uint64_t nzero,
                         unsigned long long *total, int num_sms, cudaStream_t st);
uint32_t hll_registers();
size_t hll_scratch_registers(int num_sms);
// HyperLogLog registers of keys[0, n) into regs[0, hll_registers()); regs must
// hold hll_scratch_registers(num_sms) u32 (per-CTA registers, then merged)
cudaError_t hll_regs(const int32_t *keys, int64_t n, uint32_t seed, unsigned int *regs, int num_sms,
                     cudaStream_t st);

}  // namespace mwj
