// linear_l2.h -- linear joins with one bucket on each side: the weight tables,
// e.g. S's w(b) = sum over (b, c) in S of deg_T(c), held in the L2.
#pragma once

#include "internal.h"
#include "tables.h"

namespace mwj {

// Degrees of the chain's last relation, c -> deg(c).  meta (tables.h) says
// which layout the sizing pass chose: the direct-address one (uint32 deg[c - min]),
// or 2^k packed (deg << 32 | c) slots in pairs of 16 bytes: a key lives in the
// first free slot at or after its home pair, so one 16-byte load nearly
// always settles a lookup.  Key -1 is a key like any other (a count below
// 2^31 keeps its slot different from kEmpty64).
struct DegTable {
    unsigned long long *slots;   // single_table_slots(n)
    uint32_t *meta;              // kMetaWords entries
    uint32_t seed;
    const uint32_t *heavy;       // heavy keys of the column (skew.h's table), or null
};

// Weights b -> w(b), exact modulo 2^64: the direct-address sums W[b - min], or
// 2^k slots, keys and sums apart: keys[s] in groups of four (one 16-byte load),
// W[s] the sum, added to with 64-bit adds whose results are not needed.  Key -1,
// the mark of a free slot, has its sum in W[mask + 1].  A table larger than the L2
// (from kPackedSlots slots on, tables.cu) has packed slots instead, W[s] = lower
// word of the sum << 32 | key and keys[s] the upper word: a new key is claimed and
// added with one atomic, and out there every atomic moves a sector from and to memory.
struct WTable {
    unsigned long long *W;   // w_table_slots(n) + 2 entries reserved
    uint32_t *keys;          // w_table_slots(n) entries reserved
    uint32_t *meta;          // kMetaWords entries
    uint32_t seed;
    const uint32_t *heavy;   // heavy keys of the relation's key column (skew.h's table)
};

// Heavy keys of a weight pass: a sampled share of at least 1 / (2 x this).
constexpr uint32_t kWHeavyBuckets = 128;

// Slots to reserve for S of nS tuples (the table never grows past this).
size_t w_table_slots(int64_t nS);

// The one-bucket plan of a chain R(A,B) S(B,C) T(C,D) [U(D,E)]: the last
// relation's degree table and one weight table per relation between it and R.
constexpr int kChainMax = 4;
struct OneBucket {
    DegTable deg;                   // of the last relation
    unsigned int *hll[kSizeCols];   // sizing scratch, one per key column
    WTable w[kChainMax - 2];        // w[k]: weights of relation nrel - 2 - k (w[0] is looked up by w[1]'s pass)
};
// rel[0] = R ... rel[nrel - 1]: the last (nrel 3 or 4).
void one_bucket_layout(Arena &A, const mwj_rel *rel, int nrel, int num_sms, OneBucket &L);
// Largest power of two of CTAs (at most 16) that the current device launches as one
// cluster of the small plan; 1: none.  Also allows the sizes above 8.
int chain_cluster_limit();
// COUNT (mode 0: *total) or GROUP BY A (mode 1: cnt[0, a_domain) too); the
// outputs are zeroed here.  a outside [0, a_domain) raises MWJ_ERR_DOMAIN.
cudaError_t one_bucket_run(OneBucket &L, const mwj_rel *rel, int nrel, const Seeds &sd, int mode, int32_t a_domain,
                           unsigned long long *cnt, unsigned long long *total, DevStatus *status, const DevInfo &dev,
                           cudaStream_t st);
// The same for a star join (small R and T, large S): w[0] holds R's keys.
void star_bucket_layout(Arena &A, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, int num_sms, OneBucket &L);
cudaError_t star_bucket_run(OneBucket &L, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, const Seeds &sd, int mode,
                            int32_t a_domain, unsigned long long *cnt, unsigned long long *total, DevStatus *status,
                            const DevInfo &dev, cudaStream_t st);

}  // namespace mwj
