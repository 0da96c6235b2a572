// tables.cu -- hash tables of T's C values (K4).
//
// After T is partitioned by g(C) (Algorithm 1, step 1) the probe needs, for
// each c, deg_T(c) = |{(c,d) in T}| (count modes) or c's group of D values
// (row output).  Two layouts:
//
//  * one table ("T held whole on chip", used when S is not split by C):
//    every bucket T_j is aggregated in shared memory (one CTA per bucket,
//    32-bit atomics), its (c, count) entries are appended to a compact list,
//    and the entries are then inserted into a single open-addressing table of
//    2^k >= 2 x (entries) packed (count << 32 | c) slots that stays resident
//    in L2.  A probe is one 8-byte load in the common case.
//  * bucket images (S split by (H(B), g(C)), and row output): bucket j's
//    table occupies slots [2*off[j], 2*off[j] + cap[j]) of one image array,
//    cap[j] = 2 x its distinct keys, 16-byte aligned so that it can be copied
//    into shared memory in one bulk copy.  With row output a parallel start[]
//    array gives the first position of c's D values in dlist.
//
// A bucket whose distinct keys overflow the shared-memory table is handled
// in pieces (the table is flushed and restarted), and the global insert adds
// the partial counts together, so any skew stays exact.
#include <climits>

#include "internal.h"
#include "skew.h"
#include "tables.h"
#include "warp_runs.cuh"

namespace mwj {
namespace {

constexpr int BT = 512;
constexpr uint32_t kAggSlots = 8192;          // shared-memory aggregation table
// Slots of the single T table per estimated distinct C value: the power of
// two at or above 4 x the estimate keeps the load between 1/8 and 1/4 (a
// factor of 2 measured slower: longer probe runs in both insert and lookup).
constexpr double kSingleTableFactor = 4.0;
// Above 2^21 slots (16 MB) a factor of 2: two tables of 2 million distinct keys
// at 4 x (64 MB each) spill out of the 129 MB L2 they share with the streams,
// and every probe then moves DRAM sectors (8.4 million id-keyed tuples, one pass: 0.28
// against 0.24 ms).
constexpr double kSmallTableSlots = (double)(1u << 21);
constexpr double kLargeTableFactor = 2.0;
constexpr uint32_t kImgSmemSlots = 8192;      // 64 KB of packed slots (bucket images)

// insert into a global region of arbitrary capacity (fastrange start), adding `add`
__device__ __forceinline__ uint32_t gagg_insert(unsigned long long *tbl, uint32_t cap, uint32_t k,
                                                uint32_t seed, unsigned long long add,
                                                DevStatus *st) {
    uint32_t s = fastrange(mix32(k ^ seed), cap);
    const unsigned long long fresh = (add << 32) | (unsigned long long)k;
    for (uint32_t it = 0; it < cap; ++it) {
        unsigned long long v = tbl[s];
        if (v == kEmpty64) {
            unsigned long long old = atomicCAS(&tbl[s], kEmpty64, fresh);
            if (old == kEmpty64) return s;
            v = old;
        }
        if ((uint32_t)v == k) {
            atomicAdd(&tbl[s], add << 32);
            return s;
        }
        s = (s + 1 == cap) ? 0 : s + 1;
    }
    set_status(st, MWJ_ERR_CHECK, 2);   // sized to stay half empty: cannot happen
    return 0;
}

// insert into the power-of-two single table, from the first probe (slot s,
// value v, possibly read before another thread claimed the slot)
__device__ __forceinline__ void single_insert_from(unsigned long long *tbl, uint32_t mask, uint32_t k, uint32_t s,
                                                   unsigned long long v, unsigned long long add,
                                                   DevStatus *st) {
    const unsigned long long fresh = (add << 32) | (unsigned long long)k;
    for (uint32_t it = 0; it <= mask; ++it) {
        if (v == kEmpty64) {
            unsigned long long old = atomicCAS(&tbl[s], kEmpty64, fresh);
            if (old == kEmpty64) return;
            v = old;
        }
        if ((uint32_t)v == k) {
            atomicAdd(&tbl[s], add << 32);
            return;
        }
        s = (s + 1) & mask;
        v = __ldcg(tbl + s);
    }
    set_status(st, MWJ_ERR_CHECK, 3);
}

__device__ __forceinline__ void single_insert(unsigned long long *tbl, uint32_t mask, uint32_t k,
                                              uint32_t seed, unsigned long long add, DevStatus *st) {
    const uint32_t s = slot_of(k, seed, mask);
    single_insert_from(tbl, mask, k, s, __ldcg(tbl + s), add, st);
}

// ---------------------------------------------------------------------------
// single table
// ---------------------------------------------------------------------------

// One CTA per bucket: aggregate the bucket's keys in shared memory and append
// (key, count) entries to ekey/ecnt at the bucket's tuple offset.
__global__ void __launch_bounds__(BT) k_tagg(const uint32_t *__restrict__ keys,
                                             const uint32_t *__restrict__ off, uint32_t J,
                                             uint32_t seed, uint32_t *__restrict__ ekey,
                                             uint32_t *__restrict__ ecnt,
                                             uint32_t *__restrict__ ecount, DevStatus *st) {
    extern __shared__ uint32_t sm[];
    uint32_t *tk = sm;                         // kAggSlots + 1 keys
    uint32_t *tc = sm + kAggSlots + 1;         // kAggSlots + 1 counts
    __shared__ uint32_t nd, nout;
    const uint32_t mask = kAggSlots - 1;
    for (uint32_t j = blockIdx.x; j < J; j += gridDim.x) {
        const uint32_t o0 = off[j], o1 = off[j + 1];
        if (threadIdx.x == 0) nout = 0;
        uint32_t pos = o0;
        while (pos < o1) {
            for (uint32_t s = threadIdx.x; s <= kAggSlots; s += BT) {
                tk[s] = (s < kAggSlots) ? kEmptyKey : 0u;
                tc[s] = 0u;
            }
            if (threadIdx.x == 0) nd = 0;
            // rounds of rt keys while the table stays at most 3/4 full
            const uint32_t rt = round_tuples(kAggSlots, 4 * BT);
            for (;;) {
                __syncthreads();
                const uint32_t filled = nd;
                __syncthreads();
                if (pos >= o1 || filled + rt > kAggSlots - kAggSlots / 4) break;
                uint32_t fresh_n = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    uint32_t li = threadIdx.x + k * BT;
                    uint32_t i = pos + li;
                    if (li < rt && i < o1) {
                        bool fresh;
                        int s = tbl_insert(tk, mask, __ldg(keys + i), seed, &fresh);
                        if (s < 0) {
                            set_status(st, MWJ_ERR_CHECK, 4);
                            continue;
                        }
                        fresh_n += fresh;
                        atomicAdd(&tc[s], 1u);
                    }
                }
                fresh_n = warp_sum(fresh_n);
                if ((threadIdx.x & 31) == 0 && fresh_n) atomicAdd(&nd, fresh_n);
                pos += rt;
            }
            // flush the table's entries
            for (uint32_t s = threadIdx.x; s <= kAggSlots; s += BT) {
                uint32_t c = tc[s];
                if (c) {
                    uint32_t k = (s < kAggSlots) ? tk[s] : kEmptyKey;
                    uint32_t p = atomicAdd(&nout, 1u);
                    ekey[o0 + p] = k;
                    ecnt[o0 + p] = c;
                }
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) ecount[j] = nout;
        __syncthreads();
    }
}

// Sum of the entry counts (one CTA) and the table's power-of-two mask.
__global__ void k_tsize(const uint32_t *__restrict__ ecount, uint32_t J, uint32_t *__restrict__ meta) {
    __shared__ unsigned long long red[32];
    unsigned long long s = 0;
    for (uint32_t j = threadIdx.x; j < J; j += blockDim.x) s += ecount[j];
    s = block_sum_u64(s, red);
    if (threadIdx.x == 0) {
        unsigned long long cap = 16;
        while (cap < 2 * s) cap <<= 1;
        meta[0] = (uint32_t)(cap - 1);   // mask
        meta[1] = (uint32_t)s;
        meta[kMetaDense] = 0u;           // hashed slots
    }
}

__global__ void k_tclear(unsigned long long *__restrict__ tbl, const uint32_t *__restrict__ meta) {
    const uint64_t words = (uint64_t)meta[0] + 1;
    for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s < words;
         s += (uint64_t)gridDim.x * blockDim.x)
        tbl[s] = kEmpty64;
}

__global__ void __launch_bounds__(BT) k_tinsert(const uint32_t *__restrict__ ekey,
                                                const uint32_t *__restrict__ ecnt,
                                                const uint32_t *__restrict__ off,
                                                const uint32_t *__restrict__ ecount, uint32_t J,
                                                uint32_t seed, unsigned long long *__restrict__ tbl,
                                                const uint32_t *__restrict__ meta, DevStatus *st) {
    const uint32_t mask = meta[0];
    for (uint32_t j = blockIdx.x; j < J; j += gridDim.x) {
        const uint32_t o0 = off[j], e = ecount[j];
        for (uint32_t i = threadIdx.x; i < e; i += BT)
            single_insert(tbl, mask, ekey[o0 + i], seed, ecnt[o0 + i], st);
    }
}

// ---------------------------------------------------------------------------
// bucket images
// ---------------------------------------------------------------------------

__device__ __forceinline__ void img_agg_insert(unsigned long long *tbl, uint32_t mask, uint32_t k,
                                               uint32_t seed) {
    uint32_t s = mix32(k ^ seed) & mask;
    const unsigned long long fresh = (1ull << 32) | (unsigned long long)k;
    for (uint32_t it = 0; it <= mask; ++it) {   // sized >= 2x the bucket: never full
        unsigned long long v = tbl[s];
        if (v == kEmpty64) {
            unsigned long long old = atomicCAS(&tbl[s], kEmpty64, fresh);
            if (old == kEmpty64) return;
            v = old;
        }
        if ((uint32_t)v == k) {
            atomicAdd(&tbl[s], 1ull << 32);
            return;
        }
        s = (s + 1) & mask;
    }
}

__device__ __forceinline__ uint32_t key_of(const uint32_t *keys, const uint2 *pairs, uint32_t i) {
    return keys ? keys[i] : pairs[i].x;
}

// One CTA per bucket.  keys (count modes) or pairs (row mode, (c,d)).
template <bool CSR>
__global__ void __launch_bounds__(BT) k_tbuild(const uint32_t *__restrict__ keys,
                                               const uint2 *__restrict__ pairs,
                                               const uint32_t *__restrict__ off, uint32_t J,
                                               uint32_t seed, unsigned long long *__restrict__ img,
                                               uint32_t *__restrict__ capv,
                                               uint32_t *__restrict__ startv,
                                               int32_t *__restrict__ dlist, DevStatus *st) {
    extern __shared__ unsigned long long tbl[];   // kImgSmemSlots
    __shared__ unsigned long long red[32];
    for (uint32_t j = blockIdx.x; j < J; j += gridDim.x) {
        const uint32_t o0 = off[j], o1 = off[j + 1];
        const uint32_t n = o1 - o0;
        unsigned long long *reg = img + 2ull * o0;
        uint32_t cap;
        if (n == 0) {
            if (threadIdx.x == 0) capv[j] = 0;
            continue;
        }
        if (2u * n <= kImgSmemSlots) {
            uint32_t sc = 16;
            while (sc < 2u * n) sc <<= 1;
            const uint32_t mask = sc - 1;
            for (uint32_t s = threadIdx.x; s < sc; s += BT) tbl[s] = kEmpty64;
            __syncthreads();
            for (uint32_t i = o0 + threadIdx.x; i < o1; i += BT)
                img_agg_insert(tbl, mask, key_of(keys, pairs, i), seed);
            __syncthreads();
            unsigned long long mine = 0;
            for (uint32_t s = threadIdx.x; s < sc; s += BT) mine += (tbl[s] != kEmpty64);
            const uint32_t D = (uint32_t)block_sum_u64(mine, red);
            cap = 2u * D;
            for (uint32_t s = threadIdx.x; s < cap; s += BT) reg[s] = kEmpty64;
            __syncthreads();
            for (uint32_t s = threadIdx.x; s < sc; s += BT) {
                unsigned long long v = tbl[s];
                if (v != kEmpty64) gagg_insert(reg, cap, (uint32_t)v, seed, v >> 32, st);
            }
        } else {
            cap = 2u * n;
            for (uint32_t s = threadIdx.x; s < cap; s += BT) reg[s] = kEmpty64;
            __syncthreads();
            for (uint32_t i = o0 + threadIdx.x; i < o1; i += BT)
                gagg_insert(reg, cap, key_of(keys, pairs, i), seed, 1ull, st);
        }
        if (threadIdx.x == 0) capv[j] = cap;
        __syncthreads();
        if (CSR) {
            // starts: exclusive scan of the degrees over the image's slots, as
            // absolute positions in dlist, used first as fill cursors
            uint32_t *sv = startv + 2ull * o0;
            __shared__ uint32_t scan_scratch[33];
            __shared__ uint32_t carry;
            if (threadIdx.x == 0) carry = o0;
            __syncthreads();
            for (uint32_t b = 0; b < cap; b += BT) {
                uint32_t s = b + threadIdx.x;
                unsigned long long v = (s < cap) ? reg[s] : kEmpty64;
                uint32_t d = (v == kEmpty64) ? 0u : (uint32_t)(v >> 32);
                uint32_t tot;
                uint32_t ex = block_excl_scan_u32(d, scan_scratch, &tot);
                if (s < cap) sv[s] = carry + ex;
                __syncthreads();
                if (threadIdx.x == 0) carry += tot;
                __syncthreads();
            }
            for (uint32_t i = o0 + threadIdx.x; i < o1; i += BT) {
                uint2 t = pairs[i];
                // plain loads: the image was written earlier in this kernel
                uint32_t s = fastrange(mix32(t.x ^ seed), cap);
                bool found = false;
                for (uint32_t it = 0; it < cap; ++it) {
                    unsigned long long v = reg[s];
                    if (v != kEmpty64 && (uint32_t)v == t.x) { found = true; break; }
                    s = (s + 1 == cap) ? 0 : s + 1;
                }
                if (!found) {
                    set_status(st, MWJ_ERR_CHECK, 5);
                    continue;
                }
                uint32_t p = atomicAdd(&sv[s], 1u);
                if (p >= o0 && p < o1) dlist[p] = (int32_t)t.y;
                else set_status(st, MWJ_ERR_CHECK, 6);
            }
            __syncthreads();
            for (uint32_t s = threadIdx.x; s < cap; s += BT) {
                unsigned long long v = reg[s];
                if (v != kEmpty64) sv[s] -= (uint32_t)(v >> 32);
            }
        }
        __syncthreads();
    }
}

}  // namespace

size_t single_table_slots(int64_t nT) {
    uint64_t cap = 16;
    while (cap < 2 * (uint64_t)(nT > 0 ? nT : 1)) cap <<= 1;
    return cap;
}

cudaError_t single_table_build(const uint32_t *keys, const uint32_t *off, uint32_t J, uint32_t seed,
                               uint32_t *ekey, uint32_t *ecnt, uint32_t *ecount, uint32_t *meta,
                               uint64_t *tbl, DevStatus *status, int num_sms, cudaStream_t st) {
    unsigned grid = J < (uint32_t)num_sms * 4 ? J : (unsigned)num_sms * 4;
    if (grid == 0) grid = 1;
    const size_t smem = 2 * (kAggSlots + 1) * sizeof(uint32_t);
    cudaError_t e = cudaFuncSetAttribute(k_tagg, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (J > 0) {
        ProfScope ps_("t_aggregate", st);
        k_tagg<<<grid, BT, smem, st>>>(keys, off, J, seed, ekey, ecnt, ecount, status);
    }
    {
        ProfScope ps_("t_size", st);
        k_tsize<<<1, 1024, 0, st>>>(ecount, J, meta);
    }
    {
        ProfScope ps_("t_clear", st);
        k_tclear<<<num_sms * 4, 512, 0, st>>>((unsigned long long *)tbl, meta);
    }
    if (J > 0) {
        ProfScope ps_("t_insert", st);
        k_tinsert<<<grid, BT, 0, st>>>(ekey, ecnt, off, ecount, J, seed, (unsigned long long *)tbl,
                                       meta, status);
    }
    return cudaGetLastError();
}

cudaError_t tables_build(const uint32_t *keys, const uint2 *pairs, const uint32_t *off, uint32_t J,
                         uint32_t seed, uint64_t *img, uint32_t *capv, uint32_t *startv,
                         int32_t *dlist, DevStatus *status, int num_sms, cudaStream_t st) {
    if (J == 0) return cudaSuccess;
    unsigned grid = J < (uint32_t)num_sms * 8 ? J : (unsigned)num_sms * 8;
    const size_t smem = kImgSmemSlots * sizeof(unsigned long long);
    cudaError_t e;
    if (startv) {
        e = cudaFuncSetAttribute(k_tbuild<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        ProfScope ps_("table_build_csr", st);
        k_tbuild<true><<<grid, BT, smem, st>>>(keys, pairs, off, J, seed,
                                               (unsigned long long *)img, capv, startv, dlist,
                                               status);
    } else {
        e = cudaFuncSetAttribute(k_tbuild<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        ProfScope ps_("table_build", st);
        k_tbuild<false><<<grid, BT, smem, st>>>(keys, pairs, off, J, seed,
                                                (unsigned long long *)img, capv, nullptr, nullptr,
                                                status);
    }
    return cudaGetLastError();
}

}  // namespace mwj

// ---------------------------------------------------------------------------
// single table without partitioning T: size it from a HyperLogLog estimate
// of T's distinct C values, then insert T's C column directly
// ---------------------------------------------------------------------------
namespace mwj {
namespace {

constexpr int HLL_BITS = 12;
constexpr uint32_t HLL_M = 1u << HLL_BITS;
constexpr int HLL_CTAS_PER_SM = 2;   // resident CTAs of the sizing passes (their registers allow two)
constexpr int RANGE_CTAS_PER_SM = 4;
constexpr uint32_t HLL_MB = 32;                  // registers merged per CTA
constexpr uint32_t HLL_MCTAS = HLL_M / HLL_MB;   // merge CTAs
// after the per-CTA registers: per merge CTA its part of the estimator's sum
// (double) and of the empty-register count, then the finish counter
constexpr size_t HLL_TAIL = 2 * HLL_MCTAS + HLL_MCTAS + 8;

// a column's scratch: `rows` x HLL_M registers, the merge's tail, `range_rows` (min, max) pairs
__device__ __forceinline__ unsigned int *size_tail(unsigned int *scratch, uint32_t rows) {
    return scratch + (size_t)rows * HLL_M;
}
__device__ __forceinline__ int32_t *size_ranges(unsigned int *scratch, uint32_t rows) {
    return (int32_t *)(size_tail(scratch, rows) + HLL_TAIL);
}

struct SizeArgs {
    SizeCol c[kSizeCols];
    HeavyCol h[kSizeCols];
    uint32_t nheavy, rows, range_rows;
    bool ranged;   // k_range has run: a compact column gets the direct-address layout
};

// Entries from lo to hi, 0 when there is none or they are more than `most` (or than
// 32 bits hold: a table of 2^32 entries has no span).
__device__ __forceinline__ uint32_t span_within(int32_t lo, int32_t hi, uint64_t most) {
    if (lo > hi) return 0u;
    const uint64_t span = (uint64_t)((int64_t)hi - (int64_t)lo + 1);
    return span <= most && span <= 0xFFFFFFFFull ? (uint32_t)span : 0u;
}

// Key range of every column: `rows` CTAs per column, each leaving the
// smallest and largest key it saw (INT32_MAX, INT32_MIN when it saw none).
// A pure stream, four 16-byte loads per thread in flight: 131 MB in 0.027 ms,
// where the HyperLogLog pass over the same column takes 0.037 ms (it hashes
// every key) and its merge 0.014 ms more; a column whose range is compact
// needs neither.  The first CTAs sample the heavy keys (skew.h) meanwhile.
__global__ void __launch_bounds__(BT, RANGE_CTAS_PER_SM) k_range(SizeArgs g) {
    after_previous();
    __shared__ HeavySample<2048> hsm;
    if (blockIdx.x < g.nheavy) {
        const HeavyCol &h = g.h[blockIdx.x];
        if (h.coarse)
            heavy_sample_cta<BT, 1024>(h.keys, h.n, h.buckets, h.heavy, reinterpret_cast<HeavySample<1024> &>(hsm));
        else
            heavy_sample_cta<BT, 2048>(h.keys, h.n, h.buckets, h.heavy, hsm);
        return;
    }
    const uint32_t cta = (blockIdx.x - g.nheavy) % g.range_rows;
    const SizeCol &c = g.c[(blockIdx.x - g.nheavy) / g.range_rows];
    const int32_t *keys = c.keys;
    const uint32_t n = c.n;
    int32_t lo = INT32_MAX, hi = INT32_MIN;
    auto see = [&](int32_t k) {
        lo = min(lo, k);
        hi = max(hi, k);
    };
    const uint32_t T = g.range_rows * BT, t = cta * BT + threadIdx.x;
    // the elements before the first 16-byte boundary and after the last one
    const uint32_t head = min(n, (uint32_t)(((16u - ((uintptr_t)keys & 15u)) & 15u) / 4u));
    const uint32_t quads = (n - head) / 4u;
    if (t < head) see(__ldg(keys + t));
    if (t < n - head - 4u * quads) see(__ldg(keys + head + 4u * quads + t));
    const int4 *v = (const int4 *)(keys + head);
    const uint64_t pol = l2_evict_first();
    // a thread whose keys already span more than every direct-address table stops: its
    // part of the range settles the layout
    uint64_t most = 0;
    for (uint32_t q = 0; q < c.ntargets; ++q) most = c.range[q] > most ? c.range[q] : most;
    const uint32_t wide = most > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)most;
    uint32_t i = t;
    for (; i < quads && quads - i > 3u * T; i += 4u * T) {
        if (lo < hi && (uint32_t)hi - (uint32_t)lo >= wide) break;
        int4 q[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) q[u] = ld_stream(v + i + u * T, pol);
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            lo = min(lo, min(min(q[u].x, q[u].y), min(q[u].z, q[u].w)));
            hi = max(hi, max(max(q[u].x, q[u].y), max(q[u].z, q[u].w)));
        }
    }
    for (; i < quads; i += T) {
        if (lo < hi && (uint32_t)hi - (uint32_t)lo >= wide) break;
        const int4 q = ld_stream(v + i, pol);
        see(q.x);
        see(q.y);
        see(q.z);
        see(q.w);
        if (quads - i <= T) break;   // (i + T may pass 2^32)
    }
    __shared__ int32_t slo[BT / 32], shi[BT / 32];
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
        slo[threadIdx.x >> 5] = lo;
        shi[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < BT / 32; ++w) {
            lo = min(lo, slo[w]);
            hi = max(hi, shi[w]);
        }
        int32_t *mm = size_ranges(c.scratch, g.rows);
        mm[2 * cta] = lo;
        mm[2 * cta + 1] = hi;
    }
}

// A star join's weights (SizeCol::spread): many tuples add to few keys, and adds
// that meet in an L2 line wait for one another.  Direct-address entries are set
// apart, up to a line of 16 for each, while the table takes at most 2^18 entries
// (2 MB): 2^26 facts on 1000, 3000 and 10,000 keys in no order take 2.03, 0.80 and
// 0.46 ms packed, 0.65, 0.58 and 0.36 a sector apart, 0.48, 0.35 and 0.29 a line
// apart.  Hashed tables get 16 slots a key up to 2^16 slots.
constexpr uint64_t kSpreadEntries = 1u << 18, kSpreadSlots = 1u << 16;
__device__ __forceinline__ uint32_t spread_shift(uint64_t span, uint64_t room) {
    uint32_t sh = 0;
    const uint64_t most = room < kSpreadEntries ? room : kSpreadEntries;
    while (sh < 4 && (span << (sh + 1)) <= most) ++sh;
    return sh;
}

// Slots from which a chain's weights are packed (linear_l2.h): 2^24 are more than the
// L2 holds.  Linear aggregates of 2^23 and 2^24 tuples on 0.63 times as many random
// keys take 0.87 and 2.20 ms with keys and sums apart, 0.66 and 1.62 packed; 6e6
// tuples (2^23 slots) 0.50 apart and, in packed slots of another load, 0.52.
constexpr uint64_t kPackedSlots = 1ull << 24;
// Distinct keys up to which a large range is direct-address, and one of up to `near`
// entries: 2^18 keys a line each are 32 MB a table (2.5e7 tuples over as many places,
// 2^16 and 2^18 keys 0.82 and 0.84 ms direct-address, 1.03 and 1.07 hashed).
constexpr double kFewKeys = 8192.0, kNearKeys = 1 << 18;

// HyperLogLog registers (Flajolet, Fusy, Gandouet, Meunier 2007): register
// h >> (32 - HLL_BITS) keeps the largest rank (position of the first 1 bit)
// of the remaining bits.  mix32 is a bijection of 32-bit keys, so distinct
// keys have distinct hashes.
//
// Blocks (x, y): column y.  With `ranged` every CTA first merges the column's
// key ranges: a table whose direct-address entries (range[q]) hold the whole
// range gets that layout (slot = key - min, no key stored) from the range alone
// when they are few, whatever share of them is used: only the entries of keys
// that occur are touched after the clear.  A column all of whose tables got it
// ends there.  A large range waits for the estimate: where its keys lie far apart
// every one takes an L2 line of its own, more than its hash slots do.  Linear
// GROUP BY of three relations of 2^24 tuples, 65,536 keys spread over 2^26 places:
// 1.19 ms direct-address, 0.72 hashed; 2^20 keys over 2^25 places 1.24 and 0.82, over
// 2^23 0.51 and 0.77; 2^22 keys over 2^25 (8 per key) 1.41 and 1.28.  With few keys
// the slots of a hash table are what the tuples wait for: 1000 keys over 2^26 places
// 0.79 and 1.42.
__global__ void __launch_bounds__(BT, HLL_CTAS_PER_SM) k_hll(SizeArgs g) {
    after_previous();
    __shared__ unsigned int r[HLL_M];
    const SizeCol &c = g.c[blockIdx.y];
    const int32_t *keys = c.keys;
    const uint32_t n = c.n, seed = c.seed;
    unsigned int *regs = c.scratch;
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    if (first) size_tail(c.scratch, g.rows)[3 * HLL_MCTAS] = 0;   // k_hll_merge_size's finish counter
    if (g.ranged) {
        __shared__ int32_t slo, shi;
        if (threadIdx.x == 0) {
            slo = INT32_MAX;
            shi = INT32_MIN;
        }
        __syncthreads();
        int32_t lo = INT32_MAX, hi = INT32_MIN;
        const int32_t *mm = size_ranges(c.scratch, g.rows);
        for (uint32_t b = threadIdx.x; b < g.range_rows; b += BT) {
            lo = min(lo, __ldcg(mm + 2 * b));
            hi = max(hi, __ldcg(mm + 2 * b + 1));
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&slo, lo);
            atomicMax(&shi, hi);
        }
        __syncthreads();
        lo = slo;
        hi = shi;
        bool all = true;
        for (uint32_t q = 0; q < c.ntargets; ++q) {
            const uint32_t span = span_within(lo, hi, c.range[q]);
            const bool dense = span != 0u && span <= c.sure;
            all = all && dense;
            if (first) {
                c.meta[q][kMetaDense] = dense ? 1u : 0u;
                c.meta[q][kMetaTry] = span != 0u && !dense ? 1u : 0u;
                if (span) {
                    c.meta[q][kMetaMask] = 15u;
                    c.meta[q][kMetaMin] = (uint32_t)lo;
                    c.meta[q][kMetaSpan] = span;
                    c.meta[q][kMetaShift] = spread_shift(span, c.spread);
                }
            }
        }
        if (all) return;
    } else if (first) {
        for (uint32_t q = 0; q < c.ntargets; ++q) c.meta[q][kMetaDense] = 0u;
    }
    for (uint32_t j = threadIdx.x; j < HLL_M; j += BT) r[j] = 0;
    __syncthreads();
    const bool vec = ((uintptr_t)keys & 15) == 0;
    const uint64_t pol = l2_evict_first();
    // strips of 16 consecutive keys, one per thread and iteration (four
    // 16-byte loads), so that a run of equal keys (edge lists come sorted by
    // source) costs one register update per strip: a register only grows, so
    // a key equal to its predecessor changes nothing.  The next strip's loads
    // are issued before this one is used.
    const uint32_t nst = (n + 15) / 16;
    const uint32_t T = gridDim.x * BT;
    auto load = [&](uint32_t c, int32_t (&v)[16]) -> uint32_t {
        if (c >= nst) return 0u;
        const uint32_t i = c * 16;
        const uint32_t cnt = min(16u, n - i);
        if (cnt == 16 && vec) {
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const int4 q = ld_stream((const int4 *)(keys + i) + g, pol);
                v[4 * g] = q.x; v[4 * g + 1] = q.y; v[4 * g + 2] = q.z; v[4 * g + 3] = q.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = ((uint32_t)k < cnt) ? __ldg(keys + i + k) : 0;
        }
        return cnt;
    };
    int32_t v[16];
    uint32_t st = blockIdx.x * BT + threadIdx.x;
    uint32_t cnt = load(st, v);
    for (; st < nst; st += T) {
        int32_t nv[16];
        const uint32_t ncnt = load(st + T, nv);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if ((uint32_t)k >= cnt) break;
            if (k > 0 && v[k] == v[k - 1]) continue;   // nothing a repeat could change
            const uint32_t h = mix32((uint32_t)v[k] ^ seed);
            const uint32_t w = h << HLL_BITS;
            const uint32_t rank = (w == 0) ? (33u - HLL_BITS) : (uint32_t)__clz(w) + 1u;
            unsigned int *reg = &r[h >> (32 - HLL_BITS)];
            if (*(volatile unsigned int *)reg < rank) atomicMax(reg, rank);
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = nv[k];
        cnt = ncnt;
    }
    __syncthreads();
    // this CTA's registers; the size kernel takes the maximum over CTAs
    for (uint32_t j = threadIdx.x; j < HLL_M; j += BT) regs[(size_t)blockIdx.x * HLL_M + j] = r[j];
}

// regs[0..HLL_M) = max over the rows of regs[ctas][HLL_M]
__global__ void k_hll_merge(unsigned int *__restrict__ regs, uint32_t ctas) {
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= HLL_M) return;
    unsigned int m = 0;
    for (uint32_t c = 0; c < ctas; ++c) m = max(m, regs[(size_t)c * HLL_M + j]);
    regs[j] = m;
}

// Merge a column's per-CTA registers (maximum over `rows` rows) into row 0
// and size its hashed tables: CTA b merges registers [32 b, 32 b + 32) and
// leaves its part of sum(2^-reg) and of the zero count; the last CTA to finish
// adds the parts in a fixed order (so the estimate does not depend on the
// finishing order) and writes meta: a table of 2^k >= factor x estimate slots,
// at most the reservation.  Blocks (x, y): column y.
constexpr int HLL_MW = 32;   // warps of a merge CTA, each over every HLL_MW-th row

__global__ void __launch_bounds__(HLL_MW * 32) k_hll_merge_size(SizeArgs g) {
    after_previous();
    const SizeCol &c = g.c[blockIdx.y];
    bool all = true;   // every table of the column is direct-address: nothing was counted
    for (uint32_t q = 0; q < c.ntargets; ++q) all = all && __ldcg(c.meta[q] + kMetaDense) != 0u;
    if (all) return;
    __shared__ unsigned int m[HLL_MW][HLL_MB];
    __shared__ bool last;
    unsigned int *regs = c.scratch;
    const uint32_t rows = g.rows;
    unsigned int *tail = size_tail(c.scratch, rows);
    double *part_s = (double *)tail;
    unsigned int *part_z = tail + 2 * HLL_MCTAS;
    unsigned int *done = part_z + HLL_MCTAS;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t j = blockIdx.x * HLL_MB + lane;
    // eight rows in flight per thread: the rows are independent loads
    unsigned int mx = 0;
    uint32_t r = w;
    for (; r + 7 * HLL_MW < rows; r += 8 * HLL_MW) {
        unsigned int v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcg(regs + (size_t)(r + HLL_MW * u) * HLL_M + j);
#pragma unroll
        for (int u = 0; u < 8; ++u) mx = max(mx, v[u]);
    }
    for (; r < rows; r += HLL_MW) mx = max(mx, __ldcg(regs + (size_t)r * HLL_M + j));
    m[w][lane] = mx;
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int q = 1; q < HLL_MW; ++q) mx = max(mx, m[q][lane]);
        regs[j] = mx;
        double sum = 1.0 / (double)(1ull << mx);   // exact: ranks are at most 33 - HLL_BITS
        unsigned int z = (mx == 0);
        for (int o = 16; o > 0; o >>= 1) {
            sum += __shfl_xor_sync(0xffffffffu, sum, o);
            z += __shfl_xor_sync(0xffffffffu, z, o);
        }
        if (lane == 0) {
            part_s[blockIdx.x] = sum;
            part_z[blockIdx.x] = z;
            __threadfence();
            last = atomicAdd(done, 1u) == gridDim.x - 1;
        }
    }
    __syncthreads();
    if (!last || w != 0) return;
    __threadfence();
    // the last CTA: the parts in a fixed order (lane l adds parts l, l + 32,
    // ... in turn, then a fixed butterfly)
    double S = 0.0;
    unsigned int Z = 0;
    for (uint32_t b = lane; b < gridDim.x; b += 32) {
        S += __ldcg(part_s + b);
        Z += __ldcg(part_z + b);
    }
    for (int o = 16; o > 0; o >>= 1) {
        S += __shfl_xor_sync(0xffffffffu, S, o);
        Z += __shfl_xor_sync(0xffffffffu, Z, o);
    }
    if (lane != 0) return;
    const double mm = (double)HLL_M;
    double E = (0.7213 / (1.0 + 1.079 / mm)) * mm * mm / S;
    if (E <= 2.5 * mm && Z > 0) E = mm * log(mm / (double)Z);   // small-range correction
    const double factor = kSingleTableFactor * E <= kSmallTableSlots ? kSingleTableFactor : kLargeTableFactor;
    for (uint32_t t = 0; t < c.ntargets; ++t) {
        uint32_t *mt = c.meta[t];
        if (__ldcg(mt + kMetaDense)) continue;
        const uint32_t span = g.ranged && __ldcg(mt + kMetaTry) ? __ldcg(mt + kMetaSpan) : 0u;
        if (span && ((double)span <= c.per_key * E || E <= kFewKeys || (span <= c.near && E <= kNearKeys))) {
            mt[kMetaDense] = 1u;   // (the other words are there)
            continue;
        }
        // 2^31 slots hold the keys of any relation; masks of 32 ones are none
        const uint64_t res = c.reserve[t] < (1ull << 31) ? c.reserve[t] : 1ull << 31;
        uint64_t cap = 16;
        while ((double)cap < factor * E && cap < res) cap <<= 1;
        if (cap > res) cap = res;
        while ((double)cap < 16.0 * E && 2 * cap <= kSpreadSlots && 2 * cap <= c.spread) cap <<= 1;
        if (g.ranged) mt[kMetaPacked] = c.weights && cap >= kPackedSlots ? 1u : 0u;
        mt[kMetaMask] = (uint32_t)(cap - 1);
        mt[kMetaEst] = (uint32_t)E;
    }
    *done = 0;
}

// Empty the tables that the sizing passes laid out (blocks (x, y): table y)
// and zero the call's outputs (y = ntables).
struct ClearArgs {
    ClearTable t[kSizeCols];
    uint32_t ntables;
    unsigned long long *zero, *total;
    uint64_t nzero;
};

__global__ void __launch_bounds__(BT) k_tables_clear(ClearArgs g) {
    after_previous();
    const uint64_t i0 = (uint64_t)blockIdx.x * BT + threadIdx.x, stride = (uint64_t)gridDim.x * BT;
    if (blockIdx.y == g.ntables) {
        for (uint64_t i = i0; i < g.nzero; i += stride) g.zero[i] = 0ull;
        if (i0 == 0 && g.total) *g.total = 0ull;
        return;
    }
    const ClearTable &t = g.t[blockIdx.y];
    const bool dense = t.meta[kMetaDense] != 0u;
    // arrays are 256-byte aligned and have two spare entries
    if (t.keys == nullptr) {   // degrees: u32 entries, or packed hashed slots
        const uint64_t words = dense ? (uint64_t)t.meta[kMetaSpan] / 2 + 1 : (uint64_t)t.meta[kMetaMask] + 1;
        const unsigned long long fill = dense ? 0ull : kEmpty64;
        for (uint64_t s = i0; s < (words + 1) / 2; s += stride) ((ulonglong2 *)t.tbl)[s] = make_ulonglong2(fill, fill);
        return;
    }
    // weights: zero sums (hashed: of slot mask + 1, key -1, too), free keys
    const uint64_t sums = dense ? (uint64_t)t.meta[kMetaSpan] << t.meta[kMetaShift] : (uint64_t)t.meta[kMetaMask] + 2;
    const bool packed = !dense && (t.meta[kMetaPacked] & 1u);
    const unsigned long long fill = packed ? kEmpty64 : 0ull;
    const uint64_t filled = packed ? sums - 1 : sums;   // (key -1's sum is a plain one)
    for (uint64_t s = i0; s < (filled + 1) / 2; s += stride) ((ulonglong2 *)t.tbl)[s] = make_ulonglong2(fill, fill);
    if (packed && i0 == 0) t.tbl[sums - 1] = 0ull;
    if (dense) return;
    const uint32_t u = packed ? 0u : kEmptyKey;
    const uint4 keys4 = make_uint4(u, u, u, u);
    for (uint64_t s = i0; s < ((uint64_t)t.meta[kMetaMask] + 1) / 4; s += stride) ((uint4 *)t.keys)[s] = keys4;
}

// Insert T's C column.  A warp round is four blocks of 128 consecutive keys
// (four per lane), all loaded, with the next round's loads issued, before
// they are used; every run of equal keys in a block is measured once by
// warp_run_lengths and added to its slot once, the first probes of a lane's
// four keys issued together.
__global__ void __launch_bounds__(BT, 2) k_tinsert_direct(const int32_t *__restrict__ keys, uint32_t n,
                                                          uint32_t seed, unsigned long long *__restrict__ tbl,
                                                          const uint32_t *__restrict__ meta, DevStatus *st) {
    const uint32_t mask = meta[0];
    const bool vec = ((uintptr_t)keys & 15) == 0;
    const uint64_t pol = l2_evict_first();
    constexpr uint32_t CH = 32 * kRunQ;   // keys of one block
    constexpr int G = 4;                  // blocks per warp round, loaded together
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * BT + threadIdx.x) >> 5, warps = (gridDim.x * BT) >> 5;
    const uint32_t blocks = (n + CH - 1) / CH;
    const uint32_t rounds = (blocks + G - 1) / G;
    auto load = [&](uint32_t blk, int32_t (&v)[kRunQ]) -> uint32_t {
        const uint32_t i = blk * CH + lane * kRunQ;
        if (blk >= blocks || i >= n) return 0u;
        if (vec && i + kRunQ <= n) {
            const int4 a = ld_stream((const int4 *)(keys + i), pol);
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
            return kRunQ;
        }
        const uint32_t m = min((uint32_t)kRunQ, n - i);
#pragma unroll
        for (int q = 0; q < kRunQ; ++q)
            if ((uint32_t)q < m) v[q] = __ldg(keys + i + q);
        return m;
    };
    auto insert_block = [&](const int32_t (&v)[kRunQ], uint32_t m) {
        uint32_t len[kRunQ] = {0u, 0u, 0u, 0u};
        warp_run_lengths(v, m, [&](int q, int32_t, uint32_t l) { len[q] = l; });
        uint32_t s[kRunQ];
        unsigned long long x[kRunQ];
#pragma unroll
        for (int q = 0; q < kRunQ; ++q) {
            if (len[q]) {
                s[q] = slot_of((uint32_t)v[q], seed, mask);
                x[q] = __ldcg(tbl + s[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < kRunQ; ++q)
            if (len[q]) single_insert_from(tbl, mask, (uint32_t)v[q], s[q], x[q], len[q], st);
    };
    int32_t v[G][kRunQ];
    uint32_t m[G];
    uint32_t r = warp;
#pragma unroll
    for (int g = 0; g < G; ++g) m[g] = load(r * G + g, v[g]);
    while (r < rounds) {
        const uint32_t nr = r + warps;
        int32_t nv[G][kRunQ];
        uint32_t nm[G];
#pragma unroll
        for (int g = 0; g < G; ++g) nm[g] = load(nr * G + g, nv[g]);
#pragma unroll
        for (int g = 0; g < G; ++g) insert_block(v[g], m[g]);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            m[g] = nm[g];
#pragma unroll
            for (int q = 0; q < kRunQ; ++q) v[g][q] = nv[g][q];
        }
        r = nr;
    }
}

}  // namespace

cudaError_t size_columns(const SizeCol *cols, uint32_t ncols, const HeavyCol *heavy, uint32_t nheavy, bool allow_dense,
                         int num_sms, cudaStream_t st, const char *hll_name, const char *size_name) {
    SizeArgs g{};
    for (uint32_t q = 0; q < ncols; ++q) g.c[q] = cols[q];
    for (uint32_t q = 0; q < nheavy; ++q) g.h[q] = heavy[q];
    g.nheavy = nheavy;
    g.rows = (uint32_t)num_sms * HLL_CTAS_PER_SM;
    // CTAs of a column's range pass: every one with four loads per thread
    uint32_t most = 1;
    for (uint32_t q = 0; q < ncols; ++q) most = cols[q].n > most ? cols[q].n : most;
    const uint32_t want = (most + 16u * BT - 1) / (16u * BT), full = (uint32_t)num_sms * RANGE_CTAS_PER_SM;
    g.range_rows = want < full ? want : full;
    g.ranged = allow_dense;
    if (allow_dense) {
        ProfScope ps_("key_range", st);
        const cudaError_t e = launch_after(k_range, nheavy + ncols * g.range_rows, BT, st, g);
        if (e != cudaSuccess) return e;
    }
    {
        ProfScope ps_(hll_name, st);
        const cudaError_t e = launch_after(k_hll, dim3(g.rows, ncols), BT, st, g);
        if (e != cudaSuccess) return e;
    }
    ProfScope ps_(size_name, st);
    return launch_after(k_hll_merge_size, dim3(HLL_MCTAS, ncols), HLL_MW * 32, st, g);
}

cudaError_t tables_clear(const ClearTable *t, uint32_t n, unsigned long long *zero, uint64_t nzero,
                         unsigned long long *total, int num_sms, cudaStream_t st) {
    ClearArgs g{};
    for (uint32_t q = 0; q < n; ++q) g.t[q] = t[q];
    g.ntables = n;
    g.zero = zero;
    g.nzero = nzero;
    g.total = total;
    ProfScope ps_("tables_clear", st);
    return launch_after(k_tables_clear, dim3(num_sms * 2, n + ((nzero || total) ? 1u : 0u)), BT, st, g);
}

cudaError_t single_table_size(const int32_t *keys, int64_t n, uint32_t seed, unsigned int *hll_regs,
                              uint32_t *meta, uint64_t reserve_slots, int num_sms, cudaStream_t st,
                              const char *hll_name, const char *size_name, bool allow_dense) {
    SizeCol c{keys, (uint32_t)n, seed, hll_regs, {meta}, {reserve_slots}, {reserve_slots}, 1u};
    return size_columns(&c, 1, nullptr, 0, allow_dense, num_sms, st, hll_name, size_name);
}

cudaError_t single_table_direct(const int32_t *keys, int64_t n, uint32_t seed, unsigned int *hll_regs,
                                uint32_t *meta, uint64_t *tbl, uint64_t reserve_slots,
                                DevStatus *status, int num_sms, cudaStream_t st) {
    cudaError_t e;
    if ((e = single_table_size(keys, n, seed, hll_regs, meta, reserve_slots, num_sms, st)) != cudaSuccess) return e;
    {
        ProfScope ps_("t_clear", st);
        k_tclear<<<num_sms * 4, 512, 0, st>>>((unsigned long long *)tbl, meta);
    }
    const uint32_t nn = (uint32_t)n;
    if (nn > 0) {
        ProfScope ps_("t_insert", st);
        const uint32_t groups = (nn + 4 * kRunQ * BT - 1) / (4 * kRunQ * BT);
        const uint32_t grid = groups < (uint32_t)num_sms * 4 ? groups : (uint32_t)num_sms * 4;
        k_tinsert_direct<<<grid, BT, 0, st>>>(keys, nn, seed, (unsigned long long *)tbl, meta, status);
    }
    return cudaGetLastError();
}

uint32_t hll_registers() { return HLL_M; }

cudaError_t hll_regs(const int32_t *keys, int64_t n, uint32_t seed, unsigned int *regs, int num_sms,
                     cudaStream_t st) {
    cudaError_t e;
    if (n > 0) {
        const uint32_t ctas = (uint32_t)num_sms * HLL_CTAS_PER_SM;
        {
            ProfScope ps_("sketch_hll", st);
            SizeArgs g{};
            g.c[0] = SizeCol{keys, (uint32_t)n, seed, regs, {nullptr}, {0}, {0}, 0u};
            g.rows = ctas;
            k_hll<<<ctas, BT, 0, st>>>(g);
        }
        ProfScope ps_("sketch_hll_merge", st);
        k_hll_merge<<<(HLL_M + 255) / 256, 256, 0, st>>>(regs, ctas);
    } else if ((e = cudaMemsetAsync(regs, 0, HLL_M * sizeof(unsigned int), st)) != cudaSuccess) {
        return e;
    }
    return cudaGetLastError();
}

size_t hll_scratch_registers(int num_sms) {
    const size_t ctas = (size_t)num_sms * HLL_CTAS_PER_SM;
    // registers, sizing tail, per-CTA key ranges
    return ctas * HLL_M + HLL_TAIL + 2 * (size_t)num_sms * RANGE_CTAS_PER_SM;
}

}  // namespace mwj
