// cyclic_c.cu -- the cyclic 3-way join R(A,B) S(B,C) T(C,A) with R whole and
// C split into buckets: shares (1, 1, z) (Section 5).
//
// Section 5 keeps R's (H(a), G(b)) buckets on chip and streams S and T past
// them; with cube shares (x, y, z) a tile (i, j, k) holds R_ij and T_ki in a
// CTA's shared memory and streams S_jk (cyclic.cu).  On a large graph the
// tiles that fit shared memory are so small -- millions of them -- that
// rebuilding their tables costs far more than the wedge checks.  This plan
// follows the two levels of on-chip memory of the GPU instead: R stays whole,
// grouped by B (b -> [a], in global memory and read through the L2 by every
// SM), and only C is split: T by F(c) into z buckets whose (c, a) multiset
// fits one CTA's shared memory, S by F(c) into the same buckets.  A CTA takes
// bucket k, builds T_k's set on chip and streams S_k past it: per S tuple
// (b, c) it visits every a of R[b] and counts (c, a) in the set.  These are
// the cube tiling's wedge checks, each wedge of R |x| S once, without the
// per-tile rebuilds.  A bucket whose T_k exceeds a CTA's shared-memory set
// is taken in chunks of it, S_k streamed past each (every chunk checks the
// bucket's wedges again, against its part of T_k); one above CC_TBIG tuples
// (a C value with many T tuples: skewed or tiny C domains) keeps its set in an
// L2-resident region of the workspace instead, built before the probe, so
// that its wedges are checked once.  Results do not depend on z.
#include "api_internal.h"
#include "cyclic.h"
#include "rgroup.cuh"
#include "tables.h"

namespace mwj {
namespace {

constexpr int CC_T = 640;                // threads per probe CTA (two CTAs per SM)
constexpr uint32_t CC_TAVG = 2048;       // T tuples of an average bucket under the default shares
constexpr uint32_t CC_TCAP = 6144;       // T tuples of an on-chip set: it is at most 3/4 full
constexpr uint32_t CC_TBIG = 16384;      // T tuples of a bucket above which its set moves to the L2
constexpr uint32_t CC_TSLOTS = 8192;     // slots of an on-chip (c, a) multiset (64 KB)
constexpr uint32_t CC_FWORDS = 8192;     // words of the filter in front of it (2^18 bits, 32 KB)
constexpr int RG_T = 512;                // threads of the grouping kernels
constexpr uint32_t CC_QCAP = 768;        // long R lists queued per work item
constexpr uint32_t CC_CH = 1024;         // wedges of a list per warp step (32 per lane, one mask word)
// lists this long go to the item's queue, so that a hub is shared by the CTA's warps
// (probe of the 2^22-vertex graph, lists up to 4096: 21.0 ms from 512 on, 20.7 from
// 1024, 20.4 from 2048 or none)
constexpr uint32_t kQueueMin = 2048;
// An item of few S tuples (no more than the queue has places) has about as many
// batches as warps or fewer: there lists of kFewMin entries go to the queue
// already, and are shared in pieces of kFewStep.  Three relations of 1e4 tuples,
// Zipf 1.1 (lists of 1300 in items of 32 tuples): 0.63 ms with one limit of 2048,
// 0.17 with the two; 6e4 tuples on 300 keys (lists of 200) 0.47 and 0.18.
constexpr uint32_t kFewMin = 128, kFewStep = 512;
static_assert((uint64_t)CC_QCAP * ((1ull << 31) / kFewStep + 1) < 1ull << 32, "the queue's pieces are counted in 32 bits");
constexpr uint32_t CC_STAGE = 32;        // rows that a warp of the row pass stages
constexpr uint32_t CC_QCAP_ROWS = 384;   // its queue's places: the rest hold the staged rows
constexpr uint32_t kTurned = 0x80000000u;   // row output: mark of a turned tuple, in its list's start
constexpr uint32_t CC_SCHUNK_MIN = 32;   // S tuples of a bucket's work item, at least (a warp's batch)

__device__ __forceinline__ unsigned long long cpack(uint32_t c, uint32_t a) {
    return ((unsigned long long)c << 32) | a;
}

// An on-chip (c, a) set: CC_TSLOTS / 2 buckets of two 8-byte slots (16
// bytes, one shared-memory load), one slot per distinct pair.  An insert
// takes the first slot of its home bucket or of the buckets after it that is
// free or holds its pair, so the occupied slots of a bucket are a prefix and
// a lookup can stop at the first bucket with a free slot.  T is a bag: a
// chunk that repeats a pair (rare) is rebuilt in the CTA's own region of the
// workspace with a multiplicity per slot and looked up there like a big
// bucket's set.
//
// Nearly every wedge is open (about 1 in 40 of the shorter lists' closes on the
// 2^22-vertex power-law graph), so the set is not looked up per wedge: a filter
// of 2^18 bits, two bits of one word per (c, a) pair, answers first.  The bits
// of a wedge are a multiply-add of its a (the hash of c is computed once per
// list), one 4-byte shared-memory load and two shifts, with no probe chain
// whose longest lane the whole warp waits for; the set is looked up for what
// passes (2048 pairs leave 0.1 % of the open wedges standing, 6144 pairs 0.5 %;
// with one bit per pair 0.8 and 2.3 %).  On the 2^22-vertex graph (2.79e10
// wedges, one GB300) the probe took 122 ms when it looked every wedge up in the
// set, 38 with one bit, 24.4 from the shorter lists, 21.2 with 16-byte loads and
// the second bit, and 20.4 with fewer lists queued.  Issue slots bound it (73 %
// taken), and the 3.5 shared-memory wavefronts of a divergent load.
constexpr uint32_t CC_NB = CC_TSLOTS / 2;
constexpr int CC_MAX_CTAS_PER_SM = 2;   // probe CTAs per SM (shared memory); one region each
// two probe CTAs per SM: each keeps below half of the SM's 228 KB of shared
// memory less the 1 KB the hardware reserves per CTA and the static arrays
static_assert(CC_TSLOTS * 8 + CC_FWORDS * 4 + CC_QCAP * 16 + (CC_QCAP + 1) * 4 + 1024 <= 228 * 1024 / 2 - 1024,
              "the probe's shared memory must leave room for two CTAs per SM");

// The filter bits of (c, a): word h >> 19, bits (h >> 14) & 31 and h & 31 from
// the top, of h = a * K + chash(c), so that only the multiply-add depends on a.
// (h & 31 says no more than a's low five bits, and takes no shift: 21.2 ms, with
// (h >> 9) & 31 21.6.)
constexpr uint32_t CC_FMUL = 0x9E3779B1u;
static_assert(CC_FWORDS == 1u << 13, "the filter's word index is the top 13 bits");
__device__ __forceinline__ uint32_t chash(uint32_t c, uint32_t seed) { return mix32(c ^ seed); }

__device__ __forceinline__ uint32_t chash_a(uint32_t a, uint32_t ch) { return a * CC_FMUL + ch; }
// the home bucket of (c, a) in the on-chip set
static_assert(CC_NB == 1u << 12, "the home bucket is the top 12 bits");
__device__ __forceinline__ uint32_t cbucket(uint32_t h) { return h >> 20; }

__device__ __forceinline__ void fset(uint32_t *filt, uint32_t h) {
    atomicOr(filt + (h >> 19), (0x80000000u >> ((h >> 14) & 31u)) | (0x80000000u >> (h & 31u)));
}
// on top of a word: whether both are set (shifts take their amount modulo 32)
__device__ __forceinline__ uint32_t ftop(const uint32_t *filt, uint32_t a, uint32_t ch) {
    const uint32_t h = chash_a(a, ch);
    const uint32_t w = filt[h >> 19];
    return __funnelshift_l(0u, w, h >> 14) & __funnelshift_l(0u, w, h);
}

// 1: the pair took a free slot; 2: it was there already; 0: the set is full.
__device__ __forceinline__ int cset_insert(unsigned long long *tk, unsigned long long key, uint32_t bk) {
    for (uint32_t it = 0; it < CC_NB; ++it) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            unsigned long long *p = tk + 2 * bk + q;
            unsigned long long v = *p;
            if (v == kEmpty64) {
                v = atomicCAS(p, kEmpty64, key);
                if (v == kEmpty64) return 1;
            }
            if (v == key) return 2;
        }
        bk = (bk + 1) & (CC_NB - 1);
    }
    return 0;
}

// 1 when key is in the set, else 0 (key != kEmpty64)
__device__ __forceinline__ uint32_t cset_count(const unsigned long long *tk, unsigned long long key, uint32_t bk) {
    for (uint32_t it = 0; it < CC_NB; ++it) {
        const ulonglong2 v = *(const ulonglong2 *)(tk + 2 * bk);
        if (v.x == key || v.y == key) return 1u;
        if (v.y == kEmpty64) break;   // (v.x empty implies v.y empty)
        bk = (bk + 1) & (CC_NB - 1);
    }
    return 0u;
}

__global__ void k_rg_clear(RGroup r, unsigned int *__restrict__ bump) {
    after_previous();
    if (blockIdx.x == 0 && threadIdx.x == 0) *bump = 0u;
    const uint32_t *meta = r.meta;
    const uint32_t n = rg_entries(meta);
    const bool hashed = meta[kMetaDense] == 0u;
    const uint32_t mask = meta[kMetaMask];
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        r.deg[i] = 0u;
        if (hashed) r.keys[i] = (i <= mask) ? kEmptyKey : 0u;
    }
}

// deg[index(b)] += 1 for every (a, b) of R (the hashed layout inserts b);
// with a_domain > 0 every a must lie in [0, a_domain).
__global__ void __launch_bounds__(RG_T) k_rg_count(const int32_t *__restrict__ Ra, const int32_t *__restrict__ Rb,
                                                   uint32_t n, RGroup r, int32_t a_domain, DevStatus *st) {
    after_previous();
    const uint32_t *meta = r.meta;
    const bool dense = meta[kMetaDense] != 0u;
    const uint32_t kmin = meta[kMetaMin], span = meta[kMetaSpan], mask = meta[kMetaMask];
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int32_t a = __ldg(Ra + i);
        const uint32_t b = (uint32_t)__ldg(Rb + i);
        if (a_domain > 0 && (uint32_t)a >= (uint32_t)a_domain) set_status(st, MWJ_ERR_DOMAIN, a);
        int idx;
        if (dense) {
            idx = (b - kmin < span) ? (int)(b - kmin) : -1;
        } else {
            bool fresh;
            idx = tbl_insert(r.keys, mask, b, r.seed, &fresh);
        }
        if (idx >= 0)
            atomicAdd(r.deg + idx, 1u);
        else
            set_status(st, MWJ_ERR_CHECK, 21);   // outside the sized range / table full
    }
}

// end[i] = start of entry i's list (block-aggregated bump allocation: the
// lists are contiguous per key, in no particular key order); the scatter
// advances end[i] to the list's end.
__global__ void __launch_bounds__(RG_T) k_rg_offsets(RGroup r, unsigned int *__restrict__ bump) {
    after_previous();
    __shared__ uint32_t scratch[33];
    __shared__ uint32_t base;
    const uint32_t n = rg_entries(r.meta);
    for (uint32_t b0 = blockIdx.x * RG_T; b0 < n; b0 += gridDim.x * RG_T) {
        const uint32_t i = b0 + threadIdx.x;
        const uint32_t d = i < n ? r.deg[i] : 0u;
        uint32_t tot;
        const uint32_t ex = block_excl_scan_u32(d, scratch, &tot);
        if (threadIdx.x == 0) base = tot ? atomicAdd(bump, tot) : 0u;
        __syncthreads();
        if (i < n) r.end[i] = base + ex;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(RG_T) k_rg_scatter(const int32_t *__restrict__ Ra,
                                                     const int32_t *__restrict__ Rb, uint32_t n, RGroup r,
                                                     uint32_t nR, DevStatus *st) {
    after_previous();
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int idx = rg_find(r, r.meta, (uint32_t)__ldg(Rb + i));
        if (idx < 0) {
            set_status(st, MWJ_ERR_CHECK, 22);
            continue;
        }
        const uint32_t p = atomicAdd(r.end + idx, 1u);
        if (p < nR)
            r.alist[p] = __ldg(Ra + i);
        else
            set_status(st, MWJ_ERR_CHECK, 23);
    }
}

// Self-joins (T's pairs are R's, T.x = R.y and T.y = R.x, as in triangle
// counting): R's lists b -> [a] are T's lists c -> [a] too, and R's sets are
// T's.  Then the wedges of an S tuple (b, c) may be enumerated from either
// end -- R[b]'s a checked against c's set or T[c]'s a against b's -- and each
// tuple is turned so that its first column is the end with the shorter list:
// sum of min(|R[b]|, |T[c]|) wedges instead of sum of |R[b]| (0.42 of them on the
// power-law graphs).  Two list lengths per tuple, read in one pass over S
// (0.34 ms for 6.7e7 tuples); the probe goes from 38 to 25 ms on the
// 2^22-vertex graph, the call from 45 to 31.  Row output carries a mark of the
// turned tuples: 7.6e6 triangles of a 2^20-vertex graph, with the sort of the
// rows, 7.3 to 6.4 ms (when every wedge was still enumerated twice).
__global__ void __launch_bounds__(RG_T) k_cc_orient(const int32_t *__restrict__ Sb, const int32_t *__restrict__ Sc,
                                                    uint32_t n, RGroup r, int32_t *__restrict__ u,
                                                    int32_t *__restrict__ v, int32_t *__restrict__ turned) {
    after_previous();
    constexpr uint32_t Q = 4;
    const uint32_t T = gridDim.x * RG_T;
    auto length = [&](uint32_t k) -> uint32_t {
        const int e = rg_find(r, r.meta, k);
        return e >= 0 ? __ldg(r.deg + e) : 0u;
    };
    for (uint64_t i = (uint64_t)blockIdx.x * RG_T + threadIdx.x; i < n; i += Q * T) {
        int32_t b[Q], c[Q];
        uint32_t lb[Q], lc[Q];
#pragma unroll
        for (uint32_t q = 0; q < Q; ++q) {
            b[q] = i + q * T < n ? __ldg(Sb + i + q * T) : 0;
            c[q] = i + q * T < n ? __ldg(Sc + i + q * T) : 0;
        }
#pragma unroll
        for (uint32_t q = 0; q < Q; ++q) {
            lb[q] = length((uint32_t)b[q]);
            lc[q] = length((uint32_t)c[q]);
        }
#pragma unroll
        for (uint32_t q = 0; q < Q; ++q) {
            if (i + q * T >= n) continue;
            const bool turn = lc[q] < lb[q];
            u[i + q * T] = turn ? c[q] : b[q];
            v[i + q * T] = turn ? b[q] : c[q];
            if (turned) turned[i + q * T] = turn;
        }
    }
}

__host__ __device__ __forceinline__ bool cc_big(uint32_t nt) { return nt > CC_TBIG; }

// S chunks of a bucket: S_k in pieces of at most schunk tuples
__host__ __device__ __forceinline__ uint32_t cc_schunks(uint32_t ns, uint32_t schunk) {
    return (ns + schunk - 1) / schunk;
}

// Work items of a bucket whose S_k and T_k are both non-empty: each of its
// T chunks (on-chip sets; one set when the bucket is big, cc_big) with each
// of its S chunks, item (t, s) at t * S chunks + s; a big bucket also gets a
// region of 2^k >= 2 |T_k| slots for its set in the workspace (big_slots[k],
// 0 for the others).
//
// Buckets are taken in the order of four classes of |S_k| (4x, 2x, 1.25x the
// mean and the rest): a hub's C value makes an item of some 3 ms where the
// mean item takes 0.3 ms (2^22-vertex power-law graph), and one that starts
// last leaves every other SM idle for as long.  order[p] is the bucket at
// position p, items[p] its item count.  One CTA (z <= 32768).
constexpr int CC_PLAN_T = 1024;
__device__ __forceinline__ uint32_t cc_class(uint32_t ns, uint32_t mean) {
    return ns >= 4u * mean ? 0u : ns >= 2u * mean ? 1u : 4ull * ns >= 5ull * mean ? 2u : 3u;
}

__global__ void __launch_bounds__(CC_PLAN_T) k_cc_plan(const uint32_t *__restrict__ offS,
                                                       const uint32_t *__restrict__ offT, uint32_t z,
                                                       uint32_t schunk, uint32_t *__restrict__ items,
                                                       uint32_t *__restrict__ order,
                                                       unsigned long long *__restrict__ big_slots) {
    after_previous();
    __shared__ uint32_t cursor[4];
    if (threadIdx.x < 4) cursor[threadIdx.x] = 0u;
    __syncthreads();
    const uint32_t mean = (offS[z] - offS[0]) / z + 1u;
    uint32_t mine[4] = {0u, 0u, 0u, 0u};
    for (uint32_t k = threadIdx.x; k < z; k += CC_PLAN_T) {
        const uint32_t ns = offS[k + 1] - offS[k], nt = offT[k + 1] - offT[k];
        const uint32_t c = cc_class(ns, mean);
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) mine[q] += c == q;
        unsigned long long slots = 0;
        if (ns && cc_big(nt)) {
            slots = 16;
            while (slots < 2ull * nt) slots <<= 1;
        }
        big_slots[k] = slots;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        mine[q] = warp_sum(mine[q]);
        if ((threadIdx.x & 31) == 0 && mine[q]) atomicAdd(&cursor[q], mine[q]);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t at = 0;
        for (int q = 0; q < 4; ++q) {
            const uint32_t n = cursor[q];
            cursor[q] = at;
            at += n;
        }
    }
    __syncthreads();
    for (uint32_t k = threadIdx.x; k < z; k += CC_PLAN_T) {
        const uint32_t ns = offS[k + 1] - offS[k], nt = offT[k + 1] - offT[k];
        const uint32_t p = atomicAdd(&cursor[cc_class(ns, mean)], 1u);
        order[p] = k;
        items[p] = (ns && nt) ? (cc_big(nt) ? 1u : (nt + CC_TCAP - 1) / CC_TCAP) * cc_schunks(ns, schunk) : 0u;
    }
}

// Empty every big bucket's region and zero its counts (the total is the
// scan's last entry).
__global__ void k_cc_bigclear(unsigned long long *__restrict__ gs, uint32_t *__restrict__ gc,
                              const unsigned long long *__restrict__ big_off, uint32_t z) {
    after_previous();
    const unsigned long long total = big_off[z];
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        gs[i] = kEmpty64;
        gc[i] = 0u;
    }
}

__device__ __forceinline__ uint32_t gslot(uint32_t c, uint32_t a, uint32_t seed) {
    uint32_t h = (c ^ seed) * 0x85EBCA6Bu ^ a * 0x9E3779B1u;
    h ^= h >> 15;
    h *= 0x846ca68bU;
    h ^= h >> 16;
    return h;
}

// Big buckets' sets: a CTA per bucket (buckets blockIdx.x, + gridDim.x, ...)
// inserts T_k's (c, a) pairs into the bucket's region, one slot per distinct
// pair (linear probing from gslot) and its multiplicity in gc at the same
// index; (-1, -1) pairs are counted in big_neg[k].
__global__ void k_cc_bigbuild(const uint2 *__restrict__ Tp, const uint32_t *__restrict__ offT, uint32_t z,
                              const unsigned long long *__restrict__ big_off, unsigned long long *__restrict__ gs,
                              uint32_t *__restrict__ gc, uint32_t *__restrict__ big_neg, uint32_t seed,
                              DevStatus *st) {
    after_previous();
    __shared__ uint32_t negs;
    for (uint32_t k = blockIdx.x; k < z; k += gridDim.x) {
        const unsigned long long base = big_off[k], slots = big_off[k + 1] - base;
        if (slots == 0) continue;
        if (threadIdx.x == 0) negs = 0u;
        __syncthreads();
        const uint32_t mask = (uint32_t)(slots - 1);
        unsigned long long *reg = gs + base;
        uint32_t *cnt = gc + base;
        for (uint32_t q = offT[k] + threadIdx.x; q < offT[k + 1]; q += blockDim.x) {
            const uint2 tu = __ldg(Tp + q);
            const unsigned long long key = cpack(tu.x, tu.y);
            if (key == kEmpty64) {
                atomicAdd(&negs, 1u);
                continue;
            }
            uint32_t s = gslot(tu.x, tu.y, seed) & mask;
            bool done = false;
            for (uint32_t it = 0; it <= mask; ++it) {
                unsigned long long v = reg[s];
                if (v == kEmpty64) v = atomicCAS(reg + s, kEmpty64, key);   // kEmpty64: claimed here
                if (v == kEmpty64 || v == key) {
                    atomicAdd(cnt + s, 1u);
                    done = true;
                    break;
                }
                s = (s + 1) & mask;
            }
            if (!done) set_status(st, MWJ_ERR_CHECK, 26);
        }
        __syncthreads();
        if (threadIdx.x == 0) big_neg[k] = negs;
        __syncthreads();
    }
}

// Persistent kernel over the work items (bucket, chunk): counts (COUNT, GROUP
// BY A), or writes rows.  A warp's rows are staged in shared memory and go out
// about 32 at a time, at positions that one atomic on the number of rows
// reserves; rows past the capacity are counted only.  (Counting first and
// enumerating the wedges again to write: 4.0 ms for 7.6e6 rows of 1.3e7
// edges; now 1.9.  Positions straight from the one counter would be an
// atomic on one address per warp step that finds a triangle.)
template <bool ROWS>
__global__ void __launch_bounds__(CC_T, CC_MAX_CTAS_PER_SM) k_cc_probe(CycCArgs g, const uint32_t *__restrict__ item_off,
                                                      unsigned int *__restrict__ counter,
                                                      unsigned long long *__restrict__ n_rows,
                                                      int32_t *__restrict__ rows, unsigned long long capacity,
                                                      unsigned long long *__restrict__ rep_set,
                                                      uint32_t *__restrict__ rep_cnt) {
    after_previous();
    extern __shared__ __align__(16) unsigned char smraw[];
    unsigned long long *tk = (unsigned long long *)smraw;                      // CC_TSLOTS
    uint32_t *filt = (uint32_t *)(tk + CC_TSLOTS);                              // CC_FWORDS
    uint4 *queue = (uint4 *)(filt + CC_FWORDS);                                 // CC_QCAP x (b, c, start, n)
    constexpr uint32_t QCAP = ROWS ? CC_QCAP_ROWS : CC_QCAP;
    uint32_t *cpre = (uint32_t *)(queue + QCAP);                                // QCAP + 1 chunk offsets
    int32_t *stage = (int32_t *)(cpre + QCAP + 1) + (threadIdx.x >> 5) * (3 * CC_STAGE);   // the warp's rows
    uint32_t staged = 0;
    __shared__ uint32_t item_s, tneg, batch_ctr, chunk_ctr, qn, carry, tdup;
    // this CTA's region for a chunk that repeats pairs
    unsigned long long *const my_set = rep_set + (size_t)blockIdx.x * CC_TSLOTS;
    uint32_t *const my_cnt = rep_cnt + (size_t)blockIdx.x * CC_TSLOTS;
    __shared__ uint32_t scan_scratch[33];
    __shared__ unsigned long long red[32];
    const uint32_t z = g.z;
    const uint32_t total_items = item_off[z];
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t *meta = g.r.meta;
    unsigned long long acc_all = 0;
    auto flush = [&]() {   // every lane of the warp
        __syncwarp();
        unsigned long long p = 0;
        if (lane == 0) p = atomicAdd(n_rows, (unsigned long long)staged);
        p = __shfl_sync(0xffffffffu, p, 0);
        for (uint32_t i = lane; i < 3 * staged; i += 32)
            if (3 * p + i < 3 * capacity) rows[3 * p + i] = stage[i];
        __syncwarp();
        staged = 0;
    };
    for (;;) {
        if (threadIdx.x == 0) item_s = atomicAdd(counter, 1u);
        __syncthreads();
        const uint32_t item = item_s;
        if (item >= total_items) break;
        // bucket of this item: at the last position with item_off <= item
        uint32_t lo = 0, hi = z;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (item_off[mid] <= item) lo = mid; else hi = mid;
        }
        const uint32_t k = g.order[lo];
        // (T chunk, S chunk) of this item
        const uint32_t sch = cc_schunks(g.offS[k + 1] - g.offS[k], g.schunk);
        const uint32_t li = item - item_off[lo];
        const uint32_t tci = li / sch, sci = li - tci * sch;
        const uint32_t s0 = g.offS[k] + sci * g.schunk, s1 = min(g.offS[k + 1], s0 + g.schunk);
        const bool few = s1 - s0 <= QCAP;
        const uint32_t qmin = few ? kFewMin : kQueueMin, qstep = few ? kFewStep : CC_CH;
        // T_k's set: the item's chunk on chip, or for a big bucket its region
        // of the workspace, built before this kernel
        bool big = cc_big(g.offT[k + 1] - g.offT[k]);
        const uint32_t ta = g.offT[k] + tci * CC_TCAP;
        const uint32_t tz = big ? g.offT[k + 1] : min(g.offT[k + 1], ta + CC_TCAP);
        const unsigned long long gbase = g.big_off[k];
        uint32_t gmask = (uint32_t)(g.big_off[k + 1] - gbase) - 1u;
        const unsigned long long *gset = g.bigset + gbase;
        const uint32_t *gcnt = g.bigcnt + gbase;

        // ---- T_k as a (c, a) multiset: a slot per distinct pair ----
        if (!big)
            for (uint32_t q = threadIdx.x; q < CC_NB; q += CC_T)
                ((ulonglong2 *)tk)[q] = make_ulonglong2(kEmpty64, kEmpty64);
        // (a big bucket's filter passes everything)
        const uint32_t fw = big ? 0xffffffffu : 0u;
        for (uint32_t q = threadIdx.x; q < CC_FWORDS / 4; q += CC_T) ((uint4 *)filt)[q] = make_uint4(fw, fw, fw, fw);
        if (threadIdx.x == 0) {
            tdup = 0u;
            tneg = big ? g.big_neg[k] : 0u;
            batch_ctr = 0u;
            chunk_ctr = 0u;
            qn = 0u;
            carry = 0u;
        }
        __syncthreads();
        for (uint32_t q = ta + threadIdx.x; !big && q < tz; q += CC_T) {
            const uint2 tu = __ldg(g.Tp + q);   // (c, a)
            const unsigned long long key = cpack(tu.x, tu.y);
            const uint32_t h = chash_a(tu.y, chash(tu.x, g.seed));
            fset(filt, h);
            if (key == kEmpty64) {               // (-1, -1) is the empty marker: counted apart
                atomicAdd(&tneg, 1u);
                continue;
            }
            const int r = cset_insert(tk, key, cbucket(h));
            if (r == 2 && !tdup) tdup = 1u;
            if (r == 0) set_status(g.st, MWJ_ERR_CHECK, 24);
        }
        __syncthreads();
        if (tdup) {
            // the chunk repeats pairs: its set with multiplicities in this
            // CTA's region, looked up through the L2 like a big bucket's
            for (uint32_t q = threadIdx.x; q < CC_TSLOTS; q += CC_T) {
                my_set[q] = kEmpty64;
                my_cnt[q] = 0u;
            }
            __syncthreads();
            for (uint32_t q = ta + threadIdx.x; q < tz; q += CC_T) {
                const uint2 tu = __ldg(g.Tp + q);
                const unsigned long long key = cpack(tu.x, tu.y);
                if (key == kEmpty64) continue;   // counted in tneg already
                uint32_t s = gslot(tu.x, tu.y, g.seed) & (CC_TSLOTS - 1);
                for (uint32_t it = 0; it < CC_TSLOTS; ++it) {
                    const unsigned long long v = atomicCAS(my_set + s, kEmpty64, key);
                    if (v == kEmpty64 || v == key) {
                        atomicAdd(my_cnt + s, 1u);
                        break;
                    }
                    s = (s + 1) & (CC_TSLOTS - 1);
                }
            }
            __syncthreads();
            big = true;
            gset = my_set;
            gcnt = my_cnt;
            gmask = CC_TSLOTS - 1;
        }
        const uint32_t negs = tneg;

        // ---- stream S_k past the set ----
        // One closed or open wedge per lane and call: m copies of (c, a) in
        // T_k close wedge (a, b, c).  They are added up (and into cnt[a]), or
        // staged as rows.  Every lane of the warp calls this.
        unsigned long long acc = 0;
        auto emit = [&](uint32_t a, uint32_t b, uint32_t c, uint32_t m, bool turned) {
            if (!ROWS) {
                acc += m;
                if (g.cnt && m && a < (uint32_t)g.a_domain) atomicAdd(g.cnt + a, (unsigned long long)m);
                return;
            }
            const unsigned some = __ballot_sync(0xffffffffu, m != 0u);
            if (!some) return;
            const int32_t rb = (int32_t)(turned ? c : b), rc = (int32_t)(turned ? b : c);
            // not staged: this lane's m rows, after the `ex` of the lanes before it of `all`
            auto write = [&](unsigned long long ex, unsigned long long all) {
                unsigned long long p = 0;
                if (lane == 0) p = atomicAdd(n_rows, all);
                p = __shfl_sync(0xffffffffu, p, 0) + ex;
                for (uint32_t e = 0; e < m && p < capacity; ++e, ++p) {
                    rows[3 * p] = (int32_t)a;
                    rows[3 * p + 1] = rb;
                    rows[3 * p + 2] = rc;
                }
            };
            if (__any_sync(0xffffffffu, m > CC_STAGE)) {
                // a pair of T may occur |T| times: the step's rows are added in 64 bits
                unsigned long long incl = m;
#pragma unroll 1
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
                    if ((int)lane >= o) incl += y;
                }
                write(incl - m, __shfl_sync(0xffffffffu, incl, 31));
                return;
            }
            uint32_t ex = __popc(some & ((1u << lane) - 1u)), tot = __popc(some);
            if (__any_sync(0xffffffffu, m > 1u)) {   // (at most 32 x CC_STAGE rows from here on)
                uint32_t incl = m;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if ((int)lane >= o) incl += y;
                }
                tot = __shfl_sync(0xffffffffu, incl, 31);
                ex = incl - m;
            }
            if (tot > CC_STAGE) {
                write(ex, tot);
                return;
            }
            if (staged + tot > CC_STAGE) flush();
            for (uint32_t e = 0; e < m; ++e) {
                int32_t *const row = stage + 3 * (staged + ex + e);
                row[0] = (int32_t)a;
                row[1] = rb;
                row[2] = rc;
            }
            staged += tot;
        };
        auto count = [&](uint32_t c, uint32_t a, uint32_t ch) -> uint32_t {
            const unsigned long long key = cpack(c, a);
            if (key == kEmpty64) return negs;
            if (!big) return cset_count(tk, key, cbucket(chash_a(a, ch)));
            // a big bucket's set, or this CTA's for a chunk that repeats
            // pairs (written in this kernel: read through the L2)
            uint32_t s = gslot(c, a, g.seed) & gmask;
            for (uint32_t it = 0; it <= gmask; ++it) {
                const unsigned long long v = __ldcg(gset + s);
                if (v == key) return __ldcg(gcnt + s);
                if (v == kEmpty64) break;
                s = (s + 1) & gmask;
            }
            return 0u;
        };
        // walk one list of the warp's: entries [lo, hi) from alist[jst & ~3] on,
        // those before jst left out, lo a multiple of four.  In steps of CC_CH
        // entries: first the filter bits, 16 bytes of the list per lane and load
        // (a lane's 32 bits in the order of its entries, the first one on top),
        // then the set for those that passed, whose a is read again.  Every lane
        // of the warp calls this.  (4 bytes per lane and load: 24.4 ms for the
        // probe of the 2^22-vertex graph, 22.9 this way; reading four of the
        // passed a's at once instead: 31.5.)
        auto walk = [&](uint32_t jb, uint32_t jc, uint32_t jst, uint32_t lo, uint32_t hi) {
            const uint32_t ch = chash(jc, g.seed);
            const uint32_t start = ROWS ? jst & ~kTurned : jst;
            const int32_t *list = g.r.alist + (start & ~3u);
            const uint32_t skip = start & 3u;
            for (uint32_t base = lo; base < hi; base += CC_CH) {
                const int32_t *at = list + base + 4u * lane;
                const uint32_t n = min(hi - base, CC_CH);
                uint32_t hits = 0;
                auto four = [&](const int4 &v) {
                    hits = __funnelshift_l(ftop(filt, (uint32_t)v.x, ch), hits, 1);
                    hits = __funnelshift_l(ftop(filt, (uint32_t)v.y, ch), hits, 1);
                    hits = __funnelshift_l(ftop(filt, (uint32_t)v.z, ch), hits, 1);
                    hits = __funnelshift_l(ftop(filt, (uint32_t)v.w, ch), hits, 1);
                };
                uint32_t done = 0;
                for (; done + 256u <= n; done += 256u) {
                    const int4 v0 = __ldg((const int4 *)(at + done)), v1 = __ldg((const int4 *)(at + done + 128u));
                    four(v0);
                    four(v1);
                }
                for (; done < n; done += 128u) {   // (the list's room ends 4 entries after it)
                    const uint32_t e = done + 4u * lane;
                    four(e < n ? __ldg((const int4 *)(at + done)) : make_int4(0, 0, 0, 0));
                    if (e + 4u > n) hits &= e < n ? 0xffffffffu << (e + 4u - n) : ~15u;
                }
                hits <<= 32u - done / 32u;   // (done / 32 bits so far)
                if (base == 0u && lane == 0) hits &= 0xffffffffu >> skip;
                while (!ROWS ? hits != 0u : (bool)__any_sync(0xffffffffu, hits != 0u)) {
                    uint32_t a = 0, m = 0;
                    if (hits) {
                        const uint32_t e = (uint32_t)__clz((int)hits);
                        hits &= ~(0x80000000u >> e);
                        a = (uint32_t)__ldg(at + (e >> 2) * 128u + (e & 3u));
                        m = count(jc, a, ch);
                    }
                    emit(a, jb, jc, m, ROWS && (jst & kTurned));
                }
                __syncwarp();
            }
        };
        // phase 1: warps take batches of 32 S tuples as they come free;
        // lists of qmin or more entries go to the item's queue (walked at
        // once when it is full), lists of 32 or more are walked by the warp,
        // shorter ones are spread over the warp's lanes, wedge wi going to
        // the first lane whose inclusive count exceeds it
        for (;;) {
            uint32_t bi = 0;
            if (lane == 0) bi = atomicAdd(&batch_ctr, 1u);
            bi = __shfl_sync(0xffffffffu, bi, 0);
            const uint32_t w0 = s0 + bi * 32u;
            if (w0 >= s1) break;
            const uint32_t idx = w0 + lane;
            uint32_t b = 0, c = 0, n = 0, st = 0;
            if (idx < s1) {
                const uint2 tu = __ldg(g.Sp + idx);
                b = tu.x;
                c = tu.y;
                const int e = rg_find(g.r, meta, b);
                if (e >= 0) {
                    n = __ldg(g.r.deg + e);
                    st = __ldg(g.r.end + e) - n;
                    if (ROWS && g.turned && __ldg(g.turned + idx)) st |= kTurned;
                }
            }
            bool spill = false;
            if (n >= qmin) {
                const uint32_t qs = atomicAdd(&qn, 1u);
                if (qs < QCAP)
                    queue[qs] = make_uint4(b, c, st, n);
                else
                    spill = true;
            }
            unsigned sm_ = __ballot_sync(0xffffffffu, spill);
            while (sm_) {
                const int j = __ffs(sm_) - 1;
                sm_ &= sm_ - 1u;
                walk(__shfl_sync(0xffffffffu, b, j), __shfl_sync(0xffffffffu, c, j),
                     __shfl_sync(0xffffffffu, st, j), 0u,
                     __shfl_sync(0xffffffffu, n + (st & 3u), j));
            }
            // lists of 32 .. qmin - 1 entries: the warp walks each one
            unsigned mid_ = __ballot_sync(0xffffffffu, n >= 32u && n < qmin);
            while (mid_) {
                const int j = __ffs(mid_) - 1;
                mid_ &= mid_ - 1u;
                walk(__shfl_sync(0xffffffffu, b, j), __shfl_sync(0xffffffffu, c, j),
                     __shfl_sync(0xffffffffu, st, j), 0u,
                     __shfl_sync(0xffffffffu, n + (st & 3u), j));
            }
            const uint32_t ns = n < 32u ? n : 0u;
            uint32_t incl = ns;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if ((int)lane >= o) incl += y;
            }
            const uint32_t W = __shfl_sync(0xffffffffu, incl, 31);
            const uint32_t excl = incl - ns;
            for (uint32_t base = 0; base < W; base += 32) {
                const uint32_t wi = base + lane;
                int olo = 0, ohi = 31;
                const uint32_t qv = (wi < W) ? wi : 0u;
#pragma unroll
                for (int step = 0; step < 5; ++step) {
                    const int mid = (olo + ohi) >> 1;
                    const uint32_t v = __shfl_sync(0xffffffffu, incl, mid);
                    if (v > qv) ohi = mid; else olo = mid + 1;
                }
                const uint32_t ob = __shfl_sync(0xffffffffu, b, olo);
                const uint32_t oc = __shfl_sync(0xffffffffu, c, olo);
                const uint32_t ost = __shfl_sync(0xffffffffu, st, olo);
                const uint32_t oex = __shfl_sync(0xffffffffu, excl, olo);
                uint32_t a = 0, m = 0;
                if (wi < W) {
                    a = (uint32_t)__ldg(g.r.alist + (ROWS ? ost & ~kTurned : ost) + (wi - oex));
                    const uint32_t ch = chash(oc, g.seed);
                    if ((int32_t)ftop(filt, a, ch) < 0) m = count(oc, a, ch);
                }
                emit(a, ob, oc, m, ROWS && (ost & kTurned));
            }
        }
        __syncthreads();
        // phase 2: the queued lists in chunks of qstep entries, taken by the
        // warps as they come free (a hub's long list is shared by all of them)
        const uint32_t nq = min(qn, QCAP);
        for (uint32_t q0 = 0; q0 <= nq; q0 += CC_T) {
            const uint32_t q = q0 + threadIdx.x;
            const uint32_t d = q < nq ? ((queue[q].z & 3u) + queue[q].w + qstep - 1) / qstep : 0u;
            uint32_t tot;
            const uint32_t ex = block_excl_scan_u32(d, scan_scratch, &tot);
            if (q <= nq) cpre[q] = carry + ex;
            __syncthreads();
            if (threadIdx.x == 0) carry += tot;
            __syncthreads();
        }
        const uint32_t nchunks = cpre[nq];
        for (;;) {
            uint32_t ci = 0;
            if (lane == 0) ci = atomicAdd(&chunk_ctr, 1u);
            ci = __shfl_sync(0xffffffffu, ci, 0);
            if (ci >= nchunks) break;
            uint32_t lo = 0, hi = nq;   // last list with cpre <= ci
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (cpre[mid] <= ci) lo = mid; else hi = mid;
            }
            const uint4 L = queue[lo];
            const uint32_t first = (ci - cpre[lo]) * qstep;
            walk(L.x, L.y, L.z, first, min(first + qstep, (L.z & 3u) + L.w));
        }
        acc_all += acc;
        __syncthreads();
    }
    if (ROWS) {
        if (staged) flush();
        return;
    }
    const unsigned long long tot = block_sum_u64(acc_all, red);
    if (threadIdx.x == 0 && tot) atomicAdd(g.total, tot);
}

__global__ void k_cc_rows_check(const unsigned long long *n_rows, unsigned long long capacity, unsigned long long *total,
                                DevStatus *st) {
    after_previous();
    *total = *n_rows;
    if (*n_rows > capacity) set_status(st, MWJ_ERR_CAPACITY, (long long)*n_rows);
}

}  // namespace

uint32_t cyc_c_schunk(int64_t nS, int num_sms) {
    // about four items per probe CTA over the whole of S: a join with few
    // buckets (a small T, cheap to rebuild per item) is spread over the GPU,
    // one with many buckets (S_k below the piece) is not split at all
    const uint64_t want = ((uint64_t)(nS > 0 ? nS : 0) + 4ull * num_sms * CC_MAX_CTAS_PER_SM - 1) /
                          (4ull * num_sms * CC_MAX_CTAS_PER_SM);
    return (uint32_t)(want > CC_SCHUNK_MIN ? (want < 0x7FFFFFFFull ? want : 0x7FFFFFFFull) : CC_SCHUNK_MIN);
}

size_t cyc_c_rep_slots(int num_sms) { return (size_t)num_sms * CC_MAX_CTAS_PER_SM * CC_TSLOTS; }

uint32_t cyc_c_tavg() { return CC_TAVG; }

cudaError_t rgroup_build(const int32_t *Ra, const int32_t *Rb, int64_t nR, const RGroup &r, unsigned int *hll,
                         uint64_t reserve, unsigned int *bump, int32_t a_domain, DevStatus *status, int num_sms,
                         cudaStream_t st) {
    cudaError_t e = single_table_size(Rb, nR, r.seed, hll, (uint32_t *)r.meta, reserve, num_sms, st, "rg_hll",
                                      "rg_size", true);
    if (e != cudaSuccess) return e;
    const uint32_t n = (uint32_t)nR;
    const unsigned grid = (unsigned)num_sms * 4;
    {
        ProfScope ps_("rg_clear", st);
        if ((e = launch_after(k_rg_clear, grid, RG_T, st, r, bump)) != cudaSuccess) return e;
    }
    if (n == 0) return cudaSuccess;
    {
        ProfScope ps_("rg_count", st);
        if ((e = launch_after(k_rg_count, grid, RG_T, st, Ra, Rb, n, r, a_domain, status)) != cudaSuccess) return e;
    }
    {
        ProfScope ps_("rg_offsets", st);
        if ((e = launch_after(k_rg_offsets, grid, RG_T, st, r, bump)) != cudaSuccess) return e;
    }
    ProfScope ps_("rg_scatter", st);
    return launch_after(k_rg_scatter, grid, RG_T, st, Ra, Rb, n, r, n, status);
}

cudaError_t cyc_c_orient(const int32_t *Sb, const int32_t *Sc, int64_t nS, const RGroup &r, int32_t *u, int32_t *v,
                         int32_t *turned, int num_sms, cudaStream_t st) {
    if (nS <= 0) return cudaSuccess;
    ProfScope ps_("cyc_c_orient", st);
    return launch_after(k_cc_orient, num_sms * 4, RG_T, st, Sb, Sc, (uint32_t)nS, r, u, v, turned);
}

cudaError_t cyc_c_run(const CycCArgs &g, uint32_t *items, void *scan_tmp, unsigned int *counter,
                      unsigned long long *big_slots, void *scan_tmp64b, int32_t *rows, long long capacity,
                      long long *n_rows, unsigned long long *rep_set, uint32_t *rep_cnt, int num_sms,
                      cudaStream_t st) {
    const uint32_t z = g.z;
    const bool with_rows = (n_rows != nullptr);
    cudaError_t e;
    {
        ProfScope ps_("cyc_c_plan", st);
        e = launch_after(k_cc_plan, 1, CC_PLAN_T, st, g.offS, g.offT, z, g.schunk, items, (uint32_t *)g.order, big_slots);
        if (e != cudaSuccess) return e;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(items + z, 0, sizeof(uint32_t), st)) != cudaSuccess) return e;
    if ((e = scan_excl_u32(items, z + 1, scan_tmp, st)) != cudaSuccess) return e;
    // big buckets' sets in the workspace
    if ((e = scan_excl_u64((const uint64_t *)big_slots, (uint64_t *)g.big_off, z, true, scan_tmp64b, st)) !=
        cudaSuccess)
        return e;
    {
        ProfScope ps_("cyc_c_bigclear", st);
        e = launch_after(k_cc_bigclear, num_sms * 4, 512, st, (unsigned long long *)g.bigset, (uint32_t *)g.bigcnt,
                         g.big_off, z);
        if (e != cudaSuccess) return e;
    }
    {
        ProfScope ps_("cyc_c_bigbuild", st);
        e = launch_after(k_cc_bigbuild, num_sms * 2, 512, st, g.Tp, g.offT, z, g.big_off,
                         (unsigned long long *)g.bigset, (uint32_t *)g.bigcnt, (uint32_t *)g.big_neg, g.seed, g.st);
        if (e != cudaSuccess) return e;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const uint32_t qcap = with_rows ? CC_QCAP_ROWS : CC_QCAP;
    const size_t smem = CC_TSLOTS * sizeof(unsigned long long) + CC_FWORDS * sizeof(uint32_t) +
                        qcap * sizeof(uint4) + (qcap + 1) * sizeof(uint32_t) +
                        (with_rows ? CC_T / 32 * 3 * CC_STAGE * sizeof(int32_t) : 0);
    auto probe = with_rows ? k_cc_probe<true> : k_cc_probe<false>;
    if ((e = cudaFuncSetAttribute(probe, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return e;
    int occ = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, probe, CC_T, smem) != cudaSuccess || occ < 1) occ = 1;
    if (occ > CC_MAX_CTAS_PER_SM) occ = CC_MAX_CTAS_PER_SM;   // one region per CTA for repeated pairs
    const unsigned grid = (unsigned)(num_sms * occ);
    if ((e = cudaMemsetAsync(counter, 0, sizeof(unsigned int), st)) != cudaSuccess) return e;
    if (with_rows && (e = cudaMemsetAsync(n_rows, 0, sizeof(*n_rows), st)) != cudaSuccess) return e;
    {
        ProfScope ps_(with_rows ? "cyc_c_rows" : "cyc_c_probe", st);
        e = launch_after_smem(probe, grid, CC_T, smem, st, g, items, counter, (unsigned long long *)n_rows, rows,
                              (unsigned long long)capacity, rep_set, rep_cnt);
        if (e != cudaSuccess) return e;
    }
    if (!with_rows) return cudaSuccess;
    ProfScope ps_("rows_check", st);
    return launch_after(k_cc_rows_check, 1, 1, st, (unsigned long long *)n_rows, (unsigned long long)capacity, g.total,
                        g.st);
}

}  // namespace mwj
