// fm.cu -- Flajolet-Martin sketches of the distinct friends of friends of
// friends of every A (Section 4.1's footnote; the approximate variant of
// Example 1's query):
//
//     D(a) = { d : (a,b) in R, (b,c) in S, (c,d) in T }
//
// is summarised by a PCSA sketch (Flajolet and Martin, 1985): M = 16 bitmaps
// of 32 bits; a value d sets bit rho(h div M) of bitmap h mod M, with
// h = fmix32(d xor SEED) (MurmurHash3's 32-bit finaliser) and rho the index
// of the lowest 1 bit (27 when h div M is 0).  The sketch of a union is the
// OR of the sketches, so the linear join carries sketches along the chain the
// way it carries counts for COUNT(*) GROUP BY A, with OR in place of +:
//
//     skT(c) = OR of bit(d) over T's (c, d)                  (one pass over T)
//     w(b)   = OR of skT(c) over S_i's (b, c)                (on chip, per bucket)
//     sk(a) |= w(b) for every (a, b) of R_i                  (global, per bucket)
//
// By default nothing is partitioned (the one-bucket plan of linear_l2.cu with
// sketches for weights): T's and S's sketches are rows of 64 bytes (the "~100
// bytes per tuple" of the paper's footnote) in two arrays indexed by the key,
// and the S and the R pass each gather one row per tuple.  On this GPU a
// gathered 64-byte row costs little more than a gathered word (238 against
// 289 G/s, L2-resident: the L1's tag rate bounds both), so the passes run at
// the speed of the counting ones.  With explicit shares, and for relations
// whose rows would not be reserved (kFmOneMax), R and S are partitioned by
// H(B) as in Algorithm 1; bucket i's on-chip table holds S_i's B values with
// their sketches.  F of the 2^20-vertex graph: 3.8 ms partitioned, 1.0 ms in
// one bucket.  Four lanes handle one tuple, four bitmaps (16 bytes) per lane.  The estimate of |D(a)| is (M / PHI) * 2^(mean R_j),
// R_j the lowest 0 bit of bitmap j, PHI = 0.77351.
#include "api_internal.h"
#include "group_table.cuh"
#include "tables.h"

namespace mwj {
namespace {

constexpr uint32_t FM_M = 16;                 // bitmaps per sketch
constexpr uint32_t FM_SEED = 0x5BD1E995u;
constexpr double FM_PHI = 0.77351;
constexpr int FT = 512;                        // threads per CTA
constexpr uint32_t kFmCapLog2 = 10;            // on-chip table: 1024 slots of 68 bytes

// MurmurHash3's 32-bit finalisation mix (Appleby's published constants).
__device__ __forceinline__ uint32_t fmix32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x85EBCA6Bu;
    x ^= x >> 13;
    x *= 0xC2B2AE35u;
    x ^= x >> 16;
    return x;
}

// (bitmap, bit) that value d sets
__device__ __forceinline__ void fm_bit(int32_t d, uint32_t *j, uint32_t *r) {
    const uint32_t h = fmix32((uint32_t)d ^ FM_SEED);
    *j = h & (FM_M - 1);
    const uint32_t q = h >> 4;
    *r = q ? (uint32_t)(__ffs((int)q) - 1) : 27u;
}

constexpr uint32_t kNoIndex = 0xFFFFFFFFu;

// dense sketch index of c from T's key table, whose entries hold
// (index << 32 | c) once k_fm_index has run (kNoIndex if c is absent)
__device__ __forceinline__ uint32_t tkey_index(const unsigned long long *tbl, uint32_t mask, uint32_t seed,
                                               uint32_t c) {
    uint32_t s = slot_of(c, seed, mask);
    for (uint32_t it = 0; it <= mask; ++it) {
        const unsigned long long x = __ldg(tbl + s);
        if (x == kEmpty64) return kNoIndex;
        if ((uint32_t)x == c) return (uint32_t)(x >> 32);
        s = (s + 1) & mask;
    }
    return kNoIndex;
}

// dense index of every occupied slot of T's key table (warp-aggregated
// counter; the order of the indices is immaterial), stored in the entry's
// upper half in place of the degree; count = their number.  An index is
// below 2^31, so an entry never becomes kEmpty64.
__global__ void k_fm_index(unsigned long long *__restrict__ tbl, const uint32_t *__restrict__ meta,
                           unsigned int *__restrict__ count) {
    const uint64_t slots = (uint64_t)meta[0] + 1;
    for (uint64_t s0 = (uint64_t)blockIdx.x * blockDim.x; s0 < slots; s0 += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t s = s0 + threadIdx.x;
        const unsigned long long x = s < slots ? tbl[s] : kEmpty64;
        const bool occ = x != kEmpty64;
        const unsigned m = __ballot_sync(0xffffffffu, occ);
        unsigned base = 0;
        if ((threadIdx.x & 31) == 0 && m) base = atomicAdd(count, (unsigned)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        const unsigned idx = base + __popc(m & ((1u << (threadIdx.x & 31)) - 1u));
        if (occ) tbl[s] = ((unsigned long long)idx << 32) | (uint32_t)x;
    }
}

__global__ void k_fm_zero(uint32_t *__restrict__ sk, const unsigned int *__restrict__ count) {
    const uint64_t words = (uint64_t)(*count) * FM_M;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words;
         i += (uint64_t)gridDim.x * blockDim.x)
        sk[i] = 0u;
}

// skT(c) |= bit(d) for every (c, d) of T; each thread takes 8 consecutive
// tuples and ORs a run of equal c into a local sketch first
__global__ void __launch_bounds__(256) k_fm_tsketch(const int32_t *__restrict__ tc, const int32_t *__restrict__ td,
                                                    uint32_t n, const unsigned long long *__restrict__ tbl,
                                                    const uint32_t *__restrict__ meta, uint32_t seed,
                                                    uint32_t *__restrict__ skT) {
    const uint32_t mask = __ldg(meta);
    constexpr uint32_t K = 8;
    for (uint32_t i = (blockIdx.x * 256 + threadIdx.x) * K; i < n; i += gridDim.x * 256 * K) {
        const uint32_t m = min(K, n - i);
        uint32_t loc[FM_M];
#pragma unroll
        for (uint32_t j = 0; j < FM_M; ++j) loc[j] = 0;
        int32_t cur = __ldg(tc + i);
        auto flush = [&](int32_t c) {
            const uint32_t ix = tkey_index(tbl, mask, seed, (uint32_t)c);
            if (ix == kNoIndex) return;   // cannot happen: every c of T is in the table
            uint32_t *dst = skT + (size_t)ix * FM_M;
#pragma unroll
            for (uint32_t j = 0; j < FM_M; ++j)
                if (loc[j]) atomicOr(dst + j, loc[j]);
        };
        for (uint32_t k = 0; k < m; ++k) {
            const int32_t c = __ldg(tc + i + k);
            if (c != cur) {
                flush(cur);
#pragma unroll
                for (uint32_t j = 0; j < FM_M; ++j) loc[j] = 0;
                cur = c;
            }
            uint32_t j, r;
            fm_bit(__ldg(td + i + k), &j, &r);
#pragma unroll
            for (uint32_t q = 0; q < FM_M; ++q)
                if (q == j) loc[q] |= 1u << r;
        }
        flush(cur);
    }
}

struct FmArgs {
    const uint2 *Rp, *Sp;
    const uint32_t *offR, *offS;
    const unsigned long long *ttbl;   // T's key table, entries (dense index << 32 | c)
    const uint32_t *tmeta;
    uint32_t tseed;
    const uint32_t *skT;              // dense sketches of T's keys
    uint32_t seed_slot;
    int32_t a_domain;
    uint32_t *out;                    // a_domain x FM_M
    DevStatus *st;
};

// One CTA per H(B) bucket.  S_i's B values with their sketches on chip
// (optimistic pass with inserts of at most 32 probes; bounded rounds if that
// fails), then R_i streams past: sk(a) |= w(b).
__global__ void __launch_bounds__(FT) k_fm_probe(FmArgs g) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr uint32_t cap = 1u << kFmCapLog2, mask = cap - 1;
    uint32_t *keys = (uint32_t *)smem;                                    // cap + 1
    uint32_t *w = (uint32_t *)(smem + align256((cap + 1) * 4));          // (cap + 1) x FM_M
    __shared__ uint32_t nd, bad;
    const uint32_t i = blockIdx.x;
    const uint32_t r0 = g.offR[i], r1 = g.offR[i + 1], s0 = g.offS[i], s1 = g.offS[i + 1];
    if (r0 >= r1 || s0 >= s1) return;
    const uint32_t tmask = __ldg(g.tmeta);
    // four lanes per tuple, bitmaps 4 l4 .. 4 l4 + 3 on lane l4
    const uint32_t l4 = threadIdx.x & 3, grp = threadIdx.x >> 2, groups = FT / 4;

    auto tsk = [&](int32_t c) -> uint4 {   // this lane's bitmaps of skT(c) (0 if c not in T)
        const uint32_t ix = tkey_index(g.ttbl, tmask, g.tseed, (uint32_t)c);
        return ix == kNoIndex ? make_uint4(0u, 0u, 0u, 0u)
                              : __ldg((const uint4 *)(g.skT + (size_t)ix * FM_M) + l4);
    };
    auto or_in = [&](int slot, const uint4 &v) {   // w(b) |= skT(c), this lane's 4 bitmaps
        uint32_t *dst = w + (uint32_t)slot * FM_M + 4 * l4;
        if (v.x) atomicOr(dst, v.x);
        if (v.y) atomicOr(dst + 1, v.y);
        if (v.z) atomicOr(dst + 2, v.z);
        if (v.w) atomicOr(dst + 3, v.w);
    };
    auto clear = [&]() {   // ends with a barrier
        for (uint32_t s = threadIdx.x; s <= cap; s += FT) keys[s] = kEmptyKey;
        if (threadIdx.x == 0) keys[cap] = 0u;
        for (uint32_t s = threadIdx.x; s < (cap + 1) * FM_M; s += FT) w[s] = 0u;
        if (threadIdx.x == 0) {
            nd = 0;
            bad = 0;
        }
        __syncthreads();
    };

    for (uint32_t pos = s0; pos < s1;) {
        clear();
        uint32_t cend = s1;
        bool ok = false;
        if (pos == s0) {
            // optimistic pass: one tuple per four lanes; they insert the same
            // key (idempotent: the first CAS wins) and OR four bitmaps each
            uint32_t fresh_n = 0;
            for (uint32_t t = s0 + grp; t < s1; t += groups) {
                if (*(volatile uint32_t *)&bad) break;
                const uint2 st = __ldg(g.Sp + t);
                bool fresh;
                const int slot = tbl_insert(keys, mask, st.x, g.seed_slot, &fresh);
                fresh_n += fresh;
                if (slot < 0) {
                    atomicOr(&bad, 1u);
                    break;
                }
                or_in(slot, tsk((int32_t)st.y));
            }
            fresh_n = warp_sum(fresh_n);
            if ((threadIdx.x & 31) == 0 && fresh_n) atomicAdd(&nd, fresh_n);
            __syncthreads();
            ok = !bad && nd <= cap - cap / 4;
            __syncthreads();   // every thread has read nd and bad
            if (!ok) clear();
        }
        if (!ok) {
            // bounded rounds of at most cap / 4 tuples while the table stays at
            // most 3/4 full; one tuple per four lanes again
            const uint32_t rt = cap / 4;
            cend = pos;
            for (;;) {
                __syncthreads();
                const uint32_t filled = nd;
                __syncthreads();
                if (cend >= s1 || filled + rt > cap - cap / 4) break;
                const uint32_t e = min(s1, cend + rt);
                uint32_t fresh_n = 0;
                for (uint32_t t = cend + grp; t < e; t += groups) {
                    const uint2 st = __ldg(g.Sp + t);
                    bool fresh;
                    const int slot = tbl_insert(keys, mask, st.x, g.seed_slot, &fresh);
                    fresh_n += fresh;
                    if (slot < 0) {   // cannot happen: the table is never full
                        if (l4 == 0) set_status(g.st, MWJ_ERR_CHECK, 9);
                        continue;
                    }
                    or_in(slot, tsk((int32_t)st.y));
                }
                fresh_n = warp_sum(fresh_n);
                if ((threadIdx.x & 31) == 0 && fresh_n) atomicAdd(&nd, fresh_n);
                cend = e;
            }
        }
        // R_i streams past: sk(a) |= w(b), only bits that are new cost an atomic
        for (uint32_t t = r0 + grp; t < r1; t += groups) {
            const uint2 tr = __ldg(g.Rp + t);
            if ((uint32_t)tr.x >= (uint32_t)g.a_domain) continue;   // reported by the partitioner
            const int slot = tbl_find(keys, mask, tr.y, g.seed_slot);
            if (slot < 0) continue;
            const uint4 v = *(const uint4 *)(w + (uint32_t)slot * FM_M + 4 * l4);
            if (!(v.x | v.y | v.z | v.w)) continue;
            uint32_t *dst = g.out + (size_t)tr.x * FM_M + 4 * l4;
            const uint4 cur = __ldcg((const uint4 *)dst);
            if (v.x & ~cur.x) atomicOr(dst, v.x);
            if (v.y & ~cur.y) atomicOr(dst + 1, v.y);
            if (v.z & ~cur.z) atomicOr(dst + 2, v.z);
            if (v.w & ~cur.w) atomicOr(dst + 3, v.w);
        }
        __syncthreads();   // the table is rebuilt for the next chunk
        pos = cend;
    }
}

// The estimates.  A sketch's sum of lowest zeros is at most 16 x 32, and a
// double exp2 costs more than reading the sketch (0.051 ms for 2^20 of them,
// 0.033 ms this way): every CTA tabulates the estimate of each sum first.  Four
// lanes per sketch, 16 bytes each.
constexpr uint32_t kFmSums = 32 * FM_M + 1;
__global__ void __launch_bounds__(FT) k_fm_estimate(const uint32_t *__restrict__ sk, int32_t a_domain,
                                                    float *__restrict__ est) {
    after_previous();
    __shared__ float of_sum[kFmSums];
    for (uint32_t t = threadIdx.x; t < kFmSums; t += FT) of_sum[t] = (float)((FM_M / FM_PHI) * exp2((double)t / FM_M));
    __syncthreads();
    const uint64_t words = (uint64_t)a_domain * 4;   // 16-byte quarters
    const uint64_t stride = (uint64_t)gridDim.x * FT;
    for (uint64_t i = (uint64_t)blockIdx.x * FT + threadIdx.x; i - (threadIdx.x & 31) < words; i += stride) {
        const uint4 v = i < words ? __ldg((const uint4 *)sk + i) : make_uint4(0u, 0u, 0u, 0u);
        auto low = [](uint32_t w) {   // index of the lowest 0 bit (32 when none)
            return w == 0xFFFFFFFFu ? 32u : (uint32_t)__ffs((int)~w) - 1u;
        };
        uint32_t tot = low(v.x) + low(v.y) + low(v.z) + low(v.w);
        tot += __shfl_xor_sync(0xffffffffu, tot, 1);
        tot += __shfl_xor_sync(0xffffffffu, tot, 2);
        if (i < words && (i & 3) == 0) est[i >> 2] = of_sum[tot];
    }
}

// ---------------------------------------------------------------------------
// one bucket: rows of sketches indexed by key
// ---------------------------------------------------------------------------

// A relation's rows: direct-address (row k - min), or the index that a table of
// its distinct keys gives (group_table.cuh; key -1, which marks free slots, has
// the last row).  Direct-address when the key range is at most the number of
// tuples, so that either way n + 1 rows are enough.
struct FmRows {
    uint32_t *keys, *idx;   // hashed: slots and their row indices
    uint32_t *meta;
    uint32_t *rows;         // (n + 1) x FM_M
    unsigned int *count;    // rows given out
    uint32_t seed, n;
};

struct FmOne {
    FmRows t, s;
};

// the row of a key; the layout's words are read once per thread.  DENSE: known
// to be direct-address.
template <bool DENSE>
struct FmIndex {
    const FmRows &r;
    bool dense;
    uint32_t min, span, mask;
    __device__ explicit FmIndex(const FmRows &r_) : r(r_) {
        dense = DENSE || __ldg(r.meta + kMetaDense) != 0u;
        min = dense ? __ldg(r.meta + kMetaMin) : 0u;
        span = dense ? __ldg(r.meta + kMetaSpan) : 0u;
        mask = DENSE ? 0u : __ldg(r.meta + kMetaMask);
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t k) const {
        if (DENSE || dense) return k - min < span ? k - min : kNoIndex;
        if (k == kEmptyKey) return r.n;
        const uint32_t s = w_home(k, r.seed, mask);
        const uint32_t at = w_find(r.keys, mask, k, s, __ldg((const uint4 *)(r.keys + s)));
        return at == kEmptyKey ? kNoIndex : __ldg(r.idx + at);
    }
};

// y 0 / 1: T's / S's rows (direct-address) or free keys and key -1's row
// (hashed); y 2: the output sketches.
__global__ void __launch_bounds__(FT) k_fm_clear(FmOne g, uint32_t *__restrict__ out, uint64_t out_rows) {
    after_previous();
    const uint64_t i0 = (uint64_t)blockIdx.x * FT + threadIdx.x, stride = (uint64_t)gridDim.x * FT;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    if (blockIdx.y == 2) {
        for (uint64_t i = i0; i < 4 * out_rows; i += stride) ((uint4 *)out)[i] = zero;
        return;
    }
    const FmRows &r = blockIdx.y ? g.s : g.t;
    if (i0 == 0) *r.count = 0u;
    if (__ldg(r.meta + kMetaDense)) {
        const uint64_t rows = __ldg(r.meta + kMetaSpan);
        for (uint64_t i = i0; i < 4 * rows; i += stride) ((uint4 *)r.rows)[i] = zero;
        return;
    }
    const uint4 free4 = make_uint4(kEmptyKey, kEmptyKey, kEmptyKey, kEmptyKey);
    for (uint64_t i = i0; i < ((uint64_t)__ldg(r.meta + kMetaMask) + 1) / 4; i += stride) ((uint4 *)r.keys)[i] = free4;
    if (i0 < 4) ((uint4 *)(r.rows + (size_t)r.n * FM_M))[i0] = zero;
}

// Hashed: the distinct keys of a column (y 0: T's C, y 1: S's B).
__global__ void __launch_bounds__(256) k_fm_keys(FmOne g, const int32_t *__restrict__ tc,
                                                 const int32_t *__restrict__ sb, DevStatus *st) {
    after_previous();
    const FmRows &r = blockIdx.y ? g.s : g.t;
    if (__ldg(r.meta + kMetaDense)) return;
    const int32_t *col = blockIdx.y ? sb : tc;
    const uint32_t mask = __ldg(r.meta + kMetaMask), lane = threadIdx.x & 31;
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i - lane < r.n; i += (uint64_t)gridDim.x * 256) {
        const uint32_t k = i < r.n ? (uint32_t)__ldg(col + i) : kEmptyKey;
        const uint32_t prev = __shfl_up_sync(0xffffffffu, k, 1);
        if (k == kEmptyKey || (lane > 0 && prev == k)) continue;   // (a run needs its key once)
        const uint32_t s = w_home(k, r.seed, mask);
        if (w_claim(r.keys, mask, k, s, __ldcg((const uint4 *)(r.keys + s))) == kEmptyKey)
            set_status(st, MWJ_ERR_CHECK, 10);   // table full: the sizing step under-estimated
    }
}

// Hashed: a row for every key, zeroed by the thread that gives it out.
__global__ void __launch_bounds__(256) k_fm_rows(FmOne g) {
    after_previous();
    const FmRows &r = blockIdx.y ? g.s : g.t;
    if (__ldg(r.meta + kMetaDense)) return;
    const uint64_t slots = (uint64_t)__ldg(r.meta + kMetaMask) + 1;
    const uint32_t lane = threadIdx.x & 31;
    for (uint64_t s = (uint64_t)blockIdx.x * 256 + threadIdx.x; s - lane < slots; s += (uint64_t)gridDim.x * 256) {
        const bool occ = s < slots && r.keys[s] != kEmptyKey;
        const unsigned m = __ballot_sync(0xffffffffu, occ);
        unsigned base = 0;
        if (lane == 0 && m) base = atomicAdd(r.count, (unsigned)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        const uint32_t row = base + __popc(m & ((1u << lane) - 1u));
        if (!occ || row >= r.n) continue;   // (distinct keys: at most n)
        r.idx[s] = row;
        uint4 *dst = (uint4 *)(r.rows + (size_t)row * FM_M);
        for (int q = 0; q < 4; ++q) dst[q] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// T pass: the bit of d in c's row, a tuple per lane, one 32-bit OR each (their
// results are not needed; the tuples of one c share two sectors).
__global__ void __launch_bounds__(256) k_fm_tbits(const int32_t *__restrict__ tc, const int32_t *__restrict__ td,
                                                  uint32_t n, FmRows r) {
    after_previous();
    const uint32_t T = gridDim.x * 256;
    const FmIndex<false> index(r);
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += T) {
        const uint32_t row = index((uint32_t)__ldg(tc + i));
        uint32_t j, bit;
        fm_bit(__ldg(td + i), &j, &bit);
        if (row != kNoIndex) atomicOr(r.rows + (size_t)row * FM_M + j, 1u << bit);   // (every c of T has a row)
    }
}

// S and R pass: row(x) |= row(y) over the relation's tuples (x, y).  A group of
// four lanes takes FM_K consecutive tuples, gathers their rows four at a time
// (16 bytes per lane) and ORs a run of equal x in registers; at the run's end
// only the bits that the target row lacks cost an atomic.  OUT: the target is
// the output, indexed by a in [0, a_domain).
// The next four tuples are loaded while the rows of these are on their way,
// and a run's target row is read when the run ends and compared when the next
// one does (or the group's tuples end): without the two the group waited out
// three memory latencies per four tuples (0.53 ms a pass on F, 0.37 ms with
// them and the layout's words in registers).
// DENSE: all rows of the pass direct-address; the call launches both kernels
// and the one whose layout the sizing pass did not choose returns at once.
// What bounds it now: 64 bytes per tuple from a 64 MB array that the L2 keeps
// only in part (59 % hits: 0.8 GB of row sectors come from DRAM in a pass).
constexpr uint32_t FM_K = 32;
template <bool OUT, bool DENSE>
__global__ void __launch_bounds__(256, 4) k_fm_pass(const int32_t *__restrict__ X, const int32_t *__restrict__ Y,
                                                    uint32_t n, FmRows src, FmRows dst,
                                                                uint32_t *__restrict__ out, int32_t a_domain,
                                                                DevStatus *st) {
    after_previous();
    if ((__ldg(src.meta + kMetaDense) && (OUT || __ldg(dst.meta + kMetaDense))) != DENSE) return;
    const uint32_t l4 = threadIdx.x & 3;
    const uint64_t groups = (uint64_t)gridDim.x * 64;
    const FmIndex<DENSE> from(src), to(dst);
    // lane l4 of a group holds tuple i + l4; the others read it by shuffle
    const unsigned group = 0xFu << (threadIdx.x & 28);
    auto load = [&](uint32_t i, uint32_t e, int32_t &x, int32_t &y) {
        x = i + l4 < e ? __ldg(X + i + l4) : 0;
        y = i + l4 < e ? __ldg(Y + i + l4) : 0;
    };
    // the run that ended last: its target (null: none), its OR, the target's
    // bits as read then
    uint32_t *pend = nullptr;
    uint4 pv = make_uint4(0u, 0u, 0u, 0u), pc = pv;
    auto settle = [&]() {
        if (!pend) return;
        if (pv.x & ~pc.x) atomicOr(pend, pv.x);
        if (pv.y & ~pc.y) atomicOr(pend + 1, pv.y);
        if (pv.z & ~pc.z) atomicOr(pend + 2, pv.z);
        if (pv.w & ~pc.w) atomicOr(pend + 3, pv.w);
        pend = nullptr;
    };
    auto flush = [&](int32_t x, const uint4 &v) {
        settle();
        if (!(v.x | v.y | v.z | v.w)) return;
        if (OUT) {
            if ((uint32_t)x >= (uint32_t)a_domain) return;   // reported below
            pend = out + (size_t)(uint32_t)x * FM_M + 4 * l4;
        } else {
            const uint32_t row = to((uint32_t)x);
            if (row == kNoIndex) return;   // (every b of S has a row)
            pend = dst.rows + (size_t)row * FM_M + 4 * l4;
        }
        pv = v;
        pc = __ldcg((const uint4 *)pend);
    };
    for (uint64_t i0 = ((uint64_t)blockIdx.x * 64 + (threadIdx.x >> 2)) * FM_K; i0 < n; i0 += groups * FM_K) {
        const uint32_t e = (uint32_t)(i0 + FM_K < n ? i0 + FM_K : n);
        uint4 acc = make_uint4(0u, 0u, 0u, 0u);
        int32_t x, y;
        load((uint32_t)i0, e, x, y);
        int32_t cur = __shfl_sync(group, x, 0, 4);
        for (uint32_t i = (uint32_t)i0; i < e; i += 4) {
            const uint32_t m = min(4u, e - i);
            if (OUT && l4 < m && (uint32_t)x >= (uint32_t)a_domain) set_status(st, MWJ_ERR_DOMAIN, x);
            uint4 v[4];
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) {
                const uint32_t row = from((uint32_t)__shfl_sync(group, y, q, 4));
                v[q] = make_uint4(0u, 0u, 0u, 0u);
                if (q < m && row != kNoIndex) v[q] = __ldg((const uint4 *)(src.rows + (size_t)row * FM_M) + l4);
            }
            int32_t nx, ny;
            load(i + 4, e, nx, ny);
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) {
                const int32_t xq = __shfl_sync(group, x, q, 4);
                if (q >= m) break;
                if (xq != cur) {
                    flush(cur, acc);
                    acc = make_uint4(0u, 0u, 0u, 0u);
                    cur = xq;
                }
                acc.x |= v[q].x;
                acc.y |= v[q].y;
                acc.z |= v[q].z;
                acc.w |= v[q].w;
            }
            x = nx;
            y = ny;
        }
        flush(cur, acc);
    }
    settle();
}

// Tuples of S and T up to which their rows are reserved: 64 bytes each, so at
// most 17 GB a relation; larger relations are partitioned.
constexpr int64_t kFmOneMax = 1ll << 28;
bool fm_one(const mwj_rel &S, const mwj_rel &T, const mwj_shares *sh) {
    return !sh && S.n <= kFmOneMax && T.n <= kFmOneMax;
}

struct FmOneLayout {
    FmOne one;
    unsigned int *hll[2];
};

size_t fm_one_layout(Arena &A, const mwj_rel &S, const mwj_rel &T, int num_sms, const Seeds &sd, FmOneLayout &L) {
    auto take = [&](const mwj_rel &r, uint32_t seed) {
        FmRows f{};
        f.keys = A.take<uint32_t>(single_table_slots(r.n));
        f.idx = A.take<uint32_t>(single_table_slots(r.n));
        f.meta = A.take<uint32_t>(kMetaWords);
        f.rows = A.take<uint32_t>((size_t)(r.n + 1) * FM_M);
        f.count = A.take<unsigned int>(4);
        f.seed = seed;
        f.n = (uint32_t)r.n;
        return f;
    };
    L.one.t = take(T, sd.slot2);
    L.one.s = take(S, sd.slot);
    for (int k = 0; k < 2; ++k) L.hll[k] = A.take<unsigned int>(hll_scratch_registers(num_sms));
    return A.used;
}

unsigned fm_grid(uint64_t n, uint64_t per_cta, int num_sms, int ctas_per_sm) {
    const uint64_t want = (n + per_cta - 1) / per_cta, full = (uint64_t)num_sms * ctas_per_sm;
    return (unsigned)(want < full ? (want ? want : 1) : full);
}

cudaError_t fm_one_run(const FmOneLayout &L, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, int32_t a_domain,
                       uint32_t *sketches, DevStatus *status, int sms, cudaStream_t st) {
    const FmOne &g = L.one;
    SizeCol cols[kSizeCols];
    uint32_t ncols = 1;
    cols[0] = SizeCol{T.x, (uint32_t)T.n, g.t.seed, L.hll[0], {g.t.meta}, {single_table_slots(T.n)}, {(uint64_t)T.n}, 1u};
    if (S.x == T.x && S.n == T.n) {   // a self-join: one pass sizes both
        cols[0].meta[1] = g.s.meta;
        cols[0].reserve[1] = cols[0].reserve[0];
        cols[0].range[1] = cols[0].range[0];
        cols[0].ntargets = 2;
    } else {
        cols[1] = SizeCol{S.x, (uint32_t)S.n, g.s.seed, L.hll[1], {g.s.meta}, {single_table_slots(S.n)}, {(uint64_t)S.n}, 1u};
        ncols = 2;
    }
    // entries of 64 bytes, half an L2 line (2^24 tuples, 2^20 keys over 2^24 places 2.60
    // ms direct-address and 2.87 hashed, 2^16 keys 1.96 and 1.58; 2^23 tuples, 2^16 keys
    // over 2^22 places 0.65 and 1.01)
    for (uint32_t k = 0; k < ncols; ++k) {
        cols[k].sure = 1ull << 22;
        cols[k].near = 0;
        cols[k].per_key = 40.0;
    }
    cudaError_t e;
    if ((e = size_columns(cols, ncols, nullptr, 0, true, sms, st)) != cudaSuccess) return e;
    const uint64_t most = (uint64_t)(T.n > S.n ? T.n : S.n);
    // many sketches are zeroed by a memset of their own, at memory speed (2^16 tuples,
    // 2^26 sketches: 0.82 ms with the clear kernel, 0.63 with the memset)
    const bool own = a_domain > 1 << 22;
    if (own && (e = cudaMemsetAsync(sketches, 0, sizeof(uint32_t) * FM_M * (size_t)a_domain, st)) != cudaSuccess) return e;
    {
        ProfScope ps_("fm_clear", st);
        e = launch_after(k_fm_clear, dim3(sms * 2, own ? 2 : 3), FT, st, g, sketches, (uint64_t)a_domain);
        if (e != cudaSuccess) return e;
    }
    {
        ProfScope ps_("fm_keys", st);
        e = launch_after(k_fm_keys, dim3(fm_grid(most, 256, sms, 8), 2), 256, st, g, T.x, S.x, status);
        if (e != cudaSuccess) return e;
    }
    {
        ProfScope ps_("fm_rows", st);
        if ((e = launch_after(k_fm_rows, dim3(fm_grid(4 * most, 256, sms, 8), 2), 256, st, g)) != cudaSuccess) return e;
    }
    if (T.n > 0) {
        ProfScope ps_("fm_tbits", st);
        e = launch_after(k_fm_tbits, fm_grid(T.n, 256, sms, 8), 256, st, T.x, T.y, (uint32_t)T.n, g.t);
        if (e != cudaSuccess) return e;
    }
    if (S.n > 0) {
        const unsigned grid = fm_grid(S.n, 64 * FM_K, sms, 8);
        {
            ProfScope ps_("fm_spass", st);
            e = launch_after(k_fm_pass<false, true>, grid, 256, st, S.x, S.y, (uint32_t)S.n, g.t, g.s,
                             (uint32_t *)nullptr, 0, status);
            if (e != cudaSuccess) return e;
        }
        ProfScope ps_("fm_spass_hashed", st);
        e = launch_after(k_fm_pass<false, false>, grid, 256, st, S.x, S.y, (uint32_t)S.n, g.t, g.s,
                         (uint32_t *)nullptr, 0, status);
        if (e != cudaSuccess) return e;
    }
    if (R.n > 0) {
        const unsigned grid = fm_grid(R.n, 64 * FM_K, sms, 8);
        {
            ProfScope ps_("fm_rpass", st);
            e = launch_after(k_fm_pass<true, true>, grid, 256, st, R.x, R.y, (uint32_t)R.n, g.s, g.s,
                             sketches, a_domain, status);
            if (e != cudaSuccess) return e;
        }
        ProfScope ps_("fm_rpass_hashed", st);
        e = launch_after(k_fm_pass<true, false>, grid, 256, st, R.x, R.y, (uint32_t)R.n, g.s, g.s,
                         sketches, a_domain, status);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

struct FmLayout {
    uint2 *Rp, *Sp;
    uint32_t *offR, *offS;
    uint64_t *ttbl;
    uint32_t *tmeta;
    unsigned int *hll;
    unsigned int *tcount;
    uint32_t *skT;
    void *pscratch;
    size_t pscratch_bytes;
};

size_t fm_layout(Arena &A, uint32_t I, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, int num_sms,
                 FmLayout &L) {
    L.Rp = A.take<uint2>(R.n + 2);
    L.offR = A.take<uint32_t>(I + 1);
    L.Sp = A.take<uint2>(S.n + 2);
    L.offS = A.take<uint32_t>(I + 1);
    L.ttbl = A.take<uint64_t>(single_table_slots(T.n));
    L.tmeta = A.take<uint32_t>(4);
    L.hll = A.take<unsigned int>(hll_scratch_registers(num_sms));
    L.tcount = A.take<unsigned int>(4);
    L.skT = A.take<uint32_t>((size_t)(T.n + 1) * FM_M);
    size_t ps = part_scratch_bytes(R.n, I, num_sms);
    const size_t ps2 = part_scratch_bytes(S.n, I, num_sms);
    if (ps2 > ps) ps = ps2;
    L.pscratch = A.take<char>(ps);
    L.pscratch_bytes = ps;
    return A.used;
}

// H(B) buckets: ~16K S tuples each (about 500 distinct B values of a
// friends relation fit the 1024-slot table), at least four per SM
mwj_status fm_buckets(mwj_ctx *ctx, const mwj_rel &S, const mwj_shares *sh, uint32_t *I) {
    if (sh) {
        if (sh->s[0] < 1 || (uint32_t)sh->s[0] > kMaxBuckets)
            return fail(ctx, MWJ_ERR_INVALID_ARG, "FM sketches: s[0] must be in [1, %u]", kMaxBuckets);
        *I = (uint32_t)sh->s[0];
        return MWJ_OK;
    }
    uint64_t want = (uint64_t)(S.n + 16383) / 16384;
    const uint64_t minb = (uint64_t)ctx->dev.num_sms * 4;
    if (want < minb) want = minb;
    uint32_t p = pow2_at_least(want);
    *I = p > 16384 ? 16384u : p;
    return MWJ_OK;
}

}  // namespace
}  // namespace mwj

using namespace mwj;

extern "C" mwj_status mwj_fm_workspace_size(mwj_ctx *ctx, mwj_rel R, mwj_rel S, mwj_rel T,
                                            const mwj_shares *shares, size_t *bytes) {
    if (!ctx || !bytes) return MWJ_ERR_INVALID_ARG;
    if (!rel_ok(R) || !rel_ok(S) || !rel_ok(T)) return fail(ctx, MWJ_ERR_INVALID_ARG, "bad relation");
    Arena A(nullptr, 0);
    if (fm_one(S, T, shares)) {
        FmOneLayout L;
        *bytes = fm_one_layout(A, S, T, ctx->dev.num_sms, ctx->seeds, L);
        return MWJ_OK;
    }
    uint32_t I;
    mwj_status s = fm_buckets(ctx, S, shares, &I);
    if (s != MWJ_OK) return s;
    FmLayout L;
    *bytes = fm_layout(A, I, R, S, T, ctx->dev.num_sms, L);
    return MWJ_OK;
}

extern "C" mwj_status mwj_fm_linear(mwj_ctx *ctx, mwj_rel R, mwj_rel S, mwj_rel T, const mwj_shares *shares,
                                    int32_t a_domain, uint32_t *sketches, float *estimates, void *workspace,
                                    size_t ws_bytes, void *stream) {
    if (!ctx || !sketches || a_domain <= 0 || ((uintptr_t)sketches & 15)) return MWJ_ERR_INVALID_ARG;
    ApiScope api_scope(&ctx->prof);
    if (!rel_ok(R) || !rel_ok(S) || !rel_ok(T)) return fail(ctx, MWJ_ERR_INVALID_ARG, "bad relation");
    cudaStream_t st = (cudaStream_t)stream;
    const Seeds &sd = ctx->seeds;
    const int sms = ctx->dev.num_sms;
    cudaError_t e;
    Arena A(workspace, ws_bytes);
    auto estimate = [&]() -> mwj_status {
        if (!estimates) return MWJ_OK;
        ProfScope ps_("fm_estimate", st);
        const cudaError_t ee =
            launch_after(k_fm_estimate, fm_grid((uint64_t)a_domain * 4, FT, sms, 2), FT, st, sketches, a_domain, estimates);
        return ee == cudaSuccess ? MWJ_OK : cuda_fail(ctx, ee, "fm estimate");
    };
    if (fm_one(S, T, shares)) {
        FmOneLayout L;
        fm_one_layout(A, S, T, sms, sd, L);
        if (!A.overflow && workspace) {   // else the partitioned plan, which takes less
            if ((e = fm_one_run(L, R, S, T, a_domain, sketches, ctx->status, sms, st)) != cudaSuccess)
                return cuda_fail(ctx, e, "fm one bucket");
            return estimate();
        }
        A = Arena(workspace, ws_bytes);
    }
    uint32_t I;
    mwj_status s = fm_buckets(ctx, S, shares, &I);
    if (s != MWJ_OK) return s;
    FmLayout L;
    fm_layout(A, I, R, S, T, ctx->dev.num_sms, L);
    if (A.overflow || !workspace)
        return fail(ctx, MWJ_ERR_WORKSPACE, "workspace of %zu bytes, %zu needed", ws_bytes, A.used);

    if ((e = cudaMemsetAsync(sketches, 0, sizeof(uint32_t) * FM_M * (size_t)a_domain, st)) != cudaSuccess)
        return cuda_fail(ctx, e, "memset sketches");
    if ((e = cudaMemsetAsync(L.tcount, 0, sizeof(unsigned int), st)) != cudaSuccess)
        return cuda_fail(ctx, e, "memset count");
    // T's keys, their dense indices, and the sketch of every key's D values
    if ((e = single_table_direct(T.x, T.n, sd.slot2, L.hll, L.tmeta, L.ttbl, single_table_slots(T.n), ctx->status,
                                 sms, st)) != cudaSuccess)
        return cuda_fail(ctx, e, "T keys");
    {
        ProfScope ps_("fm_index", st);
        k_fm_index<<<sms * 4, 256, 0, st>>>((unsigned long long *)L.ttbl, L.tmeta, L.tcount);
    }
    {
        ProfScope ps_("fm_zero", st);
        k_fm_zero<<<sms * 4, 256, 0, st>>>(L.skT, L.tcount);
    }
    if (T.n > 0) {
        ProfScope ps_("fm_tsketch", st);
        const uint64_t groups = ((uint64_t)T.n + 8 * 256 - 1) / (8 * 256);
        const unsigned grid = (unsigned)(groups < (uint64_t)sms * 8 ? groups : (uint64_t)sms * 8);
        k_fm_tsketch<<<grid, 256, 0, st>>>(T.x, T.y, (uint32_t)T.n, (const unsigned long long *)L.ttbl, L.tmeta,
                                          sd.slot2, L.skT);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(ctx, e, "T sketches");
    // R and S by H(B) (Algorithm 1's first level)
    PartSpec ps{0, sd.B, I, -1, 0, 1};
    ps.st = ctx->status;
    if ((e = part_run(S.x, S.y, S.n, ps, PAY_PAIR, L.Sp, L.offS, L.pscratch, L.pscratch_bytes, sms, st)) !=
        cudaSuccess)
        return cuda_fail(ctx, e, "partition S");
    PartSpec pr{1, sd.B, I, -1, 0, 1};
    pr.st = ctx->status;
    pr.dom = (uint32_t)a_domain;
    if ((e = part_run(R.x, R.y, R.n, pr, PAY_PAIR, L.Rp, L.offR, L.pscratch, L.pscratch_bytes, sms, st)) !=
        cudaSuccess)
        return cuda_fail(ctx, e, "partition R");
    FmArgs g{};
    g.Rp = L.Rp; g.Sp = L.Sp; g.offR = L.offR; g.offS = L.offS;
    g.ttbl = (const unsigned long long *)L.ttbl;
    g.tmeta = L.tmeta;
    g.tseed = sd.slot2;
    g.skT = L.skT;
    g.seed_slot = sd.slot;
    g.a_domain = a_domain;
    g.out = sketches;
    g.st = ctx->status;
    const size_t smem = align256(((1u << kFmCapLog2) + 1) * 4) + ((1u << kFmCapLog2) + 1) * FM_M * 4;
    if ((e = cudaFuncSetAttribute(k_fm_probe, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
        cudaSuccess)
        return cuda_fail(ctx, e, "fm probe attribute");
    {
        ProfScope ps_("fm_probe", st);
        k_fm_probe<<<I, FT, smem, st>>>(g);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(ctx, e, "fm probe");
    return estimate();
}
