// linear_l2.cu -- the linear 3-way join R(A,B) S(B,C) T(C,D) with shares
// I = J = 1 (Section 4, Algorithm 1, with one bucket on each side).
//
// Algorithm 1 partitions R by h(B) and T by g(C) so that one bucket of each
// fits the on-chip memory while the matching part of S streams past.  The
// shares are the smallest that make the held buckets fit; on this GPU the
// on-chip memory every SM reaches is the 129 MB L2, and the key tables of a
// relation with a few million distinct keys fit it whole.  Then I = J = 1:
// nothing is partitioned, and the aggregates become three streaming passes,
// each reading one relation once:
//
//   T pass   deg_T(c)                          (T's single table)
//   S pass   w(b)   += deg_T(c)     per (b, c) of S   (S's weight table)
//   R pass   cnt[a] += w(b), total += w(b)  per (a, b) of R
//
// which adds the terms of COUNT = sum over (b,c) in S of deg_R(b) deg_T(c)
// and of cnt(a) = sum over (a,b) in R, (b,c) in S of deg_T(c) in another
// order.  S is keyed by its own B column, so the table gets one insertion
// per distinct b, and runs of equal keys (edge lists sorted by source) are
// summed inside each warp before they reach the L2; the R pass only reads
// the table and adds each run of equal a once.
//
// A star join's GROUP BY is the same three passes with the weight table laid
// out for R's B values instead of S's (star_bucket_run): R is the small
// relation, so its column is the cheap one to size, and S tuples whose b is not
// R's are skipped.  Its COUNT needs no weights: deg_R(b) deg_T(c) summed over S.
#include <algorithm>
#include <type_traits>

#include "group_table.cuh"
#include "internal.h"
#include "linear_l2.h"
#include "skew.h"
#include "warp_runs.cuh"

namespace mwj {
namespace {

constexpr int WT = 256;     // threads per CTA
constexpr int WQ = kRunQ;   // tuples per lane per warp round: one 128-bit load per column
constexpr uint32_t WCHUNK = 32 * WQ;   // tuples per warp round

// Tuples [i, i + WQ) of two int32 columns (fewer at the end); returns how
// many are valid.
__device__ __forceinline__ uint32_t load_pairs(const int32_t *__restrict__ X, const int32_t *__restrict__ Y,
                                               uint32_t n, uint32_t i, bool vec, uint64_t pol,
                                               int32_t (&x)[WQ], int32_t (&y)[WQ]) {
    if (i >= n) return 0;
    if (vec && i + WQ <= n) {
        const int4 a = ld_stream((const int4 *)(X + i), pol);
        const int4 b = ld_stream((const int4 *)(Y + i), pol);
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
        y[0] = b.x; y[1] = b.y; y[2] = b.z; y[3] = b.w;
        return WQ;
    }
    const uint32_t m = min((uint32_t)WQ, n - i);
#pragma unroll
    for (int q = 0; q < WQ; ++q) {
        if ((uint32_t)q < m) {
            x[q] = __ldg(X + i + q);
            y[q] = __ldg(Y + i + q);
        }
    }
    return m;
}

// Hashed degrees: the pair of slots at which the search for key k starts.
__device__ __forceinline__ uint32_t deg_home(uint32_t k, uint32_t seed, uint32_t mask) {
    return slot_of(k, seed, mask) & ~1u;
}

// deg(c) from its home pair (slot s, value v): the first slot holding c, or
// none when a free slot comes first.
__device__ __forceinline__ unsigned long long deg_get(const unsigned long long *__restrict__ slots, uint32_t mask,
                                                      uint32_t c, uint32_t s, ulonglong2 v) {
    for (uint32_t it = 0; it <= mask; it += 2) {
        if ((uint32_t)v.x == c && v.x != kEmpty64) return v.x >> 32;
        if ((uint32_t)v.y == c && v.y != kEmpty64) return v.y >> 32;
        if (v.x == kEmpty64 || v.y == kEmpty64) break;
        s = (s + 2) & mask;
        v = __ldg((const ulonglong2 *)(slots + s));
    }
    return 0ull;
}

// deg(c) += x from its home pair (possibly read before other threads claimed
// slots of it: a claim is a CAS, a key once there stays).
__device__ __forceinline__ void deg_add(unsigned long long *slots, uint32_t mask, uint32_t c, uint32_t s, ulonglong2 v,
                                        uint32_t x, DevStatus *st) {
    const unsigned long long fresh = ((unsigned long long)x << 32) | c;
    for (uint32_t it = 0; it <= mask; it += 2) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            unsigned long long u = q ? v.y : v.x;
            if (u == kEmpty64) {
                u = atomicCAS(slots + s + q, kEmpty64, fresh);
                if (u == kEmpty64) return;
            }
            if ((uint32_t)u == c) {
                atomicAdd(slots + s + q, (unsigned long long)x << 32);
                return;
            }
        }
        s = (s + 2) & mask;
        v = __ldcg((const ulonglong2 *)(slots + s));
    }
    set_status(st, MWJ_ERR_CHECK, 3);   // table full: the sizing step under-estimated
}

// Direct-address weights (the sizing pass chose that layout for S's B
// values): w(b) is the plain 64-bit word W[b - min], added to with 64-bit
// atomics whose results are not needed (exact modulo 2^64, no carry word).
// FILTER: a key outside the table's range is no error but a tuple that joins
// nothing (star joins, whose table holds R's keys).
// wshift: the sum of key k is at W[(k - min) << wshift] (kMetaShift; star joins only).
template <bool FILTER>
__device__ __forceinline__ void w_add_direct(unsigned long long *__restrict__ W, uint32_t wmin, uint32_t wspan,
                                             uint32_t wshift, uint32_t b, unsigned long long x, DevStatus *st) {
    if (b - wmin < wspan)
        atomicAdd(W + ((b - wmin) << (FILTER ? wshift : 0u)), x);
    else if (!FILTER)
        set_status(st, MWJ_ERR_CHECK, 9);   // a key outside the range the sizing pass saw
}

// Packed slots: the slot at which the search for key k starts (key -1: its sum's).
__device__ __forceinline__ uint32_t packed_home(uint32_t k, uint32_t seed, uint32_t mask) {
    return k == kEmptyKey ? mask + 1 : slot_of(k, seed, mask);
}
// w(k) from the first slot (s, value v); 0 when k has none.
__device__ __forceinline__ unsigned long long packed_get(const WTable &w, uint32_t mask, uint32_t packed, uint32_t k,
                                                         uint32_t s, unsigned long long v) {
    if (k == kEmptyKey) return v;
    for (uint32_t it = 0; it < mask && v != kEmpty64 && (uint32_t)v != k; ++it) {
        s = (s + 1) & mask;
        v = __ldg(w.W + s);
    }
    if (v == kEmpty64 || (uint32_t)v != k) return 0ull;
    return (v >> 32) | (packed & 2u ? (unsigned long long)__ldg(w.keys + s) << 32 : 0ull);
}
// w(k) += x (x > 0) from the first slot (s, value v, possibly read before other
// threads claimed it).  A claim stores the key and x's lower word; later adds go to
// the upper half of the slot, and what they carry out of it goes to keys[s].
__device__ __forceinline__ void packed_add(const WTable &w, uint32_t mask, uint32_t k, uint32_t s, unsigned long long v,
                                           unsigned long long x, DevStatus *st) {
    if (k == kEmptyKey) {
        atomicAdd(w.W + mask + 1, x);
        return;
    }
    const unsigned long long lo = x & 0xFFFFFFFFull;
    const uint32_t hx = (uint32_t)(x >> 32);
    for (uint32_t it = 0; it <= mask; ++it) {
        uint32_t h = hx;
        bool mine = false;
        if (v == kEmpty64) {
            v = atomicCAS(w.W + s, kEmpty64, (lo << 32) | k);
            mine = v == kEmpty64;
        }
        if (!mine && (uint32_t)v == k) {
            const unsigned long long old = atomicAdd(w.W + s, lo << 32);
            h += (uint32_t)(((old >> 32) + lo) >> 32);
            mine = true;
        }
        if (mine) {
            if (h) {
                atomicAdd(w.keys + s, h);
                atomicOr(w.meta + kMetaPacked, 2u);
            }
            return;
        }
        s = (s + 1) & mask;
        v = __ldcg(w.W + s);
    }
    set_status(st, MWJ_ERR_CHECK, 7);   // table full: the sizing step under-estimated
}

// w(k[q]) for the lane's tuples q < m (0 for the others) from a weight table
// in either layout; hashed: the key groups are loaded together, then the sums.
template <bool WD, bool STAR = false, bool PACKED = false>
struct WLookup {
    const WTable &w;
    uint32_t mask, min, span, shift, packed;
    __device__ explicit WLookup(const WTable &w_) : w(w_) {
        mask = __ldg(w.meta);
        packed = PACKED ? __ldg(w.meta + kMetaPacked) : 0u;
        min = WD ? __ldg(w.meta + kMetaMin) : 0u;
        span = WD ? __ldg(w.meta + kMetaSpan) : 0u;
        shift = WD && STAR ? __ldg(w.meta + kMetaShift) : 0u;
    }
    __device__ __forceinline__ void operator()(const int32_t (&k)[WQ], uint32_t m, unsigned long long (&x)[WQ]) const {
        if constexpr (WD) {
#pragma unroll
            for (int q = 0; q < WQ; ++q) {
                const uint32_t i = (uint32_t)k[q] - min;
                x[q] = ((uint32_t)q < m && i < span) ? __ldg(w.W + (STAR ? i << shift : i)) : 0ull;
            }
        } else if constexpr (PACKED) {
            uint32_t s[WQ];
            unsigned long long v[WQ];
#pragma unroll
            for (int q = 0; q < WQ; ++q) {
                s[q] = packed_home((uint32_t)k[q], w.seed, mask);
                v[q] = (uint32_t)q < m ? __ldg(w.W + s[q]) : 0ull;
            }
#pragma unroll
            for (int q = 0; q < WQ; ++q)
                x[q] = (uint32_t)q < m ? packed_get(w, mask, packed, (uint32_t)k[q], s[q], v[q]) : 0ull;
        } else {
            uint32_t s[WQ];
            uint4 v[WQ];
#pragma unroll
            for (int q = 0; q < WQ; ++q) {
                s[q] = w_home((uint32_t)k[q], w.seed, mask);
                if ((uint32_t)q < m) v[q] = __ldg((const uint4 *)(w.keys + s[q]));
            }
#pragma unroll
            for (int q = 0; q < WQ; ++q)
                if ((uint32_t)q < m)
                    s[q] = (uint32_t)k[q] == kEmptyKey ? mask + 1 : w_find(w.keys, mask, (uint32_t)k[q], s[q], v[q]);
#pragma unroll
            for (int q = 0; q < WQ; ++q) x[q] = ((uint32_t)q < m && s[q] != kEmptyKey) ? __ldg(w.W + s[q]) : 0ull;
        }
    }
};

// deg(k[q]) in the same way from a direct-address degree table.
struct DegLookup {
    const uint32_t *deg;
    uint32_t min, span;
    __device__ explicit DegLookup(const DegTable &t)
        : deg((const uint32_t *)t.slots), min(__ldg(t.meta + kMetaMin)), span(__ldg(t.meta + kMetaSpan)) {}
    __device__ __forceinline__ void operator()(const int32_t (&k)[WQ], uint32_t m, unsigned long long (&x)[WQ]) const {
#pragma unroll
        for (int q = 0; q < WQ; ++q) {
            const uint32_t i = (uint32_t)k[q] - min;
            x[q] = ((uint32_t)q < m && i < span) ? (unsigned long long)__ldg(deg + i) : 0ull;
        }
    }
};

// A CTA's sums of heavy keys in shared memory, 64 bits in two 32-bit words: a
// 32-bit shared-memory add is one instruction, a 64-bit one a CAS loop, which
// spins when a warp's lanes hold the same key -- and here they do.
struct HeavySums {
    uint32_t lo[kHeavySlots], hi[kHeavySlots];
};
__device__ __forceinline__ void heavy_add(HeavySums &h, int i, unsigned long long x) {
    const uint32_t xl = (uint32_t)x;
    uint32_t xh = (uint32_t)(x >> 32);
    const uint32_t old = atomicAdd(&h.lo[i], xl);
    xh += old + xl < xl ? 1u : 0u;
    if (xh) atomicAdd(&h.hi[i], xh);
}
__device__ __forceinline__ unsigned long long heavy_sum(const HeavySums &h, uint32_t i) {
    return ((unsigned long long)h.hi[i] << 32) | h.lo[i];
}
// The table of heavy keys and zero sums (every thread of the CTA calls this;
// ends with a barrier when there are keys); null when there are none.
__device__ __forceinline__ const uint32_t *heavy_begin(const uint32_t *heavy, uint32_t *buf, HeavySums &sums) {
    const uint32_t *hs = heavy_to_smem(heavy, buf);
    if (!hs) return nullptr;
    for (uint32_t i = threadIdx.x; i < kHeavySlots; i += blockDim.x) sums.lo[i] = sums.hi[i] = 0u;
    __syncthreads();
    return hs;
}

// The source of a weight pass: the degree table of the relation below, or
// (chains of four) its weight table.
struct Source {
    DegTable t;
    WTable w;
};
template <bool SW>
using Lookup = typename std::conditional<SW, WLookup<true>, DegLookup>::type;
template <bool SW>
__device__ __forceinline__ bool source_dense(const Source &src) {
    return __ldg((SW ? src.w.meta : src.t.meta) + kMetaDense) != 0u;
}
template <bool SW>
__device__ __forceinline__ Lookup<SW> make_lookup(const Source &src) {
    if constexpr (SW)
        return WLookup<true>(src.w);
    else
        return DegLookup(src.t);
}

// S pass, both tables in the direct-address layout.  Warp-uniform loop: a warp
// takes 128 consecutive tuples per round, four per lane, and loads its next
// round before it works on this one.  Heavy keys (sampled, see skew.h) are
// summed per CTA in shared memory and added to the table once per CTA, so
// that a key holding a large share of S in no particular order does not funnel
// every warp's adds into one L2 word.
// SW: the source is a weight table (chains of four), not a degree table.
// One warp round: lane l holds tuples (b[q], c[q]), q < m, of 128 consecutive
// ones.  x = the source's value of c; heavy B keys go to the CTA's sums; runs
// of equal b are summed in the warp and added to w(b) once (one
// fire-and-forget 64-bit add).
template <bool SW, bool FILTER>
struct SPass {
    const Lookup<SW> look;
    const WTable &w;
    DevStatus *st;
    const uint32_t *hs;
    HeavySums &hacc;
    uint32_t wmin, wspan, wshift;

    __device__ SPass(const Source &src, const WTable &w_, DevStatus *st_, const uint32_t *hs_,
                     HeavySums &hacc_)
        : look(make_lookup<SW>(src)), w(w_), st(st_), hs(hs_), hacc(hacc_) {
        wmin = __ldg(w.meta + kMetaMin);
        wspan = __ldg(w.meta + kMetaSpan);
        wshift = FILTER ? __ldg(w.meta + kMetaShift) : 0u;
    }

    __device__ __forceinline__ void round(const int32_t (&b)[WQ], const int32_t (&c)[WQ], uint32_t m) {
        unsigned long long x[WQ];
        look(c, m, x);
        if (hs) {
#pragma unroll
            for (int q = 0; q < WQ; ++q) {
                if (x[q] == 0) continue;
                const int hsl = heavy_slot(hs, (uint32_t)b[q]);
                if (hsl >= 0) {
                    heavy_add(hacc, hsl, x[q]);
                    x[q] = 0;
                }
            }
        }
        warp_runs(b, x, m, [&](int32_t key, unsigned long long sum) {
            w_add_direct<FILTER>(w.W, wmin, wspan, wshift, (uint32_t)key, sum, st);
        });
    }

    // the CTA's heavy-key sums into the table (every thread of the CTA calls this)
    __device__ __forceinline__ void flush_heavy(uint32_t nthreads) {
        if (!hs) return;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < kHeavySlots; i += nthreads)
            if (heavy_sum(hacc, i)) w_add_direct<FILTER>(w.W, wmin, wspan, wshift, hs[i], heavy_sum(hacc, i), st);
    }
};

// Tuples [lo, hi) of a column pair in warp rounds of 128 (warp `warp` of
// `warps` takes a consecutive stretch of them: 1 % faster on the sorted friends
// graph and star than every warps-th one), each round's loads issued before
// the previous round is used; round(x, y, m) per round.
template <typename F>
__device__ __forceinline__ void rounds_plain(const int32_t *__restrict__ X, const int32_t *__restrict__ Y,
                                             uint32_t lo, uint32_t hi, uint32_t warp, uint32_t warps, F &&round) {
    const uint32_t lane = threadIdx.x & 31;
    const bool vec = (((uintptr_t)X | (uintptr_t)Y) & 15) == 0 && (lo & 3u) == 0;
    const uint64_t pol = l2_evict_first();
    const uint32_t n = hi;
    const uint32_t all = (hi - lo + WCHUNK - 1) / WCHUNK, per = (all + warps - 1) / warps;
    const uint32_t rounds = min(all, (warp + 1) * per);
    int32_t x[WQ], y[WQ];
    uint32_t m = 0;
    uint32_t r = warp * per;
    if (r < rounds) m = load_pairs(X, Y, n, lo + r * WCHUNK + lane * WQ, vec, pol, x, y);
    while (r < rounds) {
        const uint32_t nr = r + 1;
        int32_t nx[WQ], ny[WQ];
        uint32_t nm = 0;
        if (nr < rounds) nm = load_pairs(X, Y, n, lo + nr * WCHUNK + lane * WQ, vec, pol, nx, ny);
        round(x, y, m);
#pragma unroll
        for (int q = 0; q < WQ; ++q) {
            x[q] = nx[q];
            y[q] = ny[q];
        }
        m = nm;
        r = nr;
    }
}

// Two kernels share the S pass: the direct-address one (both tables in that
// layout) and the general one; the call launches both and the one whose
// layout the sizing passes did not choose returns at once.
//
// The general one: a tuple per lane, few registers, six CTAs per SM.  A hashed
// add is a chain of dependent accesses (key group, perhaps a claim or the next
// group, then the add) that the whole warp waits out; with four tuples per
// lane a warp waited for four such chains, one after the other, and 80
// registers left only three CTAs to fill the waits.  8.4 million id-keyed
// tuples into 1.5 million keys: 0.235 ms with four, 0.154 ms with one.
// FILTER: the table's keys are there already (k_w_keys); others are skipped.
constexpr int GC = 6;
template <bool SW, bool FILTER>
__global__ void __launch_bounds__(WT, GC) k_w_build(const int32_t *__restrict__ Sb, const int32_t *__restrict__ Sc,
                                                    uint32_t n, Source src, WTable w, DevStatus *st) {
    after_previous();
    const bool sd = source_dense<SW>(src), wd = __ldg(w.meta + kMetaDense) != 0u;
    if (sd && wd) return;
    __shared__ uint32_t hbuf[kHeavySlots];
    __shared__ HeavySums hacc;
    const uint32_t *hs = heavy_begin(w.heavy, hbuf, hacc);
    const uint32_t *smeta = SW ? src.w.meta : src.t.meta;
    const uint32_t smask = __ldg(smeta + kMetaMask), smin = sd ? __ldg(smeta + kMetaMin) : 0u,
                   sspan = sd ? __ldg(smeta + kMetaSpan) : 0u;
    const uint32_t wmask = __ldg(w.meta + kMetaMask), wmin = wd ? __ldg(w.meta + kMetaMin) : 0u,
                   wspan = wd ? __ldg(w.meta + kMetaSpan) : 0u;
    const uint32_t wshift = wd && FILTER ? __ldg(w.meta + kMetaShift) : 0u;
    const bool wp = !FILTER && !wd && (__ldg(w.meta + kMetaPacked) & 1u);
    const uint32_t sp = SW && !sd ? __ldg(smeta + kMetaPacked) : 0u;
    auto group = [&](uint32_t s) {   // four keys of the table (FILTER: none is added in this kernel)
        return FILTER ? __ldg((const uint4 *)(w.keys + s)) : __ldcg((const uint4 *)(w.keys + s));
    };
    auto value = [&](uint32_t c) -> unsigned long long {
        if (sd) {
            const uint32_t i = c - smin;
            if (i >= sspan) return 0ull;
            return SW ? __ldg(src.w.W + i) : (unsigned long long)__ldg((const uint32_t *)src.t.slots + i);
        }
        if constexpr (SW) {
            if (sp) {
                const uint32_t s = packed_home(c, src.w.seed, smask);
                return packed_get(src.w, smask, sp, c, s, __ldg(src.w.W + s));
            }
            if (c == kEmptyKey) return __ldg(src.w.W + smask + 1);
            const uint32_t s = w_home(c, src.w.seed, smask);
            const uint32_t at = w_find(src.w.keys, smask, c, s, __ldg((const uint4 *)(src.w.keys + s)));
            return at == kEmptyKey ? 0ull : __ldg(src.w.W + at);
        } else {
            const uint32_t s = deg_home(c, src.t.seed, smask);
            return deg_get(src.t.slots, smask, c, s, __ldg((const ulonglong2 *)(src.t.slots + s)));
        }
    };
    auto add = [&](uint32_t b, uint32_t s, uint4 v, unsigned long long x) {
        if (wd) {
            w_add_direct<FILTER>(w.W, wmin, wspan, wshift, b, x, st);
            return;
        }
        const uint32_t at = b == kEmptyKey ? wmask + 1
                            : FILTER       ? w_find(w.keys, wmask, b, s, v)
                                           : w_claim(w.keys, wmask, b, s, v);
        if (at != kEmptyKey)
            atomicAdd(w.W + at, x);
        else if (!FILTER)
            set_status(st, MWJ_ERR_CHECK, 7);   // table full: the sizing step under-estimated
    };
    auto tuples_in_turn = [&](auto packed) {
        constexpr bool PACKED = decltype(packed)::value;
        const uint32_t T = gridDim.x * WT, lane = threadIdx.x & 31;
        uint64_t i = (uint64_t)blockIdx.x * WT + threadIdx.x;
        int32_t b = 0, c = 0;
        if (i < n) {
            b = __ldg(Sb + i);
            c = __ldg(Sc + i);
        }
        for (; i - lane < n; i += T) {
            int32_t nb = 0, nc = 0;
            if (i + T < n) {
                nb = __ldg(Sb + i + T);
                nc = __ldg(Sc + i + T);
            }
            const bool has = i < n;
            uint32_t s = 0;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            unsigned long long p = 0;
            if (PACKED) {   // the target's slot or key group, with the source's slot
                s = slot_of((uint32_t)b, w.seed, wmask);
                p = __ldcg(w.W + s);
            } else if (!wd) {
                s = w_home((uint32_t)b, w.seed, wmask);
                v = group(s);
            }
            unsigned long long x = has ? value((uint32_t)c) : 0ull;
            if (hs && x) {
                const int hsl = heavy_slot(hs, (uint32_t)b);
                if (hsl >= 0) {
                    heavy_add(hacc, hsl, x);
                    x = 0ull;
                }
            }
            const unsigned long long sum = warp_run_sum1(b, x, has);
            if (sum && PACKED)
                packed_add(w, wmask, (uint32_t)b, s, p, sum, st);
            else if (sum)
                add((uint32_t)b, s, v, sum);
            b = nb;
            c = nc;
        }
    };
    if (wp)
        tuples_in_turn(std::integral_constant<bool, !FILTER>{});
    else
        tuples_in_turn(std::false_type{});
    if (!hs) return;
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < kHeavySlots; j += WT) {
        const unsigned long long x = heavy_sum(hacc, j);
        if (!x) continue;
        if (wp) {
            const uint32_t s = slot_of(hs[j], w.seed, wmask);
            packed_add(w, wmask, hs[j], s, __ldcg(w.W + s), x, st);
            continue;
        }
        const uint32_t s = wd ? 0u : w_home(hs[j], w.seed, wmask);
        add(hs[j], s, wd ? make_uint4(0u, 0u, 0u, 0u) : group(s), x);
    }
}

template <bool SW, bool FILTER>
__global__ void __launch_bounds__(WT) k_w_build_direct(const int32_t *__restrict__ Sb,
                                                       const int32_t *__restrict__ Sc, uint32_t n, Source src,
                                                       WTable w, DevStatus *st) {
    after_previous();
    if (!source_dense<SW>(src) || !__ldg(w.meta + kMetaDense)) return;
    __shared__ uint32_t hbuf[kHeavySlots];
    __shared__ HeavySums hacc;
    const uint32_t *hs = heavy_begin(w.heavy, hbuf, hacc);
    SPass<SW, FILTER> P(src, w, st, hs, hacc);
    const uint32_t warp = (blockIdx.x * WT + threadIdx.x) >> 5, warps = (gridDim.x * WT) >> 5;
    rounds_plain(Sb, Sc, 0u, n, warp, warps,
                 [&](const int32_t (&b)[WQ], const int32_t (&c)[WQ], uint32_t m) { P.round(b, c, m); });
    P.flush_heavy(WT);
}

// Star joins, COUNT: the sum of deg_R(b) deg_T(c) over S, two lookups a tuple and
// no add.  With R's weights, as GROUP BY has them, hot keys in no order cost many
// times as much: a call of 2^26 facts on 1000 uniform keys 2.03 ms, 2^24 on 1000
// Zipf keys 0.58, now 0.128 and 0.055 (where no key is hot, 2^26 facts on 2^20
// uniform keys, 0.45 and 0.49).  DIRECT: both tables direct-address; the call
// launches both kernels.
template <bool DIRECT>
struct Deg32 {
    const DegTable &t;
    const uint32_t mask, min, span;
    const bool dense;
    __device__ explicit Deg32(const DegTable &t_)
        : t(t_), mask(__ldg(t_.meta + kMetaMask)), min(__ldg(t_.meta + kMetaMin)), span(__ldg(t_.meta + kMetaSpan)),
          dense(DIRECT || __ldg(t_.meta + kMetaDense) != 0u) {}
    // deg(k[q]) of the lane's keys q < m, 0 for the others; hashed: the four home
    // pairs are loaded together, as key, degree, key, degree
    __device__ __forceinline__ void operator()(const int32_t (&k)[WQ], uint32_t m, uint32_t (&x)[WQ]) const {
        if (DIRECT || dense) {
#pragma unroll
            for (int q = 0; q < WQ; ++q) {
                const uint32_t i = (uint32_t)k[q] - min;
                x[q] = ((uint32_t)q < m && i < span) ? __ldg((const uint32_t *)t.slots + i) : 0u;
            }
            return;
        }
        uint4 v[WQ];
        uint32_t more = 0;
#pragma unroll
        for (int q = 0; q < WQ; ++q) {
            v[q] = make_uint4(0u, 0u, kEmptyKey, kEmptyKey);
            if ((uint32_t)q < m) v[q] = __ldg((const uint4 *)(t.slots + deg_home((uint32_t)k[q], t.seed, mask)));
        }
#pragma unroll
        for (int q = 0; q < WQ; ++q) {
            const uint32_t c = (uint32_t)k[q];
            x[q] = v[q].x == c ? v[q].y : v[q].z == c ? v[q].w : 0u;
            if (x[q] == 0u && v[q].w != kEmptyKey && (uint32_t)q < m) more |= 1u << q;   // the pair is full
            if (x[q] == kEmptyKey || (uint32_t)q >= m) x[q] = 0u;   // (key -1 against a free slot)
        }
        while (more) {   // rare: the pairs after the home pair
            const uint32_t q = (uint32_t)__ffs((int)more) - 1u;
            more &= more - 1u;
            const uint32_t c = (uint32_t)(q == 0u ? k[0] : q == 1u ? k[1] : q == 2u ? k[2] : k[3]);
            const uint32_t s = (deg_home(c, t.seed, mask) + 2u) & mask;
            const uint32_t d = (uint32_t)deg_get(t.slots, mask, c, s, __ldg((const ulonglong2 *)(t.slots + s)));
#pragma unroll
            for (uint32_t u = 0; u < WQ; ++u)
                if (u == q) x[u] = d;
        }
    }
};

template <bool DIRECT>
__global__ void __launch_bounds__(WT) k_star_total(const int32_t *__restrict__ Sb, const int32_t *__restrict__ Sc,
                                                   uint32_t n, DegTable r, DegTable t,
                                                   unsigned long long *__restrict__ total) {
    after_previous();
    if ((__ldg(r.meta + kMetaDense) && __ldg(t.meta + kMetaDense)) != DIRECT) return;
    __shared__ unsigned long long red[32];
    const Deg32<DIRECT> lr(r), lt(t);
    unsigned long long acc = 0;
    const uint32_t warp = (blockIdx.x * WT + threadIdx.x) >> 5, warps = (gridDim.x * WT) >> 5;
    rounds_plain(Sb, Sc, 0u, n, warp, warps, [&](const int32_t (&b)[WQ], const int32_t (&c)[WQ], uint32_t m) {
        uint32_t x[WQ], y[WQ];
        lr(b, m, x);
        lt(c, m, y);
#pragma unroll
        for (int q = 0; q < WQ; ++q) acc += (unsigned long long)x[q] * y[q];
    });
    acc = block_sum_u64(acc, red);
    if (threadIdx.x == 0 && acc) atomicAdd(total, acc);
}

// Star joins, hashed layout: R's keys into the weight table, so that the S pass
// keeps only the tuples that meet one.
__global__ void __launch_bounds__(WT) k_w_keys(const int32_t *__restrict__ Rb, uint32_t n, WTable w, DevStatus *st) {
    after_previous();
    if (__ldg(w.meta + kMetaDense)) return;
    const uint32_t mask = __ldg(w.meta + kMetaMask);
    for (uint64_t i = (uint64_t)blockIdx.x * WT + threadIdx.x; i < n; i += gridDim.x * WT) {
        const uint32_t k = (uint32_t)__ldg(Rb + i);
        if (k == kEmptyKey) continue;   // its sum has a place of its own
        const uint32_t s = w_home(k, w.seed, mask);
        if (w_claim(w.keys, mask, k, s, __ldcg((const uint4 *)(w.keys + s))) == kEmptyKey)
            set_status(st, MWJ_ERR_CHECK, 11);   // table full: the sizing step under-estimated
    }
}

// R pass (MODE 0: COUNT, MODE 1: GROUP BY A); same loop as the S pass.
// WD: the weight table in the direct-address layout.
// One warp round of the R pass: x = w(b) for the lane's tuples (a[q], b[q]),
// q < m, added to the thread's total and (GROUP BY A) per run of equal a to
// cnt[a].
template <int MODE, bool WD, bool STAR, bool PACKED>
struct RPass {
    const WLookup<WD, STAR, PACKED> look;
    int32_t a_domain;
    unsigned long long *cnt;
    DevStatus *st;
    unsigned long long acc = 0;

    __device__ RPass(const WTable &w, int32_t a_domain_, unsigned long long *cnt_, DevStatus *st_)
        : look(w), a_domain(a_domain_), cnt(cnt_), st(st_) {}

    __device__ __forceinline__ void round(const int32_t (&a)[WQ], const int32_t (&b)[WQ], uint32_t m) {
        unsigned long long x[WQ];
        look(b, m, x);
#pragma unroll
        for (int q = 0; q < WQ; ++q) acc += x[q];
        if (MODE == 1) {
#pragma unroll
            for (int q = 0; q < WQ; ++q)
                if ((uint32_t)q < m && (uint32_t)a[q] >= (uint32_t)a_domain) set_status(st, MWJ_ERR_DOMAIN, a[q]);
            warp_runs(a, x, m, [&](int32_t key, unsigned long long sum) {
                if ((uint32_t)key < (uint32_t)a_domain) atomicAdd(cnt + key, sum);
            });
        }
    }
};

template <int MODE, bool WD, bool STAR = false, bool PACKED = false>
__device__ __forceinline__ void w_probe_pass(const int32_t *__restrict__ Ra, const int32_t *__restrict__ Rb,
                                             uint32_t n, const WTable &w, int32_t a_domain,
                                             unsigned long long *__restrict__ cnt,
                                             unsigned long long *__restrict__ total, DevStatus *st,
                                             unsigned long long *red) {
    RPass<MODE, WD, STAR, PACKED> P(w, a_domain, cnt, st);
    const uint32_t warp = (blockIdx.x * WT + threadIdx.x) >> 5, warps = (gridDim.x * WT) >> 5;
    rounds_plain(Ra, Rb, 0u, n, warp, warps,
                 [&](const int32_t (&a)[WQ], const int32_t (&b)[WQ], uint32_t m) { P.round(a, b, m); });
    const unsigned long long acc = block_sum_u64(P.acc, red);
    if (threadIdx.x == 0 && acc) atomicAdd(total, acc);
}

// The R pass as two kernels in the same way: direct-address weights, hashed.
template <int MODE>
__global__ void __launch_bounds__(WT) k_w_probe(const int32_t *__restrict__ Ra, const int32_t *__restrict__ Rb,
                                                uint32_t n, WTable w, int32_t a_domain,
                                                unsigned long long *__restrict__ cnt,
                                                unsigned long long *__restrict__ total, DevStatus *st) {
    after_previous();
    if (__ldg(w.meta + kMetaDense)) return;
    __shared__ unsigned long long red[32];
    if (__ldg(w.meta + kMetaPacked) & 1u)
        w_probe_pass<MODE, false, false, true>(Ra, Rb, n, w, a_domain, cnt, total, st, red);
    else
        w_probe_pass<MODE, false>(Ra, Rb, n, w, a_domain, cnt, total, st, red);
}

template <int MODE, bool STAR>
__global__ void __launch_bounds__(WT) k_w_probe_direct(const int32_t *__restrict__ Ra,
                                                       const int32_t *__restrict__ Rb, uint32_t n, WTable w,
                                                       int32_t a_domain, unsigned long long *__restrict__ cnt,
                                                       unsigned long long *__restrict__ total, DevStatus *st) {
    after_previous();
    if (!__ldg(w.meta + kMetaDense)) return;
    __shared__ unsigned long long red[32];
    w_probe_pass<MODE, true, STAR>(Ra, Rb, n, w, a_domain, cnt, total, st, red);
}

// T pass: the degrees of the last relation's key column.
//
// Direct-address layout: a warp round is two blocks of 128 consecutive keys,
// four per lane, both loaded, with the next round's loads issued, before they
// are used.  deg[k] += i at the end of every run of equal keys k
// and -= i at its start, i counted inside the block (32-bit adds whose results
// are not needed, exact modulo 2^32): a lane needs only the keys beside its
// own, no search for where a run ends, and a run inside one lane is one add.
// Hashed slots: a key per lane, as in the general S pass.
// In the direct-address layout heavy keys (sampled) are counted per CTA in shared
// memory: keys that hold a large share in no order lie side by side there, and adds
// that meet in an L2 sector wait for one another (this pass over 2^22 and 2^23 keys,
// Zipf 1.1, the most frequent the smallest: 757 and 1500 us without, 392 and 790 with;
// two keys in turn at random 880 and 18).
// The first nheavy CTAs sample the heavy keys of the weight passes instead (the
// medium plan, which has no range pass to do it in).
constexpr int DT = 512;
struct HeavyArgs {
    HeavyCol h[kChainMax - 2];
    uint32_t n;
};
__global__ void __launch_bounds__(DT, 3) k_deg_build(const int32_t *__restrict__ keys, uint32_t n, DegTable t,
                                                     HeavyArgs heavy, DevStatus *st) {
    after_previous();
    __shared__ HeavySample<1024> hsm;
    if (blockIdx.x < heavy.n) {
        const HeavyCol &h = heavy.h[blockIdx.x];
        heavy_sample_cta<DT, 1024>(h.keys, h.n, h.buckets, h.heavy, hsm);
        return;
    }
    const uint32_t cta = blockIdx.x - heavy.n, ctas = gridDim.x - heavy.n;
    const uint32_t mask = t.meta[kMetaMask];
    const bool dense = t.meta[kMetaDense] != 0u;
    const uint32_t kmin = t.meta[kMetaMin], span = t.meta[kMetaSpan];   // (dense)
    uint32_t *deg = (uint32_t *)t.slots;
    const bool vec = ((uintptr_t)keys & 15) == 0;
    const uint64_t pol = l2_evict_first();
    constexpr int G = 2;   // blocks per warp round
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t warp = (cta * DT + threadIdx.x) >> 5, warps = (ctas * DT) >> 5;
    const uint32_t blocks = (n + WCHUNK - 1) / WCHUNK;
    auto load = [&](uint32_t blk, int32_t (&v)[WQ]) -> uint32_t {
        const uint32_t i = blk * WCHUNK + lane * WQ;
        if (blk >= blocks || i >= n) return 0u;
        if (vec && i + WQ <= n) {
            const int4 a = ld_stream((const int4 *)(keys + i), pol);
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
            return WQ;
        }
        const uint32_t m = min((uint32_t)WQ, n - i);
#pragma unroll
        for (int q = 0; q < WQ; ++q)
            if ((uint32_t)q < m) v[q] = __ldg(keys + i + q);
        return m;
    };
    if (!dense) {
        const uint32_t T = ctas * DT;
        uint64_t i = (uint64_t)cta * DT + threadIdx.x;
        int32_t k = i < n ? __ldg(keys + i) : 0;
        for (; i - lane < n; i += T) {
            const int32_t nk = i + T < n ? __ldg(keys + i + T) : 0;
            const uint32_t s = deg_home((uint32_t)k, t.seed, mask);
            const ulonglong2 u = __ldcg((const ulonglong2 *)(t.slots + s));
            const uint32_t len = (uint32_t)warp_run_sum1(k, 1ull, i < n);
            if (len) deg_add(t.slots, mask, (uint32_t)k, s, u, len, st);
            k = nk;
        }
        return;
    }
    // the first keys are on their way while the heavy ones are looked at
    int32_t v[G][WQ];
    uint32_t m[G];
#pragma unroll
    for (int g = 0; g < G; ++g) m[g] = load(warp * G + g, v[g]);
    // heavy keys are counted in shared memory (in the sample's place)
    uint32_t *const hbuf = hsm.key, *const hsum = hsm.cnt;
    static_assert(HeavySample<1024>::slots >= kHeavySlots, "room for the table and its sums");
    for (uint32_t i = threadIdx.x; i < kHeavySlots; i += DT) hsum[i] = 0u;
    const uint32_t *const hs = heavy_to_smem(t.heavy, hbuf);   // (ends with a barrier when there are any)
    auto heavy_counted = [&](uint32_t k, uint32_t x) -> bool {
        const uint32_t s = slot_of(k, kHeavySeed, kHeavySlots - 1), q = hs[s];
        if (q == kEmptyKey) return false;
        const int i = q == k ? (int)s : heavy_slot(hs, k);
        if (i >= 0) atomicAdd(hsum + i, x);
        return i >= 0;
    };
    auto add_word = [&](uint32_t key, uint32_t x) {
        const uint32_t k = key - kmin;
        if (k < span)
            atomicAdd(deg + k, x);
        else
            set_status(st, MWJ_ERR_CHECK, 8);   // a key outside the range the sizing pass saw
    };
    auto block_dense = [&](const int32_t (&v)[WQ], uint32_t m, uint32_t valid, auto &&add) {
        const int32_t prev = __shfl_up_sync(0xffffffffu, v[WQ - 1], 1);
        const int32_t next = __shfl_down_sync(0xffffffffu, v[0], 1);
        if (m == 0) return;
        const uint32_t i0 = lane * WQ;
        uint32_t starts = 0;   // bit q: a run starts at the lane's key q > 0
#pragma unroll
        for (int q = 1; q < WQ; ++q) starts |= (uint32_t)((uint32_t)q < m && v[q] != v[q - 1]) << q;
        int32_t cur = v[0];
        // minus the position where cur's run starts, when it starts in this lane
        uint32_t x = lane == 0 || v[0] != prev ? 0u - i0 : 0u;
        while (starts) {
            const uint32_t q = (uint32_t)__ffs((int)starts) - 1u;
            starts &= starts - 1u;
            add(cur, x + i0 + q);
            cur = q == 1u ? v[1] : (q == 2u ? v[2] : v[3]);
            x = 0u - (i0 + q);
        }
        if (i0 + m == valid || cur != next) x += i0 + m;   // the run ends with this lane
        if (x) add(cur, x);
    };
    auto blocks_in_turn = [&](auto &&add) {
        const uint32_t rounds = (blocks + G - 1) / G;
        uint32_t r = warp;
        while (r < rounds) {
            const uint32_t nr = r + warps;
            int32_t nv[G][WQ];
            uint32_t nm[G];
#pragma unroll
            for (int g = 0; g < G; ++g) nm[g] = load(nr * G + g, nv[g]);
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const uint32_t b0 = (r * G + g) * WCHUNK;
                block_dense(v[g], m[g], b0 < n ? min(WCHUNK, n - b0) : 0u, add);
            }
#pragma unroll
            for (int g = 0; g < G; ++g) {
                m[g] = nm[g];
#pragma unroll
                for (int q = 0; q < WQ; ++q) v[g][q] = nv[g][q];
            }
            r = nr;
        }
    };
    if (!hs) {
        blocks_in_turn([&](int32_t key, uint32_t x) { add_word((uint32_t)key, x); });
        return;
    }
    blocks_in_turn([&](int32_t key, uint32_t x) {
        if (!heavy_counted((uint32_t)key, x)) add_word((uint32_t)key, x);
    });
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < kHeavySlots; j += DT)
        if (hsum[j]) add_word(hs[j], hsum[j]);
}

// ---------------------------------------------------------------------------
// small chains
// ---------------------------------------------------------------------------
//
// A call on a few thousand tuples spends its time between kernels: nine
// launches of 2 to 4 us each, most of them sizing and choosing layouts.  Two
// ways around that, both on hashed tables of two slots per tuple, which need
// neither:
//
//  * up to kSmallMax tuples per relation the whole call is one launch: one
//    thread-block cluster does the passes in turn, with the cluster's hardware
//    barrier between them (no flags in memory, no co-residency to ask for
//    beyond the cluster itself).  A cluster is at most 16 SMs.
//  * up to kMediumMax: four launches, one that empties the tables and says how
//    large they are, then the general passes on the whole GPU.
//
// Device time of a call with uniform keys, GROUP BY A (2^20 groups; a replayed
// graph of ten), and in brackets of calls queued back to back by the binding, us:
//
//   tuples per relation   nine launches   four launches   one cluster
//   2^10                  26 (41)         11 (26)         20 (23)
//   2^14                  27 (38)         13 (25)         22 (24)
//   2^16                  28 (39)         15 (26)         40 (41)
//   2^18                  34 (39)         20 (26)         102 (104)
//   2^19                  41 (42)         31 (32)
//   2^20                  56 (56)         56 (55)
//
// Up to 2^14 what a queue of calls waits for is the host, and the cluster's one
// launch is the cheapest there.  (id keys at 2^20, before launches overlapped:
// nine 109, four 75.)
constexpr int CT = 1024;              // threads per CTA
constexpr int kSmallCtas = 16;        // CTAs of the largest cluster
constexpr int64_t kSmallMax = 1 << 14;      // tuples per relation
constexpr int64_t kMediumMax = 1 << 19;
constexpr int64_t kMediumHeavy = 1 << 16;   // relations above it have their heavy keys sampled
constexpr int64_t kSmallGroups = 1 << 21;   // groups zeroed by the cluster

struct SmallArgs {
    mwj_rel rel[kChainMax];
    int nrel, mode;
    DegTable deg;
    WTable w[kChainMax - 2];
    uint32_t dmask, wmask[kChainMax - 2];
    int32_t a_domain;
    unsigned long long *cnt, *total;
    DevStatus *st;
};

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}

// Tables written in this kernel are read through the L2 (ld.cg).
__device__ __forceinline__ unsigned long long small_deg(const DegTable &t, uint32_t mask, uint32_t c, uint32_t s,
                                                        ulonglong2 v) {
    for (uint32_t it = 0; it <= mask; it += 2) {
        if ((uint32_t)v.x == c && v.x != kEmpty64) return v.x >> 32;
        if ((uint32_t)v.y == c && v.y != kEmpty64) return v.y >> 32;
        if (v.x == kEmpty64 || v.y == kEmpty64) break;
        s = (s + 2) & mask;
        v = __ldcg((const ulonglong2 *)(t.slots + s));
    }
    return 0ull;
}

__device__ __forceinline__ unsigned long long small_w(const WTable &w, uint32_t mask, uint32_t k, uint32_t s, uint4 v) {
    if (k == kEmptyKey) return __ldcg(w.W + mask + 1);
    for (uint32_t it = 0; it <= mask; it += 4) {
        const uint32_t at = v.x == k ? 0u : v.y == k ? 1u : v.z == k ? 2u : v.w == k ? 3u : 4u;
        if (at < 4u) return __ldcg(w.W + s + at);
        if (v.w == kEmptyKey) break;
        s = (s + 4) & mask;
        v = __ldcg((const uint4 *)(w.keys + s));
    }
    return 0ull;
}

// Empty tables and zero outputs (thread t of T).
__device__ __forceinline__ void small_clear(const SmallArgs &g, uint32_t t, uint32_t T) {
    for (uint32_t s = t; s <= g.dmask / 2; s += T) ((ulonglong2 *)g.deg.slots)[s] = make_ulonglong2(kEmpty64, kEmpty64);
    for (int k = 0; k < g.nrel - 2; ++k) {
        const uint32_t m = g.wmask[k];
        for (uint32_t s = t; s <= m / 4; s += T)
            ((uint4 *)g.w[k].keys)[s] = make_uint4(kEmptyKey, kEmptyKey, kEmptyKey, kEmptyKey);
        for (uint32_t s = t; s <= m / 2; s += T) ((ulonglong2 *)g.w[k].W)[s] = make_ulonglong2(0ull, 0ull);
        if (t == 0) g.w[k].W[m + 1] = 0ull;
    }
    if (g.mode == 1)
        for (uint32_t a = t; a < (uint32_t)g.a_domain; a += T) g.cnt[a] = 0ull;
    if (t == 0) *g.total = 0ull;
}

__global__ void __launch_bounds__(WT) k_chain_clear(SmallArgs g) {
    after_previous();
    const uint32_t t = blockIdx.x * WT + threadIdx.x;
    small_clear(g, t, gridDim.x * WT);
    if (t == 0) {
        g.deg.meta[kMetaMask] = g.dmask;
        g.deg.meta[kMetaDense] = 0u;
        for (int k = 0; k < g.nrel - 2; ++k) {
            g.w[k].meta[kMetaMask] = g.wmask[k];
            g.w[k].meta[kMetaDense] = 0u;
            g.w[k].meta[kMetaPacked] = 0u;
        }
    }
}

__global__ void __launch_bounds__(CT) k_chain_small(SmallArgs g) {
    constexpr int U = 4;   // tuples per thread in flight
    __shared__ unsigned long long red[32];
    const uint32_t T = gridDim.x * CT, t = blockIdx.x * CT + threadIdx.x, lane = threadIdx.x & 31;
    small_clear(g, t, T);
    cluster_barrier();
    {   // degrees of the last relation
        const mwj_rel r = g.rel[g.nrel - 1];
        const uint32_t n = (uint32_t)r.n, mask = g.dmask;
        for (uint32_t i = t; i - lane < n; i += U * T) {
            int32_t k[U];
            uint32_t s[U], len[U];
            ulonglong2 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) k[u] = i + u * T < n ? __ldg(r.x + i + u * T) : 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                s[u] = deg_home((uint32_t)k[u], g.deg.seed, mask);
                if (i + u * T < n) v[u] = __ldcg((const ulonglong2 *)(g.deg.slots + s[u]));
                len[u] = (uint32_t)warp_run_sum1(k[u], 1ull, i + u * T < n);
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (len[u]) deg_add(g.deg.slots, mask, (uint32_t)k[u], s[u], v[u], len[u], g.st);
        }
    }
    cluster_barrier();
    for (int p = 0; p < g.nrel - 2; ++p) {   // weights, from the bottom up
        const mwj_rel r = g.rel[g.nrel - 2 - p];
        const WTable &w = g.w[p];
        const uint32_t n = (uint32_t)r.n, mask = g.wmask[p];
        for (uint32_t i = t; i - lane < n; i += U * T) {
            int32_t b[U], c[U];
            uint32_t s[U];
            uint4 v[U];
            unsigned long long x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool has = i + u * T < n;
                b[u] = has ? __ldg(r.x + i + u * T) : 0;
                c[u] = has ? __ldg(r.y + i + u * T) : 0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                s[u] = w_home((uint32_t)b[u], w.seed, mask);
                if (i + u * T < n) v[u] = __ldcg((const uint4 *)(w.keys + s[u]));
            }
            if (p == 0) {
                uint32_t ds[U];
                ulonglong2 dv[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    ds[u] = deg_home((uint32_t)c[u], g.deg.seed, g.dmask);
                    if (i + u * T < n) dv[u] = __ldcg((const ulonglong2 *)(g.deg.slots + ds[u]));
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    x[u] = i + u * T < n ? small_deg(g.deg, g.dmask, (uint32_t)c[u], ds[u], dv[u]) : 0ull;
            } else {
                const WTable &src = g.w[p - 1];
                const uint32_t sm = g.wmask[p - 1];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t q = w_home((uint32_t)c[u], src.seed, sm);
                    x[u] = i + u * T < n
                               ? small_w(src, sm, (uint32_t)c[u], q, __ldcg((const uint4 *)(src.keys + q)))
                               : 0ull;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned long long sum = warp_run_sum1(b[u], x[u], i + u * T < n);
                if (!sum) continue;
                const uint32_t k = (uint32_t)b[u];
                const uint32_t at = k == kEmptyKey ? mask + 1 : w_claim(w.keys, mask, k, s[u], v[u]);
                if (at != kEmptyKey)
                    atomicAdd(w.W + at, sum);
                else
                    set_status(g.st, MWJ_ERR_CHECK, 7);   // cannot happen: two slots per tuple
            }
        }
        cluster_barrier();
    }
    // R
    const mwj_rel r = g.rel[0];
    const WTable &w = g.w[g.nrel - 3];
    const uint32_t n = (uint32_t)r.n, mask = g.wmask[g.nrel - 3];
    unsigned long long acc = 0;
    for (uint32_t i = t; i - lane < n; i += U * T) {
        int32_t a[U], b[U];
        uint32_t s[U];
        uint4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool has = i + u * T < n;
            a[u] = has && g.mode == 1 ? __ldg(r.x + i + u * T) : 0;
            b[u] = has ? __ldg(r.y + i + u * T) : 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            s[u] = w_home((uint32_t)b[u], w.seed, mask);
            if (i + u * T < n) v[u] = __ldcg((const uint4 *)(w.keys + s[u]));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool has = i + u * T < n;
            const unsigned long long x = has ? small_w(w, mask, (uint32_t)b[u], s[u], v[u]) : 0ull;
            acc += x;
            if (g.mode == 1) {
                const unsigned long long sum = warp_run_sum1(a[u], x, has);
                if (has && (uint32_t)a[u] >= (uint32_t)g.a_domain)
                    set_status(g.st, MWJ_ERR_DOMAIN, a[u]);
                else if (sum)
                    atomicAdd(g.cnt + a[u], sum);
            }
        }
    }
    acc = block_sum_u64(acc, red);
    if (threadIdx.x == 0 && acc) atomicAdd(g.total, acc);
}

bool chain_within(const mwj_rel *rel, int nrel, int64_t most) {
    for (int k = 0; k < nrel; ++k)
        if (rel[k].n > most) return false;
    return true;
}
// CTAs of the cluster that takes the call: one per 1024 tuples (and per 16K groups to
// zero), a power of two up to 16; 0: the call is too large for one.
int chain_cluster(const mwj_rel *rel, int nrel, int mode, int32_t a_domain) {
    if (!chain_within(rel, nrel, kSmallMax) || (mode == 1 && a_domain > kSmallGroups)) return 0;
    int64_t most = 1;
    for (int k = 0; k < nrel; ++k) most = rel[k].n > most ? rel[k].n : most;
    const int64_t want = (most + CT - 1) / CT, wantg = mode == 1 ? ((int64_t)a_domain + 16383) / 16384 : 1;
    int ctas = 1;
    while (ctas < kSmallCtas && (ctas < want || ctas < wantg)) ctas <<= 1;
    return ctas;
}

// Tables as one_bucket_layout laid them out (at least two slots per tuple).
SmallArgs small_args(const OneBucket &L, const mwj_rel *rel, int nrel, int mode, int32_t a_domain,
                     unsigned long long *cnt, unsigned long long *total, DevStatus *status) {
    SmallArgs g{};
    for (int k = 0; k < nrel; ++k) g.rel[k] = rel[k];
    g.nrel = nrel;
    g.mode = mode;
    g.deg = L.deg;
    g.dmask = (uint32_t)single_table_slots(rel[nrel - 1].n) - 1u;
    for (int k = 0; k < nrel - 2; ++k) {
        g.w[k] = L.w[k];
        g.wmask[k] = (uint32_t)w_table_slots(rel[nrel - 2 - k].n) - 1u;
    }
    g.a_domain = a_domain;
    g.cnt = cnt;
    g.total = total;
    g.st = status;
    return g;
}

struct ClusterLaunch {
    cudaLaunchConfig_t c{};
    cudaLaunchAttribute at[1];
    ClusterLaunch(int ctas, cudaStream_t st) {
        c.gridDim = dim3(ctas);
        c.blockDim = dim3(CT);
        c.stream = st;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = ctas;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        c.attrs = at;
        c.numAttrs = 1;
    }
};
cudaError_t chain_small(const SmallArgs &g, int ctas, cudaStream_t st) {
    const ClusterLaunch l(ctas, st);
    ProfScope ps_("chain_small", st);
    return cudaLaunchKernelEx(&l.c, k_chain_small, g);
}

// CTAs of a grid-stride pass: per_sm of them on every SM (what the registers
// leave room for), no more warps than rounds of per_warp tuples.
uint32_t pass_grid(uint32_t n, int num_sms, uint32_t per_sm, uint32_t per_warp) {
    const uint64_t want = ((uint64_t)n + per_warp * (WT / 32) - 1) / (per_warp * (WT / 32));
    const uint64_t full = (uint64_t)num_sms * per_sm;
    return (uint32_t)(want < full ? (want ? want : 1) : full);
}
constexpr uint32_t kDirectCtas = 5, kProbeCtas = 5, kHashedProbeCtas = 4;

}  // namespace

size_t w_table_slots(int64_t nS) { return single_table_slots(nS); }

int chain_cluster_limit() {
    for (int ctas = kSmallCtas; ctas > 1; ctas >>= 1) {
        const ClusterLaunch l(ctas, nullptr);
        int n = 0;
        if ((ctas <= 8 || cudaFuncSetAttribute(k_chain_small, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
            cudaOccupancyMaxActiveClusters(&n, k_chain_small, &l.c) == cudaSuccess && n > 0)
            return ctas;
        cudaGetLastError();
    }
    return 1;
}

namespace {

cudaError_t deg_build(const int32_t *keys, int64_t nkeys, const DegTable &t, DevStatus *status, int num_sms,
                      cudaStream_t st, const HeavyArgs &heavy = HeavyArgs{}) {
    const uint32_t n = (uint32_t)nkeys;
    if (n + heavy.n == 0) return cudaSuccess;
    const uint32_t groups = (n + WQ * DT - 1) / (WQ * DT), full = (uint32_t)num_sms * 3;
    ProfScope ps_("t_insert", st);
    return launch_after(k_deg_build, heavy.n + (groups < full ? (groups ? groups : 1u) : full), DT, st, keys, n, t, heavy,
                        status);
}

enum Pass { PASS_DEGREES, PASS_WEIGHTS, PASS_STAR };   // what a weight pass looks up, or a star's S pass

// hashed_only: the tables are known to be hashed (the other kernel of the pass
// is not launched)
cudaError_t w_table_build(const mwj_rel &S, const Source &src, Pass pass, const WTable &w, DevStatus *status,
                          int num_sms, cudaStream_t st, bool hashed_only = false) {
    if (S.n <= 0) return cudaSuccess;
    const uint32_t n = (uint32_t)S.n;
    auto direct = pass == PASS_STAR      ? k_w_build_direct<false, true>
                  : pass == PASS_WEIGHTS ? k_w_build_direct<true, false>
                                         : k_w_build_direct<false, false>;
    auto hashed = pass == PASS_STAR      ? k_w_build<false, true>
                  : pass == PASS_WEIGHTS ? k_w_build<true, false>
                                         : k_w_build<false, false>;
    if (!hashed_only) {
        ProfScope ps_(pass == PASS_STAR ? "star_probe" : "w_build", st);
        const cudaError_t e = launch_after(direct, pass_grid(n, num_sms, kDirectCtas, WCHUNK), WT, st, S.x, S.y, n, src, w,
                                           status);
        if (e != cudaSuccess) return e;
    }
    ProfScope ps_(pass == PASS_STAR ? "star_probe_hashed" : "w_build_hashed", st);
    return launch_after(hashed, pass_grid(n, num_sms, GC, 32), WT, st, S.x, S.y, n, src, w, status);
}

cudaError_t w_table_probe(const mwj_rel &R, const WTable &w, int mode, int32_t a_domain, unsigned long long *cnt,
                          unsigned long long *total, DevStatus *status, int num_sms, cudaStream_t st,
                          bool hashed_only = false, bool star = false) {
    if (R.n <= 0) return cudaSuccess;
    const uint32_t n = (uint32_t)R.n;
    auto direct = star ? k_w_probe_direct<1, true> : mode == 1 ? k_w_probe_direct<1, false> : k_w_probe_direct<0, false>;
    auto hashed = mode == 1 ? k_w_probe<1> : k_w_probe<0>;
    if (!hashed_only) {
        ProfScope ps_(mode == 1 ? "w_probe_groupby" : "w_probe_count", st);
        const cudaError_t e = launch_after(direct, pass_grid(n, num_sms, mode == 1 ? kProbeCtas : kProbeCtas + 1, WCHUNK), WT,
                                           st, R.x, R.y, n, w, a_domain, cnt, total, status);
        if (e != cudaSuccess) return e;
    }
    ProfScope ps_(mode == 1 ? "w_probe_groupby_hashed" : "w_probe_count_hashed", st);
    return launch_after(hashed, pass_grid(n, num_sms, mode == 1 ? kHashedProbeCtas : kHashedProbeCtas + 1, WCHUNK), WT, st,
                        R.x, R.y, n, w, a_domain, cnt, total, status);
}

}  // namespace

namespace {

// Many groups are zeroed by a memset of their own: the CTAs that clear them beside
// the tables do not reach memory speed (2^20 tuples a relation, 2^26, 2^27 and 2^28
// groups 178, 288 and 499 us in all that way, 145, 214 and 353 with the memset).
constexpr int32_t kMemsetGroups = 1 << 24;
cudaError_t zero_groups(int mode, int32_t a_domain, unsigned long long *cnt, bool *zeroed, cudaStream_t st) {
    *zeroed = mode == 1 && a_domain > kMemsetGroups;
    return *zeroed ? cudaMemsetAsync(cnt, 0, sizeof(*cnt) * (size_t)a_domain, st) : cudaSuccess;
}

// The small plans; false when the call is larger.  A device, partition or stream
// whose SMs have no room for the cluster gets the four launches.
bool small_run(const OneBucket &L, const mwj_rel *rel, int nrel, int mode, int32_t a_domain, unsigned long long *cnt,
               unsigned long long *total, DevStatus *status, const DevInfo &dev, cudaStream_t st, cudaError_t *e) {
    if (!chain_within(rel, nrel, kMediumMax)) return false;
    const int num_sms = dev.num_sms;
    SmallArgs g = small_args(L, rel, nrel, mode, a_domain, cnt, total, status);
    DegTable deg = L.deg;
    deg.heavy = nullptr;   // (not sampled)
    const int ctas = chain_cluster(rel, nrel, mode, a_domain);
    if (ctas > 0 && ctas <= dev.cluster) {
        if ((*e = chain_small(g, ctas, st)) == cudaSuccess) return true;
        cudaGetLastError();   // refused (nothing of it runs): not the call's error
    }
    {
        ProfScope ps_("chain_clear", st);
        if ((*e = launch_after(k_chain_clear, num_sms * 2, WT, st, g)) != cudaSuccess) return true;
    }
    HeavyArgs heavy{};
    for (int k = 0; k < nrel - 2; ++k) {
        const mwj_rel &r = rel[nrel - 2 - k];
        if (r.n > kMediumHeavy)
            heavy.h[heavy.n++] = HeavyCol{r.x, (uint32_t)r.n, kWHeavyBuckets, (uint32_t *)L.w[k].heavy};
    }
    if ((*e = deg_build(rel[nrel - 1].x, rel[nrel - 1].n, deg, status, num_sms, st, heavy)) != cudaSuccess) return true;
    Source src{};
    src.t = deg;
    for (int k = 0; k < nrel - 2; ++k) {
        WTable w = L.w[k];
        if (rel[nrel - 2 - k].n <= kMediumHeavy) w.heavy = nullptr;
        if ((*e = w_table_build(rel[nrel - 2 - k], src, k > 0 ? PASS_WEIGHTS : PASS_DEGREES, w, status, num_sms, st,
                                true)) != cudaSuccess)
            return true;
        src.w = w;
    }
    *e = w_table_probe(rel[0], L.w[nrel - 3], mode, a_domain, cnt, total, status, num_sms, st, true);
    return true;
}

}  // namespace

void one_bucket_layout(Arena &A, const mwj_rel *rel, int nrel, int num_sms, OneBucket &L) {
    L = OneBucket{};
    L.deg.slots = A.take<unsigned long long>(single_table_slots(rel[nrel - 1].n) + 2);
    L.deg.meta = A.take<uint32_t>(kMetaWords);
    for (int k = 0; k < nrel - 2; ++k) {
        const size_t ws = w_table_slots(rel[nrel - 2 - k].n) + 2;
        L.w[k].W = A.take<unsigned long long>(ws);
        L.w[k].keys = A.take<uint32_t>(ws);
        L.w[k].meta = A.take<uint32_t>(kMetaWords);
        L.w[k].heavy = A.take<uint32_t>(kHeavyTableWords);
    }
    for (int k = 0; k < nrel - 1; ++k) L.hll[k] = A.take<unsigned int>(hll_scratch_registers(num_sms));
    L.deg.heavy = A.take<uint32_t>(kHeavyTableWords);
}

cudaError_t one_bucket_run(OneBucket &L, const mwj_rel *rel, int nrel, const Seeds &sd, int mode, int32_t a_domain,
                           unsigned long long *cnt, unsigned long long *total, DevStatus *status, const DevInfo &dev,
                           cudaStream_t st) {
    cudaError_t e;
    const int num_sms = dev.num_sms;
    const mwj_rel &last = rel[nrel - 1];
    const uint32_t seeds[kChainMax - 2] = {nrel == 3 ? sd.slot : sd.slot ^ sd.D, sd.slot};
    // the key columns (of every relation but R); a column that plays two
    // parts (a self-join) is read once
    SizeCol cols[kSizeCols];
    uint32_t ncols = 0;
    auto add = [&](const mwj_rel &r, uint32_t seed, uint32_t *meta, uint64_t reserve) {
        for (uint32_t q = 0; q < ncols; ++q) {
            if (cols[q].keys == r.x && cols[q].n == (uint32_t)r.n) {
                cols[q].meta[cols[q].ntargets] = meta;
                cols[q].reserve[cols[q].ntargets] = reserve;
                cols[q].range[cols[q].ntargets++] = reserve;
                return;
            }
        }
        cols[ncols] = SizeCol{r.x, (uint32_t)r.n, seed, L.hll[ncols], {meta}, {reserve}, {reserve}, 1u};
        cols[ncols].weights = true;
        ++ncols;
    };
    HeavyCol heavy[kSizeCols];
    ClearTable clear[kSizeCols];
    L.deg.seed = sd.slot2;
    const uint32_t *const own = L.deg.heavy;
    add(last, L.deg.seed, L.deg.meta, single_table_slots(last.n));
    clear[0] = ClearTable{L.deg.slots, nullptr, L.deg.meta};
    for (int k = 0; k < nrel - 2; ++k) {
        const mwj_rel &r = rel[nrel - 2 - k];
        WTable &w = L.w[k];
        w.seed = seeds[k];
        add(r, w.seed, w.meta, w_table_slots(r.n));
        heavy[k] = HeavyCol{r.x, (uint32_t)r.n, kWHeavyBuckets, (uint32_t *)w.heavy};
        if (r.x == last.x && r.n == last.n) L.deg.heavy = w.heavy;   // one sample does
        clear[k + 1] = ClearTable{w.W, w.keys, w.meta};
    }
    if (small_run(L, rel, nrel, mode, a_domain, cnt, total, status, dev, st, &e)) return e;
    uint32_t nheavy = (uint32_t)nrel - 2u;
    if (L.deg.heavy == own)
        heavy[nheavy++] = HeavyCol{last.x, (uint32_t)last.n, kWHeavyBuckets, (uint32_t *)own, true};
    if ((e = size_columns(cols, ncols, heavy, nheavy, true, num_sms, st)) != cudaSuccess) return e;
    bool zeroed;
    if ((e = zero_groups(mode, a_domain, cnt, &zeroed, st)) != cudaSuccess) return e;
    const bool zero = mode == 1 && !zeroed;
    if ((e = tables_clear(clear, (uint32_t)nrel - 1u, zero ? cnt : nullptr, zero ? (uint64_t)a_domain : 0ull, total,
                          num_sms, st)) != cudaSuccess)
        return e;
    if ((e = deg_build(last.x, last.n, L.deg, status, num_sms, st)) != cudaSuccess) return e;
    Source src{};
    src.t = L.deg;
    for (int k = 0; k < nrel - 2; ++k) {
        if ((e = w_table_build(rel[nrel - 2 - k], src, k > 0 ? PASS_WEIGHTS : PASS_DEGREES, L.w[k], status, num_sms, st)) != cudaSuccess) return e;
        src.w = L.w[k];
    }
    return w_table_probe(rel[0], L.w[nrel - 3], mode, a_domain, cnt, total, status, num_sms, st);
}

// The weights are R's, not S's, except in a small call (a chain like any other):
// room for either, so that what a call asks for grows with its sizes.
static int64_t star_weights(const mwj_rel &R, const mwj_rel &S) { return std::max(R.n, std::min(S.n, kMediumMax)); }

void star_bucket_layout(Arena &A, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, int num_sms, OneBucket &L) {
    mwj_rel w = R;
    w.n = star_weights(R, S);
    const mwj_rel rel[3] = {R, w, T};
    one_bucket_layout(A, rel, 3, num_sms, L);
}

namespace {

// COUNT: R's degrees in the place of the weight table.
cudaError_t star_count(const OneBucket &L, const SizeCol (&cols)[2], const mwj_rel &R, const mwj_rel &S, const mwj_rel &T,
                       unsigned long long *total, DevStatus *status, int num_sms, cudaStream_t st) {
    cudaError_t e;
    const DegTable r{L.w[0].W, L.w[0].meta, L.w[0].seed, nullptr};
    const ClearTable clear[2] = {ClearTable{L.deg.slots, nullptr, L.deg.meta}, ClearTable{r.slots, nullptr, r.meta}};
    if ((e = size_columns(cols, 2, nullptr, 0, true, num_sms, st)) != cudaSuccess) return e;
    if ((e = tables_clear(clear, 2, nullptr, 0ull, total, num_sms, st)) != cudaSuccess) return e;
    if ((e = deg_build(T.x, T.n, L.deg, status, num_sms, st)) != cudaSuccess) return e;
    if ((e = deg_build(R.y, R.n, r, status, num_sms, st)) != cudaSuccess) return e;
    if (S.n <= 0) return cudaSuccess;
    const uint32_t n = (uint32_t)S.n;
    {
        ProfScope ps_("star_count", st);
        e = launch_after(k_star_total<true>, pass_grid(n, num_sms, kDirectCtas, WCHUNK), WT, st, S.x, S.y, n, r, L.deg, total);
        if (e != cudaSuccess) return e;
    }
    ProfScope ps_("star_count_hashed", st);
    return launch_after(k_star_total<false>, pass_grid(n, num_sms, kHashedProbeCtas, WCHUNK), WT, st, S.x, S.y, n, r, L.deg,
                        total);
}

}  // namespace

cudaError_t star_bucket_run(OneBucket &L, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, const Seeds &sd, int mode,
                            int32_t a_domain, unsigned long long *cnt, unsigned long long *total, DevStatus *status,
                            const DevInfo &dev, cudaStream_t st) {
    cudaError_t e;
    const int num_sms = dev.num_sms;
    L.deg.seed = sd.slot2;
    L.deg.heavy = nullptr;   // (a dimension's keys hardly repeat)
    L.w[0].seed = sd.slot;
    const mwj_rel rel[3] = {R, S, T};
    if (small_run(L, rel, 3, mode, a_domain, cnt, total, status, dev, st, &e)) return e;
    const uint64_t tr = single_table_slots(T.n), rr = w_table_slots(R.n);
    const uint64_t rw = w_table_slots(star_weights(R, S));   // what is reserved
    const SizeCol cols[2] = {SizeCol{T.x, (uint32_t)T.n, sd.slot2, L.hll[0], {L.deg.meta}, {tr}, {tr}, 1u},
                             SizeCol{R.y, (uint32_t)R.n, sd.slot, L.hll[1], {L.w[0].meta}, {rr}, {rr}, 1u, mode == 1 ? rw : 0ull}};
    if (mode == 0) return star_count(L, cols, R, S, T, total, status, num_sms, st);
    const HeavyCol heavy{S.x, (uint32_t)S.n, kWHeavyBuckets, (uint32_t *)L.w[0].heavy};
    const ClearTable clear[2] = {ClearTable{L.deg.slots, nullptr, L.deg.meta},
                                 ClearTable{L.w[0].W, L.w[0].keys, L.w[0].meta}};
    if ((e = size_columns(cols, 2, &heavy, 1, true, num_sms, st)) != cudaSuccess) return e;
    bool zeroed;
    if ((e = zero_groups(mode, a_domain, cnt, &zeroed, st)) != cudaSuccess) return e;
    const bool zero = mode == 1 && !zeroed;
    if ((e = tables_clear(clear, 2, zero ? cnt : nullptr, zero ? (uint64_t)a_domain : 0ull, total, num_sms, st)) !=
        cudaSuccess)
        return e;
    if ((e = deg_build(T.x, T.n, L.deg, status, num_sms, st)) != cudaSuccess) return e;
    if (R.n > 0) {
        ProfScope ps_("star_keys", st);
        if ((e = launch_after(k_w_keys, pass_grid((uint32_t)R.n, num_sms, 8, 32), WT, st, R.y, (uint32_t)R.n, L.w[0],
                              status)) != cudaSuccess)
            return e;
    }
    Source src{};
    src.t = L.deg;
    if ((e = w_table_build(S, src, PASS_STAR, L.w[0], status, num_sms, st)) != cudaSuccess) return e;
    return w_table_probe(R, L.w[0], mode, a_domain, cnt, total, status, num_sms, st, false, true);
}

}  // namespace mwj
