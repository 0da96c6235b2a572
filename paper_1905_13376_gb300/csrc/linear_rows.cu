// linear_rows.cu -- row output of the linear join R(A,B) S(B,C) T(C,D) with one
// bucket on each side.
//
// R is grouped by B (b -> [a]) and T by C (c -> [d]) in global memory, both read
// through the L2 by every SM (rgroup_build), and S is streamed past them once
// without being partitioned: an S tuple (b, c) makes |R[b]| |T[c]| rows.
//
//   pass 1  the rows of every chunk of S, at the place that one atomic on the
//           number of rows reserves for the chunk; tuples that make more than
//           kBigRows are set aside
//   pass 2  the rows of those, cut into pieces of kPiece that are dealt out
//           evenly to the warps of the whole GPU
//
// Rows past the capacity are counted only.
//
// A warp lays the rows of its 32 tuples side by side and writes 32 consecutive
// ones per step, so that the output, most of the traffic, is written in whole
// 512-byte stretches whatever the degrees are.
//
// 2^21 R, 2^22 S and 2^20 T tuples, 2^23 rows: the partitioned plan (R and S by
// H(B), T's bucket images with lists, rows per bucket) took 0.77 ms in 25
// launches, this one 0.29 ms in 17 (0.34 with a pass of its own that counts every
// chunk's rows and a scan that places them).  The lists cost about as much as the
// partitions did, but S is not moved and a row is not looked for in a
// shared-memory table.
//
// kBigRows: a warp writes its own tuples' rows at one step of 32 rows per 0.37 us,
// so a few tuples of hundreds of rows leave the rest of the GPU idle; pass 2
// spreads them (ms, and in brackets the partitioned plan):
//
//   tuples x rows       set aside above 4096, one at a time   now
//   64 x 4032           1.26                                  0.103   (0.42)
//   1024 x 4032         2.49                                  0.097   (0.73)
//   65,536 x 256        0.239                                 0.127   (0.86)
//   65,536 x 4032       2.50                                  0.75    (11.8)
//   65,536 x 8192       38.0                                  1.40    (33.3)
//
// the last being 8.6 GB of rows, written at 6.1 TB/s.
#include "api_internal.h"
#include "linear_rows.h"
#include "rgroup.cuh"

namespace mwj {
namespace {

constexpr int LT = 256;                      // threads per CTA
constexpr uint32_t LQ = 2;                   // S tuples per thread
constexpr uint32_t LCHUNK = LT * LQ;         // S tuples of a chunk
constexpr unsigned long long kBigRows = 128;
constexpr uint32_t kPiece = 256;             // rows of a piece of a tuple set aside
constexpr uint32_t kSpan = 1024;             // rows between two divisions by a long list's length

struct Lists {
    uint32_t nr, r0, nt, t0;   // list lengths and starts; no rows when either is empty
};

__device__ __forceinline__ Lists lists_of(const LinRowsArgs &g, int32_t b, int32_t c) {
    Lists l{0u, 0u, 0u, 0u};
    const int er = rg_find(g.r, g.r.meta, (uint32_t)b), et = rg_find(g.t, g.t.meta, (uint32_t)c);
    if (er >= 0 && et >= 0) {
        l.nr = __ldg(g.r.deg + er);
        l.r0 = __ldg(g.r.end + er) - l.nr;
        l.nt = __ldg(g.t.deg + et);
        l.t0 = __ldg(g.t.end + et) - l.nt;
    }
    return l;
}

__device__ __forceinline__ void put_row(const LinRowsArgs &g, unsigned long long p, int32_t a, int32_t b, int32_t c,
                                        int32_t d) {
    if (p < (unsigned long long)g.capacity) g.rows[p] = make_int4(a, b, c, d);
}

// Sets aside the warp's tuples that make many rows (k > kBigRows; the lane's
// is S tuple i): each gets its place p behind the chunk's cursor, and those with
// room for a row below the capacity an entry and their pieces.  *big_n counts both
// (entries in the upper half, pieces in the lower one) in one atomic, so that the
// entries' first pieces ascend.  Every lane of the warp calls this.
__device__ __forceinline__ void set_aside(const LinRowsArgs &g, unsigned long long k, uint32_t i,
                                          unsigned long long *cursor, const BigTuples &big) {
    const uint32_t lane = threadIdx.x & 31;
    const bool many = k > kBigRows;
    unsigned long long incl = many ? k : 0ull;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane >= o) incl += y;
    }
    unsigned long long p = 0;
    if (lane == 31) p = atomicAdd(cursor, incl);
    p = __shfl_sync(0xffffffffu, p, 31) + incl - k;
    const unsigned long long cap = (unsigned long long)g.capacity;
    const uint32_t pieces = many && p < cap ? (uint32_t)((min(k, cap - p) + kPiece - 1) / kPiece) : 0u;
    uint32_t upto = pieces;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, upto, o);
        if ((int)lane >= o) upto += y;
    }
    const unsigned kept = __ballot_sync(0xffffffffu, pieces != 0u);
    if (!kept) return;
    unsigned long long at = 0;
    if (lane == 31) at = atomicAdd(big.n, ((unsigned long long)__popc(kept) << 32) | upto);
    at = __shfl_sync(0xffffffffu, at, 31);
    if (!pieces) return;
    const uint32_t e = (uint32_t)(at >> 32) + __popc(kept & ((1u << lane) - 1u));
    big.i[e] = i;
    big.p[e] = p;
    big.s[e] = (uint32_t)at + upto - pieces;
}

__global__ void __launch_bounds__(LT) k_lrows_write(LinRowsArgs g, unsigned long long *__restrict__ n_rows,
                                                    BigTuples big) {
    after_previous();
    __shared__ unsigned long long cursor;
    __shared__ unsigned long long red[32];
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t i0 = blockIdx.x * LCHUNK + threadIdx.x;
    int32_t b[LQ], c[LQ];
    Lists l[LQ];
#pragma unroll
    for (uint32_t q = 0; q < LQ; ++q) {
        const uint32_t i = i0 + q * LT;
        b[q] = i < g.n ? __ldg(g.sb + i) : 0;
        c[q] = i < g.n ? __ldg(g.sc + i) : 0;
    }
#pragma unroll
    for (uint32_t q = 0; q < LQ; ++q) l[q] = i0 + q * LT < g.n ? lists_of(g, b[q], c[q]) : Lists{0u, 0u, 0u, 0u};
    unsigned long long all = 0;
#pragma unroll
    for (uint32_t q = 0; q < LQ; ++q) all += (unsigned long long)l[q].nr * l[q].nt;
    all = block_sum_u64(all, red);
    if (threadIdx.x == 0 && all) cursor = atomicAdd(n_rows, all);
    __syncthreads();
#pragma unroll
    for (uint32_t q = 0; q < LQ; ++q) {
        // the warp's rows: the small tuples' first, in lane order, then the big ones'
        const unsigned long long k = (unsigned long long)l[q].nr * l[q].nt;
        const uint32_t small = k <= kBigRows ? (uint32_t)k : 0u;
        uint32_t incl = small;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if ((int)lane >= o) incl += y;
        }
        const uint32_t W = __shfl_sync(0xffffffffu, incl, 31), excl = incl - small;
        unsigned long long p0 = 0;
        if (lane == 0 && W) p0 = atomicAdd(&cursor, (unsigned long long)W);
        p0 = __shfl_sync(0xffffffffu, p0, 0);
        if (__any_sync(0xffffffffu, k > kBigRows)) set_aside(g, k, i0 + q * LT, &cursor, big);
        for (uint32_t w0 = 0; w0 < W && p0 + w0 < (unsigned long long)g.capacity; w0 += 32) {
            const uint32_t w = w0 + lane;
            int lo = 0, hi = 31;   // the tuple of row w: the first whose inclusive count exceeds it
            const uint32_t wq = w < W ? w : 0u;
#pragma unroll
            for (int step = 0; step < 5; ++step) {
                const int mid = (lo + hi) >> 1;
                const uint32_t v = __shfl_sync(0xffffffffu, incl, mid);
                if (v > wq) hi = mid; else lo = mid + 1;
            }
            const int32_t ob = __shfl_sync(0xffffffffu, b[q], lo), oc = __shfl_sync(0xffffffffu, c[q], lo);
            const uint32_t nt = __shfl_sync(0xffffffffu, l[q].nt, lo), r0 = __shfl_sync(0xffffffffu, l[q].r0, lo);
            const uint32_t t0 = __shfl_sync(0xffffffffu, l[q].t0, lo), ox = __shfl_sync(0xffffffffu, excl, lo);
            if (w < W) {
                const uint32_t r = w - ox, ia = r / nt, id = r - ia * nt;
                put_row(g, p0 + w, __ldg(g.r.alist + r0 + ia), ob, oc, __ldg(g.t.alist + t0 + id));
            }
        }
    }
}

// The rows of the tuples set aside: warp w of W takes a consecutive W-th of the
// pieces, so that every warp writes as much whether there are a few tuples of 10^7
// rows or 10^5 of 5000.  32 entries are looked up at once, one per lane, and
// written one after the other by the whole warp.
__global__ void __launch_bounds__(LT) k_lrows_big(LinRowsArgs g, BigTuples big) {
    after_previous();
    const unsigned long long both = *big.n, cap = (unsigned long long)g.capacity;
    const uint32_t n = (uint32_t)(both >> 32), pieces = (uint32_t)both;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t w = (blockIdx.x * LT + threadIdx.x) >> 5, W = (gridDim.x * LT) >> 5;
    const uint32_t lo = (uint32_t)((uint64_t)pieces * w / W), hi = (uint32_t)((uint64_t)pieces * (w + 1) / W);
    if (lo >= hi) return;
    uint32_t first = 0, end = n;   // the last entry that starts at or before piece lo
    while (end - first > 1) {
        const uint32_t mid = first + (end - first) / 2;
        if (big.s[mid] <= lo) first = mid; else end = mid;
    }
    for (uint32_t e0 = first; e0 < n; e0 += 32) {
        const uint32_t e = e0 + lane;
        const uint32_t s = e < n ? big.s[e] : 0xFFFFFFFFu;
        int32_t b = 0, c = 0;
        Lists l{0u, 0u, 0u, 0u};
        unsigned long long p = 0;
        if (s < hi) {
            const uint32_t i = big.i[e];
            p = big.p[e];
            b = __ldg(g.sb + i);
            c = __ldg(g.sc + i);
            l = lists_of(g, b, c);
        }
        const uint32_t mine = __popc(__ballot_sync(0xffffffffu, s < hi));   // (a prefix of the lanes)
        for (uint32_t j = 0; j < mine; ++j) {
            const uint32_t sj = __shfl_sync(0xffffffffu, s, j);
            const int32_t bj = __shfl_sync(0xffffffffu, b, j), cj = __shfl_sync(0xffffffffu, c, j);
            const uint32_t nr = __shfl_sync(0xffffffffu, l.nr, j), r0 = __shfl_sync(0xffffffffu, l.r0, j);
            const uint32_t nt = __shfl_sync(0xffffffffu, l.nt, j), t0 = __shfl_sync(0xffffffffu, l.t0, j);
            const unsigned long long pj = __shfl_sync(0xffffffffu, p, j);
            const unsigned long long k = min((unsigned long long)nr * nt, cap - pj);
            const unsigned long long q0 = lo > sj ? (unsigned long long)(lo - sj) * kPiece : 0ull;
            const unsigned long long q1 = min(k, (unsigned long long)(hi - sj) * kPiece);
            for (unsigned long long base = q0; base < q1; base += kSpan) {
                const uint32_t m = (uint32_t)min(q1 - base, (unsigned long long)kSpan);
                const uint32_t ia0 = (uint32_t)(base < 0xFFFFFFFFull ? (uint32_t)base / nt : base / nt);
                const uint32_t id0 = (uint32_t)(base - (unsigned long long)ia0 * nt);
#pragma unroll 4
                for (uint32_t off = lane; off < m; off += 32) {
                    const uint32_t t = id0 + off, q = t / nt;   // (id0 < nt < 2^31)
                    g.rows[pj + base + off] =
                        make_int4(__ldg(g.r.alist + r0 + ia0 + q), bj, cj, __ldg(g.t.alist + t0 + (t - q * nt)));
                }
            }
        }
        if (mine < 32) break;
    }
}

// total = n_rows; more rows than the capacity is an error.
__global__ void k_lrows_check(const unsigned long long *n_rows, unsigned long long capacity, unsigned long long *total,
                              DevStatus *st) {
    after_previous();
    *total = *n_rows;
    if (*n_rows > capacity) set_status(st, MWJ_ERR_CAPACITY, (long long)*n_rows);
}

uint32_t lrows_chunks(int64_t nS) { return (uint32_t)((nS + LCHUNK - 1) / LCHUNK); }

}  // namespace

void lin_rows_layout(Arena &A, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, int num_sms, LinRowsLayout &L) {
    auto group = [&](const mwj_rel &r, uint32_t **meta) {
        const size_t reserve = single_table_slots(r.n);
        RGroup g{};
        *meta = A.take<uint32_t>(kMetaWords);
        g.meta = *meta;
        g.keys = A.take<uint32_t>(reserve + 2);
        g.deg = A.take<uint32_t>(reserve + 2);
        g.end = A.take<uint32_t>(reserve + 2);
        g.alist = A.take<int32_t>(r.n + 4);
        return g;
    };
    L.r = group(R, &L.rmeta);
    L.t = group(T, &L.tmeta);
    L.hll = A.take<unsigned int>(hll_scratch_registers(num_sms));
    L.bump = A.take<unsigned int>(4);
    L.big.n = (unsigned long long *)(L.bump + 2);
    L.big.i = A.take<uint32_t>(S.n + 1);
    L.big.p = A.take<unsigned long long>(S.n + 1);
    L.big.s = A.take<uint32_t>(S.n + 1);
}

cudaError_t lin_rows_run(LinRowsLayout &L, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, const Seeds &sd,
                         int4 *rows, long long capacity, long long *n_rows, unsigned long long *total,
                         DevStatus *status, int num_sms, cudaStream_t st) {
    cudaError_t e;
    L.r.seed = sd.slot;
    L.t.seed = sd.slot2;
    if ((e = cudaMemsetAsync(n_rows, 0, sizeof(*n_rows), st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(L.big.n, 0, sizeof(*L.big.n), st)) != cudaSuccess) return e;
    if ((e = rgroup_build(R.x, R.y, R.n, L.r, L.hll, single_table_slots(R.n), L.bump, 0, status, num_sms, st)) !=
        cudaSuccess)
        return e;
    if ((e = rgroup_build(T.y, T.x, T.n, L.t, L.hll, single_table_slots(T.n), L.bump + 1, 0, status, num_sms, st)) !=
        cudaSuccess)
        return e;
    LinRowsArgs g{};
    g.sb = S.x;
    g.sc = S.y;
    g.n = (uint32_t)S.n;
    g.r = L.r;
    g.t = L.t;
    g.rows = rows;
    g.capacity = capacity;
    g.st = status;
    const uint32_t chunks = lrows_chunks(S.n);
    if (chunks) {
        {
            ProfScope ps_("lin_rows", st);
            e = launch_after(k_lrows_write, chunks, LT, st, g, (unsigned long long *)n_rows, L.big);
            if (e != cudaSuccess) return e;
        }
        ProfScope ps_("lin_rows_big", st);
        if ((e = launch_after(k_lrows_big, num_sms * 4, LT, st, g, L.big)) != cudaSuccess) return e;
    }
    ProfScope ps_("rows_check", st);
    return launch_after(k_lrows_check, 1, 1, st, (unsigned long long *)n_rows, (unsigned long long)capacity, total,
                        status);
}

}  // namespace mwj
