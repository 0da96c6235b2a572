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
//   pass 2  the rows of those, one tuple at a time by the whole GPU
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
#include "api_internal.h"
#include "linear_rows.h"
#include "rgroup.cuh"

namespace mwj {
namespace {

constexpr int LT = 256;                      // threads per CTA
constexpr uint32_t LQ = 2;                   // S tuples per thread
constexpr uint32_t LCHUNK = LT * LQ;         // S tuples of a chunk
constexpr unsigned long long kBigRows = 4096;

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

__global__ void __launch_bounds__(LT) k_lrows_write(LinRowsArgs g, unsigned long long *__restrict__ n_rows,
                                                    uint32_t *__restrict__ big_n, uint32_t *__restrict__ big_i,
                                                    unsigned long long *__restrict__ big_p) {
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
        if (k > kBigRows) {
            const uint32_t at = atomicAdd(big_n, 1u);
            big_i[at] = i0 + q * LT;
            big_p[at] = atomicAdd(&cursor, k);
        }
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

__global__ void __launch_bounds__(LT) k_lrows_big(LinRowsArgs g, const uint32_t *__restrict__ big_n,
                                                  const uint32_t *__restrict__ big_i,
                                                  const unsigned long long *__restrict__ big_p) {
    after_previous();
    const uint32_t n = *big_n;
    const unsigned long long T = (unsigned long long)gridDim.x * LT;
    for (uint32_t e = 0; e < n; ++e) {
        const uint32_t i = big_i[e];
        const unsigned long long p = big_p[e];
        const int32_t b = __ldg(g.sb + i), c = __ldg(g.sc + i);
        const Lists l = lists_of(g, b, c);
        const unsigned long long room = p < (unsigned long long)g.capacity ? (unsigned long long)g.capacity - p : 0ull;
        const unsigned long long k = min((unsigned long long)l.nr * l.nt, room);
        for (unsigned long long r = (unsigned long long)blockIdx.x * LT + threadIdx.x; r < k; r += T) {
            const unsigned long long ia = r / l.nt;
            put_row(g, p + r, __ldg(g.r.alist + l.r0 + ia), b, c, __ldg(g.t.alist + l.t0 + (r - ia * l.nt)));
        }
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
    L.big_i = A.take<uint32_t>(S.n + 1);
    L.big_p = A.take<unsigned long long>(S.n + 1);
}

cudaError_t lin_rows_run(LinRowsLayout &L, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, const Seeds &sd,
                         int4 *rows, long long capacity, long long *n_rows, unsigned long long *total,
                         DevStatus *status, int num_sms, cudaStream_t st) {
    cudaError_t e;
    L.r.seed = sd.slot;
    L.t.seed = sd.slot2;
    uint32_t *big_n = L.bump + 2;
    if ((e = cudaMemsetAsync(n_rows, 0, sizeof(*n_rows), st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(big_n, 0, sizeof(*big_n), st)) != cudaSuccess) return e;
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
            e = launch_after(k_lrows_write, chunks, LT, st, g, (unsigned long long *)n_rows, big_n, L.big_i, L.big_p);
            if (e != cudaSuccess) return e;
        }
        ProfScope ps_("lin_rows_big", st);
        if ((e = launch_after(k_lrows_big, num_sms * 4, LT, st, g, big_n, L.big_i, L.big_p)) != cudaSuccess) return e;
    }
    ProfScope ps_("rows_check", st);
    return launch_after(k_lrows_check, 1, 1, st, (unsigned long long *)n_rows, (unsigned long long)capacity, total,
                        status);
}

}  // namespace mwj
