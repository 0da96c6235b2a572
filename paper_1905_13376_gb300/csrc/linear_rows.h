// linear_rows.h -- row output of the linear join with one bucket on each side.
#pragma once

#include "cyclic.h"
#include "internal.h"

namespace mwj {

struct LinRowsArgs {
    const int32_t *sb, *sc;   // S
    uint32_t n;
    RGroup r, t;              // b -> [a], c -> [d]
    int4 *rows;
    long long capacity;
    DevStatus *st;
};

// S tuples that make many rows: entry e is S tuple i[e], its rows go to p[e] and
// its first piece is number s[e].
struct BigTuples {
    unsigned long long *n;   // entries << 32 | pieces
    uint32_t *i, *s;
    unsigned long long *p;
};

struct LinRowsLayout {
    RGroup r, t;
    uint32_t *rmeta, *tmeta;
    unsigned int *hll, *bump;
    BigTuples big;
};
// Relations whose lists are numbered in 31 bits (a relation's entries, at most four
// times its tuples, and one for key -1); larger ones run the partitioned plan.
inline bool lin_rows_takes(const mwj_rel &R, const mwj_rel &T) { return R.n < 1ll << 29 && T.n < 1ll << 29; }
void lin_rows_layout(Arena &A, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, int num_sms, LinRowsLayout &L);
// rows (a, b, c, d) into rows[0, min(n_rows, capacity)); *total = n_rows; more rows than the capacity is an error.
cudaError_t lin_rows_run(LinRowsLayout &L, const mwj_rel &R, const mwj_rel &S, const mwj_rel &T, const Seeds &sd,
                         int4 *rows, long long capacity, long long *n_rows, unsigned long long *total,
                         DevStatus *status, int num_sms, cudaStream_t st);

}  // namespace mwj
