// Internal interfaces of the tuple-set operators (bind, filter, sort, join,
// union, project) shared by the translation units.
#pragma once

#include "tid_internal.cuh"

namespace tid {

constexpr int MAX_PREDS = 4;  // predicates fused into one compaction pass

struct Pred {  // a FILTER predicate on column `col` of the set being produced: a value passes
               // when it is bound (not 0) and (lo <= value <= lo + span) != neg
    int col;
    int neg;
    int32_t lo;
    uint32_t span;
};

// A set of terms as a bitmap over [lo, lo + w) in sort order (int32 ^ 0x80000000)
struct Members {
    const uint32_t *bits;
    uint32_t lo, w;
};
constexpr int MAX_MEMBERS = 2;
struct BindMember {  // a bound row is kept when its column `col` is a member
    Members m;
    int col;
};

struct OutCols {
    int32_t *col[TID_MAX_COLS];
};

// Rows of k int32 columns packed into one unsigned key: field c holds
// order_key(col_c) - min[c] (order_key flips the sign bit, so unsigned order is
// int32 order) in bits [shift[c], shift[c] + width); column 0 is the most
// significant field, so key order is row order.
struct PackSpec {
    uint32_t min[TID_MAX_COLS];
    uint32_t shift[TID_MAX_COLS];
    unsigned long long mask[TID_MAX_COLS];
};

// The same for the rows of a union: where bit c of `zero` is set, column c's field
// 0 stands for 0 (unbound, a branch without the variable) and its other values,
// all above 0, start at min[c] + 1.
struct MergePack {
    PackSpec ps;
    unsigned zero;
};

// Column value bounds in sort order (int32 ^ 0x80000000); any valid bounds
// serve the packed sort, exact ones make its keys narrowest.
struct Bounds {
    uint32_t lo[TID_MAX_COLS], hi[TID_MAX_COLS];
};

// Where a kernel that writes a set's rows leaves their columns' bounds (sort order;
// at most BOUND_COLS columns).  Every CTA merges its rows' into `acc` (word c the
// least, word 8 + c the largest value of column c; least values start at ~0, largest
// at 0); the last one of the grid moves them to the set's slot and makes acc neutral
// again, so an extraction needs no launch to preset its bounds and no copy to read
// them: they are on the host with its row count, beside it, and no other extraction
// of the context, queued by another thread meanwhile, writes there.
struct BoundsOut {
    uint32_t *acc = nullptr;  // null: not wanted
    unsigned *done = nullptr;
    uint32_t *host = nullptr;
};
int bounds_out(tid_set *set, BoundsOut *b);
// bounds of set's columns [0, k), once the kernel that leaves them is done
void read_bounds(const tid_set *set, int k, uint32_t *lo, uint32_t *hi);

struct VarMember {  // the same by variable
    Members m;
    int8_t var;
};

// exclusive scan of n uint32 (out may alias in); *total_dev receives the sum; sums:
// the sum of every tile of SCAN_TILE items, if the caller has them
constexpr int SCAN_TILE = 4096;
int scan_exclusive_u32(tid_ctx *ctx, const uint32_t *in, uint32_t *out, int64_t n,
                       unsigned long long *total_dev, const uint32_t *sums = nullptr);

// row selections (compact.cu); `out` must have capacity >= n
// bind, with the bounds of the kept rows
int compact_bind(tid_ctx *ctx, const tid_store *st, const tid_pattern &pat, const int32_t *idx, int64_t n,
                 const Pred *preds, int n_preds, const BindMember *mem, int n_mem, tid_set *out, const BoundsOut &mm);
// the terms of col[0, n) in [lo, hi] (sort order, hi - lo < 2^32 - 1) as a bitmap,
// allocated here (m->bits, freed by the caller)
int member_bits(tid_ctx *ctx, const int32_t *col, int64_t n, uint32_t lo, uint32_t hi, Members *m);
// rows of `in` whose first column is a member, in order
int compact_member(tid_ctx *ctx, const tid_set *in, int64_t n, const Members &m, tid_set *out);
int compact_filter(tid_ctx *ctx, const tid_set *in, int64_t n, const Pred *preds, int n_preds, tid_set *out);
int compact_unique(tid_ctx *ctx, const int32_t *const *cols, int k, const int32_t *perm, int64_t n,
                   tid_set *out);
// flag's row count: 1 if some of the n > 0 sorted rows of `in` repeats, else 0
int find_repeats(tid_ctx *ctx, const tid_set *in, int64_t n, tid_set *flag);
// sorted packed keys (64-bit if wide, else 32-bit) -> distinct rows of k columns
int compact_unique_packed(tid_ctx *ctx, const void *keys, bool wide, int k, int64_t n, const PackSpec &ps,
                          tid_set *out);

// sorting (sort.cu)
// perm receives the stable permutation that orders rows 0..n-1 lexicographically
// by the key columns keys[0..nk-1] (signed int32 order).
int sort_perm(tid_ctx *ctx, const int32_t *const *keys, int nk, int64_t n, int32_t *perm);
// out[c][i] = in[c][perm[i]] for c < k, i < n
int gather_cols(tid_ctx *ctx, const int32_t *const *in, int k, const int32_t *perm, int64_t n,
                int32_t *const *out);
// canonical form (rows sorted in column order; duplicates dropped if dedupe);
// bounds of the input columns if known (else they are computed); the output
// set records the bounds used
// sorted_tail: the rows are already sorted by their last sorted_tail columns
// (lexicographically, in that order), so only the leading columns are sorted
int canonicalize(tid_ctx *ctx, const int32_t *const *cols, int k, const int8_t *vars, int64_t n,
                 bool dedupe, const Bounds *bounds, tid_set **out, int sorted_tail = 0);

// write a known row count into a set (device count and host mirror)
int set_rows_const(tid_set *set, int64_t n);

// row count known on the host (waits for the producer if needed)
int set_rows_host(tid_set *set, int64_t *rows);
int set_rows_host(const tid_set *set, int64_t *rows);

// joins (join.cu); right and full outer joins composed from the left join (ops.cu)
// sorted_out = false (internal use, hash join of inputs in any row order): the
// joined rows in the order written, not canonical (the caller sorts what it keeps)
int join_sets(tid_ctx *ctx, const tid_set *L, const tid_set *R, int algo, tid_set **out, bool sorted_out = true);
int outer_join_sets(tid_ctx *ctx, const tid_set *L, const tid_set *R, int algo, tid_set **out);

// merge (merge.cu): the distinct rows of two sets each sorted in the same nu
// columns (acols / bcols, null = absent column, read as 0) into out (capacity
// >= na + nb), in order; writes the row count; mp (or null): how every row of
// both packs into 64 bits
int merge_unique(tid_ctx *ctx, const int32_t *const *acols, int64_t na, const int32_t *const *bcols, int64_t nb,
                 int nu, const MergePack *mp, tid_set *out);

// rows that one CTA sorts (sort.cu), dropping repeats on the way
constexpr int ONE_CTA_ROWS = 4096;

// the union of at most SMALL_UNION_INPUTS sets of at most SMALL_UNION_ROWS rows in all,
// in one launch (sort.cu): cols[i][c] column c of input i (null: absent), packed by mp
constexpr int SMALL_UNION_ROWS = 1024, SMALL_UNION_INPUTS = 4;
int small_union(tid_ctx *ctx, const int32_t *const (*cols)[TID_MAX_COLS], const int64_t *rows, int inputs, int k,
                const MergePack &mp, tid_set *out);

// set operators (ops.cu)
int filter_set(tid_ctx *ctx, const tid_set *in, const tid_pred *preds, int n_preds, tid_set **out);
int union_sets(tid_ctx *ctx, const tid_set *const *in, int k, tid_set **out);
int project_set(tid_ctx *ctx, const tid_set *in, const int8_t *vars, int n_vars, tid_set **out);

// plans (exec.cu): checks a plan's shape and patterns; evaluates a checked plan,
// taking over matched[i] (an index list, or null to search it) for MATCH nodes
int validate_plan(const tid_plan_node *nodes, int n_nodes);
int exec_plan(tid_ctx *ctx, const tid_store *st, const tid_plan_node *nodes, int n_nodes, tid_set **matched,
              tid_set **out);

}  // namespace tid
