// Row selection over tuple sets, and a device-wide exclusive scan.
//
// Serves the operators that keep a subset of rows in their original order and
// write k output columns:
//   * bind     -- from triple indices, the terms at a pattern's variable slots,
//                 dropping rows whose repeated variable disagrees; the FILTER
//                 predicates of the subquery are applied in the same pass
//                 (Section 4.3: the filter is applied while the matched triples
//                 are extracted into the subquery's vector);
//   * filter   -- a predicate on one column of a set;
//   * member   -- rows whose key is in another set's key column (the join with
//                 a set of keys only);
//   * unique   -- after a sort, a row is kept when it differs from its
//                 predecessor in sorted order (DISTINCT, Section 4.3), on
//                 column rows or on packed row keys;
//   * repeats  -- whether a sorted set repeats a row at all;
//   * keyed    -- the rows of the entailment's keyed store pass (Section 5), which
//                 entail.cu marks itself: expand only.
// Short inputs: k_compact, one launch (ranks from ballots, tile offsets from
// the decoupled look-back of lookback.cuh).  Long inputs: k_sel_mark, which
// tests every row and writes one keep bit per row, and k_sel_expand, which
// reads the kept rows' values and writes them in order; no CTA of either waits
// for another.

#include <stddef.h>

#include <algorithm>
#include <type_traits>

#include "lookback.cuh"
#include "ops.cuh"
#include "keys.cuh"
#include "select.cuh"

namespace tid {

namespace {

constexpr int CP_THREADS = 256;
constexpr int CP_WARPS = CP_THREADS / 32;
constexpr int CP_ITEMS = 8;
constexpr int CP_TILE = CP_THREADS * CP_ITEMS;

__device__ __forceinline__ bool pred_ok(const Pred &p, int32_t x) {  // an unbound value never passes
    return x != 0 && (((uint32_t)x - (uint32_t)p.lo <= p.span) != (p.neg != 0));
}

// Membership of a term in a set of terms held as a bit per term of [lo, lo + w)
// (sort order); 0 (unbound) is never a member.
__device__ __forceinline__ bool is_member(const Members &m, int32_t x) {
    const uint32_t d = ((uint32_t)x ^ 0x80000000u) - m.lo;
    return d < m.w && ((__ldg(m.bits + (d >> 5)) >> (d & 31)) & 1u);
}

// ---- row sources -----------------------------------------------------------

// A row source says, for a row r < n, whether it is kept (keep: reads only
// what the test needs) and gives its K output values (values<K>: v[0..K)); at
// most MAX_K columns.  keep_step tests a lane's 32 rows of a full step (rows
// r0 + 128 g + (0..3), r0 a multiple of 4): bit e of m[g] is row r0 + 128 g + e.
// It loads 16 bytes at a time and issues a group of loads before using any.
__device__ __forceinline__ int4 ld4(const int32_t *p) { return __ldg(reinterpret_cast<const int4 *>(p)); }

template <class F>
__device__ __forceinline__ unsigned test4(int4 x, F f) {
    return (unsigned)f(x.x) | ((unsigned)f(x.y) << 1) | ((unsigned)f(x.z) << 2) | ((unsigned)f(x.w) << 3);
}

struct BindRow {  // triple index -> variable values
    static constexpr int MAX_K = 3;
    const int32_t *S, *P, *O;
    const int32_t *idx;
    int k;
    int need;                   // slots (bit 0 s, 1 p, 2 o) that carry a variable
    int test;                   // slots that a test reads
    int8_t src[TID_MAX_COLS];   // slot (0,1,2) giving output column c
    int8_t eq_a[3], eq_b[3];    // pairs of slots that must be equal
    int n_eq;
    Pred preds[MAX_PREDS];      // col: a slot
    int n_preds;
    int32_t *stash;             // row r's value of the one tested slot, written by keep_step (or null)
    Members mem[MAX_MEMBERS];   // terms a slot's value must be among
    int8_t mem_slot[MAX_MEMBERS];
    int n_mem;
    __device__ __forceinline__ bool ok(int32_t t0, int32_t t1, int32_t t2) const {
        auto at = [&](int slot) { return slot == 0 ? t0 : (slot == 1 ? t1 : t2); };
        bool ok = true;
#pragma unroll
        for (int e = 0; e < 3; ++e)
            if (e < n_eq) ok = ok && at(eq_a[e]) == at(eq_b[e]);
#pragma unroll
        for (int q = 0; q < MAX_PREDS; ++q)
            if (q < n_preds) ok = ok && pred_ok(preds[q], at(preds[q].col));
#pragma unroll
        for (int q = 0; q < MAX_MEMBERS; ++q)
            if (q < n_mem) ok = ok && is_member(mem[q], at(mem_slot[q]));
        return ok;
    }
    __device__ __forceinline__ bool keep(int64_t r) const {
        const int64_t t = idx[r];
        if (stash) stash[r] = (test & 1) ? S[t] : ((test & 2) ? P[t] : O[t]);
        return keep_at(t);
    }
    __device__ __forceinline__ bool keep_at(int64_t t) const {
        return ok((test & 1) ? S[t] : 0, (test & 2) ? P[t] : 0, (test & 4) ? O[t] : 0);
    }
    __device__ __forceinline__ void keep_step(uint32_t r0, unsigned *m) const {
#pragma unroll 1
        for (int h = 0; h < 8; h += 4) {  // 16 rows at a time: their indices, then their gathers, in flight
            int4 t[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) t[g] = ld4(idx + r0 + (h + g) * 128);
            unsigned k4[4];
            if (n_eq == 0 && (test & (test - 1)) == 0) {  // one slot is tested
                const int32_t *col = test == 1 ? S : (test == 2 ? P : O);
                int4 x[4];
#pragma unroll
                for (int g = 0; g < 4; ++g) x[g] = make_int4(col[t[g].x], col[t[g].y], col[t[g].z], col[t[g].w]);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    k4[g] = test4(x[g], [&](int32_t v) { return ok(v, v, v); });
                    if (stash) *reinterpret_cast<int4 *>(stash + r0 + (h + g) * 128) = x[g];
                }
            } else {
#pragma unroll
                for (int g = 0; g < 4; ++g) k4[g] = test4(t[g], [&](int32_t i) { return keep_at(i); });
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                if (h == 0) m[g] = k4[g];
                else m[g + 4] = k4[g];
            }
        }
    }
    template <int K>
    __device__ __forceinline__ void values(int64_t r, int32_t *v) const {
        const int64_t t = idx[r];
        // only the variable slots are read: a bound slot holds the key itself.
        // The tested slot of a kept row comes from the stash: at one kept triple
        // in sixteen its column's gather would read nearly every line again.
        const int skip = stash ? test : 0;
        const int32_t x = skip ? stash[r] : 0;
        const int32_t t0 = (skip & 1) ? x : ((need & 1) ? S[t] : 0), t1 = (skip & 2) ? x : ((need & 2) ? P[t] : 0),
                      t2 = (skip & 4) ? x : ((need & 4) ? O[t] : 0);
#pragma unroll
        for (int c = 0; c < K; ++c)
            if (c < k) v[c] = src[c] == 0 ? t0 : (src[c] == 1 ? t1 : t2);
    }
};

struct FilterRow {
    static constexpr int MAX_K = TID_MAX_COLS;
    const int32_t *col[TID_MAX_COLS];
    int k;
    Pred preds[MAX_PREDS];
    int n_preds;
    __device__ __forceinline__ const int32_t *column(int c) const {  // constant indices: no local copy of col[]
        const int32_t *p = col[0];
#pragma unroll
        for (int i = 1; i < TID_MAX_COLS; ++i)
            if (c == i) p = col[i];
        return p;
    }
    __device__ __forceinline__ bool keep(int64_t r) const {  // the predicates' columns only
        bool ok = true;
#pragma unroll
        for (int q = 0; q < MAX_PREDS; ++q)
            if (q < n_preds) ok = ok && pred_ok(preds[q], column(preds[q].col)[r]);
        return ok;
    }
    __device__ __forceinline__ void keep_step(uint32_t r0, unsigned *m) const {
#pragma unroll
        for (int g = 0; g < 8; ++g) m[g] = 0xFu;
#pragma unroll 1
        for (int q = 0; q < n_preds; ++q) {
            const Pred p = preds[q];
            const int32_t *cp = column(p.col);
            int4 x[8];
#pragma unroll
            for (int g = 0; g < 8; ++g) x[g] = ld4(cp + r0 + g * 128);
#pragma unroll
            for (int g = 0; g < 8; ++g) m[g] &= test4(x[g], [&](int32_t v) { return pred_ok(p, v); });
        }
    }
    template <int K>
    __device__ __forceinline__ void values(int64_t r, int32_t *v) const {
#pragma unroll
        for (int c = 0; c < K; ++c)
            if (c < k) v[c] = col[c][r];
    }
};

struct MemberRow {  // rows of a set whose first column is among the members
    static constexpr int MAX_K = TID_MAX_COLS;
    const int32_t *col[TID_MAX_COLS];
    int k;
    Members m;
    __device__ __forceinline__ bool keep(int64_t r) const { return is_member(m, col[0][r]); }
    __device__ __forceinline__ void keep_step(uint32_t r0, unsigned *k4) const {
        int4 x[8];
#pragma unroll
        for (int g = 0; g < 8; ++g) x[g] = ld4(col[0] + r0 + g * 128);
#pragma unroll
        for (int g = 0; g < 8; ++g) k4[g] = test4(x[g], [&](int32_t v) { return is_member(m, v); });
    }
    template <int K>
    __device__ __forceinline__ void values(int64_t r, int32_t *v) const {
#pragma unroll
        for (int c = 0; c < K; ++c)
            if (c < k) v[c] = col[c][r];
    }
};

struct UniqueRow {  // rows in perm order; keep the first of each run of equal rows
    static constexpr int MAX_K = TID_MAX_COLS;
    const int32_t *col[TID_MAX_COLS];
    const int32_t *perm;  // may be null (rows already in order)
    int k;
    __device__ __forceinline__ bool keep(int64_t r) const {
        if (r == 0) return true;
        const int64_t a = perm ? perm[r] : r;
        const int64_t b = perm ? perm[r - 1] : r - 1;
        bool same = true;
#pragma unroll
        for (int c = 0; c < TID_MAX_COLS; ++c)
            if (c < k) same = same && col[c][b] == col[c][a];
        return !same;
    }
    __device__ __forceinline__ void keep_step(uint32_t r0, unsigned *m) const {
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            const uint32_t r = r0 + g * 128;
            m[g] = test4(make_int4(0, 1, 2, 3), [&](int32_t e) { return keep(r + e); });
        }
    }
    template <int K>
    __device__ __forceinline__ void values(int64_t r, int32_t *v) const {
        const int64_t a = perm ? perm[r] : r;
#pragma unroll
        for (int c = 0; c < K; ++c)
            if (c < k) v[c] = col[c][a];
    }
};

// Whether some row of a sorted set equals the one before it (1 or 0 as the "row
// count" of a set): a reordering of all columns of a set whose rows are distinct
// needs no DISTINCT.  A warp tests steps of 1024 rows, columns from the last to the
// first, and leaves a step when no row of it can be a repeat any more: neighbours of a
// sorted set differ in the last column, so mostly that one is read.  Bound: HBM (24M
// rows of two columns: 23 us on GB300).
struct SetCols {
    const int32_t *col[TID_MAX_COLS];
};
constexpr int RP_THREADS = 256;
__global__ void __launch_bounds__(RP_THREADS) k_repeats(SetCols in, int k, uint32_t n, unsigned steps, unsigned *acc,
                                                        unsigned *done, int64_t *__restrict__ d_rows,
                                                        int64_t *__restrict__ h_rows) {
    const unsigned lane = threadIdx.x & 31;
    const unsigned warps = gridDim.x * (RP_THREADS / 32);
    unsigned found = 0;
    for (unsigned step = blockIdx.x * (RP_THREADS / 32) + (threadIdx.x >> 5); step < steps; step += warps) {
        const uint32_t r0 = step * SEL_STEP + lane * 4;  // < 2^32: n < 2^31
        unsigned same[8], any = 1;
#pragma unroll
        for (int g = 0; g < 8; ++g) {  // rows past n, and the first row, equal no predecessor
            const uint32_t r = r0 + g * 128;
            same[g] = r + 4 <= n ? 0xFu : (r < n ? (1u << (n - r)) - 1u : 0u);
            if (r == 0) same[g] &= ~1u;
        }
        const bool whole = (step + 1) * SEL_STEP <= n;
#pragma unroll
        for (int c = TID_MAX_COLS - 1; c >= 0; --c) {
            if (c >= k || !any) continue;
            const int32_t *p = in.col[c];
            int4 x[8];
            int32_t before[8];
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const uint32_t r = r0 + g * 128;
                if (whole) {
                    x[g] = ld4(p + r);
                } else {
                    x[g] = make_int4(r < n ? p[r] : 0, r + 1 < n ? p[r + 1] : 0, r + 2 < n ? p[r + 2] : 0,
                                     r + 3 < n ? p[r + 3] : 0);
                }
                before[g] = lane == 0 && r > 0 && r < n ? p[r - 1] : 0;
            }
            unsigned left = 0;
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const int32_t up = __shfl_up_sync(0xffffffffu, x[g].w, 1);
                const int32_t b = lane == 0 ? before[g] : up;
                same[g] &= (unsigned)(x[g].x == b) | ((unsigned)(x[g].y == x[g].x) << 1) |
                           ((unsigned)(x[g].z == x[g].y) << 2) | ((unsigned)(x[g].w == x[g].z) << 3);
                left |= same[g];
            }
            any = __any_sync(0xffffffffu, left);
        }
        found |= any;
    }
    if (lane == 0 && found) atomicOr(acc, 1u);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(done, 1u) == gridDim.x - 1) {
            __threadfence();
            *d_rows = *h_rows = (int64_t)atomicExch(acc, 0u);
            *done = 0;
        }
    }
}

struct KeyedRow {  // row r of a keyed pass (entail.cu marks its rows), some slots as they are,
                   // the key slot's term also through a map by key number
    static constexpr int MAX_K = 3;
    const int32_t *S, *P, *O;
    int key_slot;
    KeySet keys;
    const int32_t *map;
    int k;
    int8_t src[3];  // slot giving output column c; 3: map[key number]
    template <int K>
    __device__ __forceinline__ void values(int64_t r, int32_t *v) const {
#pragma unroll
        for (int c = 0; c < K; ++c) {
            if (c >= k) break;
            const int s = src[c] == 3 ? key_slot : src[c];
            const int32_t x = (s == 0 ? S : (s == 1 ? P : O))[r];
            v[c] = src[c] == 3 ? map[key_number(keys, x)] : x;
        }
    }
};

template <typename W>
struct PackedUniqueRow {  // sorted packed keys; keep the first of each run of equal keys
    static constexpr int MAX_K = TID_MAX_COLS;
    const W *keys;
    PackSpec ps;
    int k;
    __device__ __forceinline__ bool keep(int64_t r) const { return r == 0 || keys[r - 1] != keys[r]; }
    __device__ __forceinline__ void keep_step(uint32_t r0, unsigned *m) const {
        W x[8][4], before[8];
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            const uint32_t r = r0 + g * 128;
            const int4 a = ld4(reinterpret_cast<const int32_t *>(keys + r));
            if constexpr (sizeof(W) == 4) {
                x[g][0] = a.x, x[g][1] = a.y, x[g][2] = a.z, x[g][3] = a.w;
            } else {
                const int4 b = ld4(reinterpret_cast<const int32_t *>(keys + r + 2));
                x[g][0] = (W)(uint32_t)a.x | ((W)(uint32_t)a.y << 32);
                x[g][1] = (W)(uint32_t)a.z | ((W)(uint32_t)a.w << 32);
                x[g][2] = (W)(uint32_t)b.x | ((W)(uint32_t)b.y << 32);
                x[g][3] = (W)(uint32_t)b.z | ((W)(uint32_t)b.w << 32);
            }
            before[g] = keys[r > 0 ? r - 1 : 0];
        }
#pragma unroll
        for (int g = 0; g < 8; ++g)
            m[g] = (unsigned)(x[g][0] != before[g] || r0 + g * 128 == 0) | ((unsigned)(x[g][1] != x[g][0]) << 1) |
                   ((unsigned)(x[g][2] != x[g][1]) << 2) | ((unsigned)(x[g][3] != x[g][2]) << 3);
    }
    template <int K>
    __device__ __forceinline__ void values(int64_t r, int32_t *v) const {
        const W key = keys[r];
#pragma unroll
        for (int c = 0; c < K; ++c) {
            if (c < k) {
                const uint32_t f = ps.mask[c] ? (uint32_t)((key >> ps.shift[c]) & ps.mask[c]) : 0u;
                v[c] = (int32_t)((f + ps.min[c]) ^ 0x80000000u);
            }
        }
    }
};

// bounds (sort order) of the values a thread wrote, merged per warp into mm.acc;
// the last CTA moves the result to the set's slot (all threads of every CTA call this)
template <int K>
__device__ __forceinline__ void merge_bounds(const BoundsOut &mm, int k_out, const uint32_t *lo, const uint32_t *hi) {
    const unsigned lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < K; ++c) {
        if (c < k_out) {
            const uint32_t a = __reduce_min_sync(0xffffffffu, lo[c]), b = __reduce_max_sync(0xffffffffu, hi[c]);
            // the bounds only tighten, so a warp that cannot improve the
            // current one (read from L2; a stale read only costs an atomic)
            // skips its atomic: many warps otherwise queue on one address
            if (lane == 0 && a <= b) {
                if (a < __ldcg(mm.acc + c)) atomicMin(mm.acc + c, a);
                if (b > __ldcg(mm.acc + TID_MAX_COLS + c)) atomicMax(mm.acc + TID_MAX_COLS + c, b);
            }
        }
    }
    __shared__ unsigned s_end;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_end = atomicAdd(mm.done, 1u) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!s_end) return;
    if (threadIdx.x < 2 * TID_MAX_COLS) {
        const unsigned c = threadIdx.x % TID_MAX_COLS;
        if (c < BOUND_COLS) mm.host[threadIdx.x / TID_MAX_COLS * BOUND_COLS + c] = __ldcg(mm.acc + threadIdx.x);
        mm.acc[threadIdx.x] = threadIdx.x < TID_MAX_COLS ? 0xFFFFFFFFu : 0u;
    }
    if (threadIdx.x == 0) *mm.done = 0;
}

// ---- single-pass compaction (small inputs) ----------------------------------------

// The tile's kept rows are staged in shared memory at their place in the tile
// (the block's own scan gives it) while warp 0 looks back for the tile's
// offset, so the value reads overlap that wait; the tile is then written with
// coalesced stores.  Dynamic shared memory: k_out x CP_TILE int32.
template <class Row>
__global__ void __launch_bounds__(CP_THREADS)
k_compact(Row row, int64_t n, int k_out, OutCols out, int64_t cap, int64_t *__restrict__ d_rows,
          int64_t *__restrict__ h_rows, Lookback lb, BoundsOut mm) {
    extern __shared__ int32_t s_vals[];  // column c of staged row i at s_vals[c * CP_TILE + i]
    __shared__ unsigned s_tile, s_total;
    __shared__ unsigned s_off[CP_ITEMS * CP_WARPS];
    __shared__ long long s_prefix;
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = lb_ticket(lb);
    __syncthreads();
    const unsigned tile = s_tile;
    if (tile >= lb.num_tiles) return;
    const int64_t base = (int64_t)tile * CP_TILE;
    const unsigned lt = (1u << lane) - 1u;

    unsigned keep = 0, wpre[CP_ITEMS];
    bool kp[CP_ITEMS];
#pragma unroll
    for (int j = 0; j < CP_ITEMS; ++j) {  // all tests first: their loads are in flight together
        const int64_t r = base + j * CP_THREADS + threadIdx.x;
        kp[j] = row.keep(r < n ? r : n - 1) && r < n;  // rows past n test row n - 1 and are dropped
    }
#pragma unroll
    for (int j = 0; j < CP_ITEMS; ++j) {
        keep |= (unsigned)kp[j] << j;
        const unsigned b = __ballot_sync(0xffffffffu, kp[j]);
        wpre[j] = __popc(b & lt);
        if (lane == 0) s_off[j * CP_WARPS + warp] = __popc(b);
    }
    __syncthreads();
    if (warp == 0) {  // 64 (item, warp) counts in order; each lane scans two consecutive entries
        const unsigned a0 = s_off[2 * lane], a1 = s_off[2 * lane + 1];
        unsigned x = a0 + a1;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, d);
            if ((int)lane >= d) x += y;
        }
        const unsigned ex = x - a0 - a1;
        s_off[2 * lane] = ex;
        s_off[2 * lane + 1] = ex + a0;
        if (lane == 31) s_total = x;
    }
    __syncthreads();
    const unsigned total = s_total;
    auto stage = [&]() {  // this thread's kept rows to their place in the tile
#pragma unroll
        for (int j = 0; j < CP_ITEMS; ++j) {
            if (!((keep >> j) & 1u)) continue;
            int32_t v[TID_MAX_COLS];
            row.template values<TID_MAX_COLS>(base + j * CP_THREADS + threadIdx.x, v);
            const unsigned at = s_off[j * CP_WARPS + warp] + wpre[j];
#pragma unroll
            for (int c = 0; c < TID_MAX_COLS; ++c)
                if (c < k_out) s_vals[c * CP_TILE + at] = v[c];
        }
    };
    if (warp == 0) {
        const long long excl = lb_exclusive_prefix(lb, tile, total);
        if (lane == 0) {
            s_prefix = excl;
            if (tile == lb.num_tiles - 1 && excl >= 0) {
                *d_rows = excl + total;
                *h_rows = excl + total;
            }
        }
    }
    stage();  // warps 1.. stage while warp 0 waits for the tile's offset
    __syncthreads();
    const long long prefix = s_prefix;
    if (prefix < 0) return;
    uint32_t lo[TID_MAX_COLS], hi[TID_MAX_COLS];
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c) {
        lo[c] = 0xFFFFFFFFu;
        hi[c] = 0u;
    }
    for (unsigned i = threadIdx.x; i < total; i += CP_THREADS) {  // coalesced: row prefix + i
        const long long pos = prefix + i;
#pragma unroll
        for (int c = 0; c < TID_MAX_COLS; ++c) {
            if (c < k_out) {
                const int32_t v = s_vals[c * CP_TILE + i];
                if (pos < cap) out.col[c][pos] = v;
                const uint32_t u = (uint32_t)v ^ 0x80000000u;
                lo[c] = min(lo[c], u);
                hi[c] = max(hi[c], u);
            }
        }
    }
    if (mm.acc) merge_bounds<TID_MAX_COLS>(mm, k_out, lo, hi);  // column bounds of the kept rows
}

// ---- mark and expand (long inputs) -------------------------------------------------
//
// k_sel_mark and k_sel_expand: mark and expand (select.cuh) of rows.  A step that
// keeps many rows is read word by word (lane l the word's row l: coalesced loads
// and stores); of one that keeps few, the positions go to shared memory first and
// only the kept rows are read, all lanes at work.  The test's columns are read
// twice, every other value once; in the one-launch form a tile waits for its
// predecessors' counts longer than its own work takes.
// Bound: memory latency of the expansion's dependent loads (ncu: 57 % of DRAM
// throughput binding 23.6M triples, long-scoreboard stalls).  Measured on GB300
// (kernels, before -> after this form): FILTER of 24M two-column rows, half kept,
// 227 -> 83 us; bind of 23.6M triples of a 200M store with a range FILTER
// 700 -> 400 us (the tested column is gathered once and stashed); before, per
// 2048-row tile: a count and a write launch (filter), one look-back launch (bind).
// A mark phase with 4-byte loads in place of 16-byte ones took 58 us on the
// filter against 32 us; one large range per resident CTA with block scans took
// 97 us to expand against 83 us.

// Below this, the single-pass kernel: its tiles of 2048 rows test eight rows per
// thread one after another, so it pays while the input is a few tiles (binding
// 36K matched triples with a test, and the set's sort: 106 us with one launch, 98 with two).
constexpr int64_t SEL_MIN_ROWS = (int64_t)1 << 13;

template <class Row>
__global__ void __launch_bounds__(SEL_THREADS)
k_sel_mark(Row row, uint32_t n, SelScratch sc, int64_t *__restrict__ d_rows, int64_t *__restrict__ h_rows) {
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned r0 = blockIdx.x * sc.per, r1 = min(r0 + sc.per, sc.steps);
    unsigned kept = 0;
    for (unsigned step = r0 + warp; step < r1; step += SEL_WARPS) {
        const uint32_t base = step * SEL_STEP + lane * 4;  // < 2^32: n < 2^31
        unsigned m[8];
        if ((step + 1) * SEL_STEP <= n) {
            row.keep_step(base, m);
        } else {  // ragged last step
#pragma unroll 1
            for (int g = 0; g < 8; ++g) {
                unsigned k4 = 0;
                for (int e = 0; e < 4; ++e) {
                    const uint32_t r = base + g * 128 + e;
                    if (r < n && row.keep(r)) k4 |= 1u << e;
                }
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q == g) m[q] = k4;
            }
        }
        const uint32_t word = sel_word(m);
        sc.bits[(size_t)step * 32 + sel_word_index()] = word;
        const unsigned c = __reduce_add_sync(0xffffffffu, __popc(word));
        if (lane == 0) sc.cnt[step] = c;
        kept += c;
    }
    sel_finish(sc, kept, d_rows, h_rows);
}

template <class Row, int K, bool BOUNDS>
__global__ void __launch_bounds__(SEL_THREADS, K == 2 ? 5 : (K <= 3 ? 4 : 2))
k_sel_expand(Row row, int k_out, OutCols out, int64_t cap, SelScratch sc, BoundsOut mm) {
    __shared__ uint16_t s_stage[SEL_WARPS][SEL_DENSE];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t lo[K], hi[K];
#pragma unroll
    for (int c = 0; c < K; ++c) {
        lo[c] = 0xFFFFFFFFu;
        hi[c] = 0u;
    }
    auto put = [&](const int32_t *v, unsigned long long pos) {
#pragma unroll
        for (int c = 0; c < K; ++c) {
            if (c < k_out) {
                if (pos < (unsigned long long)cap) out.col[c][pos] = v[c];
                if (BOUNDS) {
                    const uint32_t u = (uint32_t)v[c] ^ 0x80000000u;
                    lo[c] = min(lo[c], u);
                    hi[c] = max(hi[c], u);
                }
            }
        }
    };
    constexpr int UX = K == 1 ? 8 : 4;  // rows per lane read together
    uint16_t *stage = s_stage[warp];
    sel_walk(sc, blockIdx.x, warp, SEL_WARPS, [&](unsigned step, uint32_t word, unsigned xo, unsigned sn, unsigned long long o0) {
        const int64_t base = (int64_t)step * SEL_STEP;
        if (sn >= SEL_DENSE) {
#pragma unroll 1
            for (int w0 = 0; w0 < 32; w0 += UX) {
                int32_t v[UX][K];
                unsigned bw[UX];
#pragma unroll
                for (int u = 0; u < UX; ++u) {
                    bw[u] = __shfl_sync(0xffffffffu, word, w0 + u);
                    if ((bw[u] >> lane) & 1u) row.template values<K>(base + (w0 + u) * 32 + lane, v[u]);
                }
#pragma unroll
                for (int u = 0; u < UX; ++u) {
                    const unsigned at = __shfl_sync(0xffffffffu, xo, w0 + u) + __popc(bw[u] & lt);
                    if ((bw[u] >> lane) & 1u) put(v[u], o0 + at);
                }
            }
        } else {
            sel_stage(word, xo, stage);
#pragma unroll 1
            for (unsigned e0 = 0; e0 < sn; e0 += 32 * UX) {
                int32_t v[UX][K];
#pragma unroll
                for (int u = 0; u < UX; ++u) {
                    const unsigned e = e0 + u * 32 + lane;
                    if (e < sn) row.template values<K>(base + stage[e], v[u]);
                }
#pragma unroll
                for (int u = 0; u < UX; ++u) {
                    const unsigned e = e0 + u * 32 + lane;
                    if (e < sn) put(v[u], o0 + e);
                }
            }
            __syncwarp();  // the stage is rewritten by the next step
        }
    });
    if (BOUNDS) merge_bounds<K>(mm, k_out, lo, hi);
}

template <class Row, int K>
int expand_k(tid_ctx *ctx, const Row &row, int k_out, const OutCols &out, int64_t cap, const SelScratch &sc,
             const BoundsOut &mm) {
    if (mm.acc) k_sel_expand<Row, K, true><<<sc.ranges, SEL_THREADS, 0, ctx->stream>>>(row, k_out, out, cap, sc, mm);
    else k_sel_expand<Row, K, false><<<sc.ranges, SEL_THREADS, 0, ctx->stream>>>(row, k_out, out, cap, sc, mm);
    return launch_check("k_sel_expand");
}

template <class Row>
int launch_compact(tid_ctx *ctx, Row row, int64_t n, int k_out, const OutCols &out, int64_t cap,
                   int64_t *d_rows, int64_t *h_rows_dev, const BoundsOut &mm = BoundsOut{}) {
    if (n == 0) {
        TID_TRY_CUDA(cudaMemsetAsync(d_rows, 0, sizeof(int64_t), ctx->stream), "memset rows");
        TID_TRY_CUDA(cudaMemsetAsync(h_rows_dev, 0, sizeof(int64_t), ctx->stream), "memset rows");
        return TID_OK;
    }
    if (n < SEL_MIN_ROWS) {
        static bool opted = false;  // staging of up to TID_MAX_COLS columns of a tile
        if (!opted) {
            TID_TRY_CUDA(cudaFuncSetAttribute(k_compact<Row>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)(sizeof(int32_t) * TID_MAX_COLS * CP_TILE)),
                         "k_compact smem");
            opted = true;
        }
        const unsigned tiles = (unsigned)ceil_div(n, CP_TILE);
        Lookback lb{};
        TID_TRY(lookback_scratch(ctx, tiles, &lb));
        const size_t smem = sizeof(int32_t) * (size_t)std::max(1, k_out) * CP_TILE;
        k_compact<Row><<<tiles, CP_THREADS, smem, ctx->stream>>>(row, n, k_out, out, cap, d_rows, h_rows_dev, lb, mm);
        return launch_check("k_compact");
    }
    size_t stash_b = 0;
    if constexpr (std::is_same_v<Row, BindRow>) {
        if (row.n_eq == 0 && (row.test & (row.test - 1)) == 0) stash_b = (size_t)n * 4;
    }
    SelScratch sc{};
    void *blk = nullptr, *stash = nullptr;
    TID_TRY(sel_scratch(ctx, n, 1, stash_b, &sc, &blk, &stash));
    if constexpr (std::is_same_v<Row, BindRow>) {
        if (stash_b) row.stash = (int32_t *)stash;
    }
    k_sel_mark<Row><<<sc.ranges, SEL_THREADS, 0, ctx->stream>>>(row, (uint32_t)n, sc, d_rows, h_rows_dev);
    int rc = launch_check("k_sel_mark");
    if (rc == TID_OK) {
        if (k_out <= 1) rc = expand_k<Row, 1>(ctx, row, k_out, out, cap, sc, mm);
        else if (k_out == 2) rc = expand_k<Row, 2>(ctx, row, k_out, out, cap, sc, mm);
        else if (Row::MAX_K == 3 || k_out == 3) rc = expand_k<Row, 3>(ctx, row, k_out, out, cap, sc, mm);
        else if constexpr (Row::MAX_K > 3) rc = expand_k<Row, Row::MAX_K>(ctx, row, k_out, out, cap, sc, mm);
    }
    dev_free(ctx, blk);
    return rc;
}

// Bind with nothing to test (no repeated variable, no predicate): every row is
// kept in index order, so row r is written at r -- a plain gather, no
// compaction -- with the column bounds of the output.
__global__ void __launch_bounds__(256) k_bind_gather(BindRow row, int64_t n, OutCols out, BoundsOut mm,
                                                     int64_t *__restrict__ d_rows, int64_t *__restrict__ h_rows) {
    constexpr int K = 3, U = 4;  // a pattern has at most three variables; rows per thread in flight
    uint32_t lo[K], hi[K];
#pragma unroll
    for (int c = 0; c < K; ++c) {
        lo[c] = 0xFFFFFFFFu;
        hi[c] = 0u;
    }
    const int64_t stride = (int64_t)gridDim.x * (256 * U);
    for (int64_t r0 = (int64_t)blockIdx.x * (256 * U) + threadIdx.x; r0 < n; r0 += stride) {
        int32_t v[U][K];
#pragma unroll
        for (int u = 0; u < U; ++u) row.template values<K>(min(r0 + u * 256, n - 1), v[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t r = r0 + u * 256;
            if (r >= n) continue;
#pragma unroll
            for (int c = 0; c < K; ++c) {
                if (c < row.k) {
                    out.col[c][r] = v[u][c];
                    const uint32_t x = (uint32_t)v[u][c] ^ 0x80000000u;
                    lo[c] = min(lo[c], x);
                    hi[c] = max(hi[c], x);
                }
            }
        }
    }
    if (mm.acc) merge_bounds<K>(mm, row.k, lo, hi);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *d_rows = n;
        *h_rows = n;
    }
}

// bits: one per term of the column that lies in [lo, lo + w); 0 sets none
__global__ void __launch_bounds__(256) k_member_bits(const int32_t *__restrict__ col, int64_t n, uint32_t lo,
                                                     uint32_t w, uint32_t *__restrict__ bits) {
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const int32_t x = col[i];
        const uint32_t d = ((uint32_t)x ^ 0x80000000u) - lo;
        if (x != 0 && d < w) atomicOr(bits + (d >> 5), 1u << (d & 31));
    }
}

// ---- exclusive scan of uint32 (look-back) --------------------------------------

constexpr int SC_THREADS = 256, SC_ITEMS = 16, SC_TILE = SC_THREADS * SC_ITEMS;
static_assert(SC_TILE == SCAN_TILE, "the callers' tile");
static_assert(SC_ITEMS == 16, "k_scan_u32 splits tile positions as (e >> 4, e & 15)");

// Exclusive scan of one 4096-item tile; the tile's first output is `prefix`
// (from offs[tile] when offs is given, else by decoupled look-back -- used for a
// single tile, where nothing waits).  total_out: the sum of all items.
__global__ void __launch_bounds__(SC_THREADS)
k_scan_u32(const uint32_t *__restrict__ in, uint32_t *__restrict__ out, int64_t n,
           unsigned long long *__restrict__ total_out, Lookback lb, const uint32_t *__restrict__ offs) {
    __shared__ unsigned s_tile;
    __shared__ uint32_t s_w[SC_THREADS / 32];
    __shared__ long long s_prefix;
    // the tile, thread-blocked (thread t's items at t * 17 .. t * 17 + 15: the
    // odd stride keeps a warp's blocked reads on distinct banks); global loads
    // and stores go through it striped, so they are coalesced
    __shared__ uint32_t s_t[SC_THREADS * (SC_ITEMS + 1)];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = offs ? blockIdx.x : lb_ticket(lb);
    __syncthreads();
    const unsigned tile = s_tile;
    if (!offs && tile >= lb.num_tiles) return;
    const int64_t base0 = (int64_t)tile * SC_TILE;
#pragma unroll
    for (int i = 0; i < SC_ITEMS; ++i) {
        const int e = i * SC_THREADS + threadIdx.x;
        s_t[(e >> 4) * (SC_ITEMS + 1) + (e & 15)] = base0 + e < n ? in[base0 + e] : 0u;
    }
    __syncthreads();
    uint32_t v[SC_ITEMS];
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < SC_ITEMS; ++i) {
        v[i] = s_t[threadIdx.x * (SC_ITEMS + 1) + i];
        sum += v[i];
    }
    uint32_t x = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if ((int)lane >= d) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < SC_THREADS / 32 ? s_w[lane] : 0u;
        uint32_t y = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t z = __shfl_up_sync(0xffffffffu, y, d);
            if ((int)lane >= d) y += z;
        }
        if (lane < SC_THREADS / 32) s_w[lane] = y - w;
        const uint32_t total = __shfl_sync(0xffffffffu, y, 31);
        if (offs) {
            if (lane == 0) s_prefix = offs[tile];
        } else {
            const long long excl = lb_exclusive_prefix(lb, tile, total);
            if (lane == 0) {
                s_prefix = excl;
                if (tile == lb.num_tiles - 1 && excl >= 0 && total_out) *total_out = excl + total;
            }
        }
    }
    __syncthreads();
    if (s_prefix < 0) return;
    uint32_t run = (uint32_t)s_prefix + s_w[warp] + (x - sum);
#pragma unroll
    for (int i = 0; i < SC_ITEMS; ++i) {
        s_t[threadIdx.x * (SC_ITEMS + 1) + i] = run;
        run += v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SC_ITEMS; ++i) {
        const int e = i * SC_THREADS + threadIdx.x;
        if (base0 + e < n) out[base0 + e] = s_t[(e >> 4) * (SC_ITEMS + 1) + (e & 15)];
    }
}

// sums[t] = sum of the items of tile t (SC_TILE items)
__global__ void __launch_bounds__(SC_THREADS) k_tile_sums(const uint32_t *__restrict__ in, int64_t n,
                                                          uint32_t *__restrict__ sums) {
    __shared__ uint32_t s_w[SC_THREADS / 32];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * SC_TILE;
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < SC_ITEMS; ++i) {  // striped: coalesced
        const int64_t j = base + i * SC_THREADS + threadIdx.x;
        sum += j < n ? in[j] : 0u;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
    if (lane == 0) s_w[warp] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < SC_THREADS / 32; ++w) t += s_w[w];
        sums[blockIdx.x] = t;
    }
}

}  // namespace

int bounds_out(tid_set *set, BoundsOut *b) {
    tid_ctx *ctx = set->ctx;
    if (set->k > BOUND_COLS) return fail(TID_ERR_ARG, "bounds of %d columns", set->k);
    if (!ctx->kept) TID_TRY(keep_scratch(ctx));
    b->acc = ctx->bounds_dev;
    b->done = ctx->bounds_dev + 2 * TID_MAX_COLS;
    b->host = (uint32_t *)(set->slot.dev + 1);
    static_assert(offsetof(SlotWords, bounds) == sizeof(int64_t), "the bounds follow the row count");
    return TID_OK;
}

void read_bounds(const tid_set *set, int k, uint32_t *lo, uint32_t *hi) {
    const volatile uint32_t *w = set->slot.words->bounds;
    for (int c = 0; c < k; ++c) {
        lo[c] = w[c];
        hi[c] = w[BOUND_COLS + c];
    }
}

int sel_scratch(tid_ctx *ctx, int64_t n, int lists, size_t extra, SelScratch *sc, void **block, void **extra_at,
                unsigned per) {
    sc->steps = (unsigned)ceil_div(n, (int64_t)SEL_STEP);
    // a range is one step per warp, or four once that still gives every SM eight CTAs
    sc->per = per ? per : sc->steps >= (unsigned)sm_count() * 256 ? 4 * SEL_WARPS : SEL_WARPS;
    sc->ranges = (unsigned)ceil_div(sc->steps, (int64_t)sc->per);
    auto pad = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t bits_b = (size_t)sc->steps * 32 * 4 * lists, cnt_b = pad((size_t)sc->steps * 4 * lists);
    const size_t off_b = pad((size_t)sc->ranges * 8 * lists), tot_b = pad((size_t)sc->ranges * 4 * lists);
    // a graph counts in its own word: it may run beside the context's later work
    const bool in_graph = capturing(ctx);
    if (!in_graph && !ctx->kept) TID_TRY(keep_scratch(ctx));
    const size_t extra_b = pad(extra);
    void *blk = nullptr;
    TID_TRY(dev_alloc(ctx, &blk, bits_b + cnt_b + off_b + tot_b + extra_b + (in_graph ? 256 : 0)));
    char *p = (char *)blk;
    sc->bits = (uint32_t *)p;
    sc->cnt = (uint32_t *)(p += bits_b);
    sc->off = (unsigned long long *)(p += cnt_b);
    sc->tot = (uint32_t *)(p += off_b);
    p += tot_b;
    if (extra_at) *extra_at = p;
    sc->done = ctx->sel_done;
    if (in_graph) {
        sc->done = (unsigned *)(p + extra_b);
        cudaError_t e = cudaMemsetAsync(sc->done, 0, sizeof(unsigned), ctx->stream);
        if (e != cudaSuccess) {
            dev_free(ctx, blk);
            return fail_cuda(e, "row selection");
        }
    }
    *block = blk;
    return TID_OK;
}

int scan_exclusive_u32(tid_ctx *ctx, const uint32_t *in, uint32_t *out, int64_t n,
                       unsigned long long *total_dev, const uint32_t *tile_sums) {
    if (n == 0) {
        if (total_dev) TID_TRY_CUDA(cudaMemsetAsync(total_dev, 0, 8, ctx->stream), "memset");
        return TID_OK;
    }
    const unsigned tiles = (unsigned)ceil_div(n, SC_TILE);
    if (tiles == 1) {  // one tile: nothing to wait for
        Lookback lb{};
        TID_TRY(lookback_scratch(ctx, 1, &lb));
        k_scan_u32<<<1, SC_THREADS, 0, ctx->stream>>>(in, out, n, total_dev, lb, nullptr);
        return launch_check("k_scan_u32");
    }
    // reduce, scan the tile sums (recursively), scan each tile from its offset:
    // no tile waits for another
    uint32_t *sums = nullptr;
    TID_TRY(dev_alloc(ctx, (void **)&sums, sizeof(uint32_t) * 2 * (size_t)tiles + 256));
    uint32_t *offs = sums + tiles;
    int rc = TID_OK;
    if (!tile_sums) {
        k_tile_sums<<<tiles, SC_THREADS, 0, ctx->stream>>>(in, n, sums);
        rc = launch_check("k_tile_sums");
    }
    if (rc == TID_OK) rc = scan_exclusive_u32(ctx, tile_sums ? tile_sums : sums, offs, tiles, total_dev);
    if (rc == TID_OK) {
        k_scan_u32<<<tiles, SC_THREADS, 0, ctx->stream>>>(in, out, n, nullptr, Lookback{}, offs);
        rc = launch_check("k_scan_u32");
    }
    dev_free(ctx, sums);
    return rc;
}

int compact_bind(tid_ctx *ctx, const tid_store *st, const tid_pattern &pat, const int32_t *idx, int64_t n,
                 const Pred *preds, int n_preds, const BindMember *mem, int n_mem, tid_set *out, const BoundsOut &mm) {
    BindRow r{};
    r.S = st->s;
    r.P = st->p;
    r.O = st->o;
    r.idx = idx;
    r.k = out->k;
    const int8_t var[3] = {pat.var[0], pat.var[1], pat.var[2]};
    r.need = (var[0] >= 0 ? 1 : 0) | (var[1] >= 0 ? 2 : 0) | (var[2] >= 0 ? 4 : 0);
    for (int c = 0; c < out->k; ++c) {
        r.src[c] = -1;
        for (int j = 0; j < 3; ++j)
            if (var[j] == out->vars[c]) {
                r.src[c] = (int8_t)j;
                break;
            }
    }
    r.n_eq = 0;
    for (int a = 0; a < 3; ++a)
        for (int b = a + 1; b < 3; ++b)
            if (var[a] >= 0 && var[a] == var[b]) {
                r.eq_a[r.n_eq] = (int8_t)a;
                r.eq_b[r.n_eq] = (int8_t)b;
                r.n_eq++;
            }
    r.n_preds = n_preds;
    for (int q = 0; q < n_preds; ++q) {  // a test reads a slot of the triple
        r.preds[q] = preds[q];
        r.preds[q].col = r.src[preds[q].col];
        r.test |= 1 << r.preds[q].col;
    }
    for (int e = 0; e < r.n_eq; ++e) r.test |= (1 << r.eq_a[e]) | (1 << r.eq_b[e]);
    r.n_mem = n_mem;
    for (int q = 0; q < n_mem; ++q) {
        r.mem[q] = mem[q].m;
        r.mem_slot[q] = r.src[mem[q].col];
        r.test |= 1 << r.mem_slot[q];
    }
    OutCols oc{};
    for (int c = 0; c < out->k; ++c) oc.col[c] = out->col[c];
    if (n > 0 && r.test == 0 && n <= out->cap) {
        k_bind_gather<<<grid_for(n, 256 * 4, 8), 256, 0, ctx->stream>>>(r, n, oc, mm, out->d_rows, out->slot.dev);
        return launch_check("k_bind_gather");
    }
    return launch_compact(ctx, r, n, out->k, oc, out->cap, out->d_rows, out->slot.dev, mm);
}

int expand_keyed(tid_ctx *ctx, const KeyedScan &ks, const SelScratch &sc, const int8_t *src, const int32_t *map,
                 tid_set *out, const BoundsOut &mm) {
    KeyedRow r{};
    r.S = ks.col[0];
    r.P = ks.col[1];
    r.O = ks.col[2];
    r.key_slot = ks.key_slot;
    r.keys = ks.keys;
    r.map = map;
    r.k = out->k;
    OutCols oc{};
    for (int c = 0; c < out->k; ++c) {
        r.src[c] = src[c];
        oc.col[c] = out->col[c];
    }
    if (out->k == 2) return expand_k<KeyedRow, 2>(ctx, r, out->k, oc, out->cap, sc, mm);
    return expand_k<KeyedRow, 3>(ctx, r, out->k, oc, out->cap, sc, mm);
}

int compact_filter(tid_ctx *ctx, const tid_set *in, int64_t n, const Pred *preds, int n_preds, tid_set *out) {
    FilterRow r{};
    r.k = in->k;
    for (int c = 0; c < in->k; ++c) r.col[c] = in->col[c];
    r.n_preds = n_preds;
    for (int q = 0; q < n_preds; ++q) r.preds[q] = preds[q];
    OutCols oc{};
    for (int c = 0; c < out->k; ++c) oc.col[c] = out->col[c];
    return launch_compact(ctx, r, n, out->k, oc, out->cap, out->d_rows, out->slot.dev);
}

int member_bits(tid_ctx *ctx, const int32_t *col, int64_t n, uint32_t lo, uint32_t hi, Members *m) {
    const uint64_t w = (uint64_t)hi - lo + 1;
    const size_t words = (size_t)((w + 31) / 32);
    void *p = nullptr;
    TID_TRY(dev_alloc(ctx, &p, words * 4));
    m->bits = (uint32_t *)p;
    m->lo = lo;
    m->w = (uint32_t)std::min<uint64_t>(w, 0xFFFFFFFFu);
    cudaError_t e = cudaMemsetAsync(p, 0, words * 4, ctx->stream);
    int rc = e == cudaSuccess ? TID_OK : fail_cuda(e, "member bits");
    if (rc == TID_OK && n > 0) {
        k_member_bits<<<grid_for(n, 256, 8), 256, 0, ctx->stream>>>(col, n, m->lo, m->w, (uint32_t *)p);
        rc = launch_check("k_member_bits");
    }
    if (rc != TID_OK) {
        dev_free(ctx, p);
        m->bits = nullptr;
    }
    return rc;
}

int compact_member(tid_ctx *ctx, const tid_set *in, int64_t n, const Members &m, tid_set *out) {
    MemberRow r{};
    r.k = in->k;
    for (int c = 0; c < in->k; ++c) r.col[c] = in->col[c];
    r.m = m;
    OutCols oc{};
    for (int c = 0; c < out->k; ++c) oc.col[c] = out->col[c];
    return launch_compact(ctx, r, n, out->k, oc, out->cap, out->d_rows, out->slot.dev);
}

int compact_unique(tid_ctx *ctx, const int32_t *const *cols, int k, const int32_t *perm, int64_t n,
                   tid_set *out) {
    UniqueRow r{};
    r.k = k;
    for (int c = 0; c < k; ++c) r.col[c] = cols[c];
    r.perm = perm;
    OutCols oc{};
    for (int c = 0; c < out->k; ++c) oc.col[c] = out->col[c];
    return launch_compact(ctx, r, n, out->k, oc, out->cap, out->d_rows, out->slot.dev);
}

int find_repeats(tid_ctx *ctx, const tid_set *in, int64_t n, tid_set *flag) {
    if (!ctx->kept) TID_TRY(keep_scratch(ctx));
    SetCols sc{};
    for (int c = 0; c < in->k; ++c) sc.col[c] = in->col[c];
    const unsigned steps = (unsigned)ceil_div(n, (int64_t)SEL_STEP);
    k_repeats<<<grid_for(steps, RP_THREADS / 32, 8), RP_THREADS, 0, ctx->stream>>>(
        sc, in->k, (uint32_t)n, steps, ctx->sel_done + 1, ctx->sel_done, flag->d_rows, flag->slot.dev);
    return launch_check("k_repeats");
}

int compact_unique_packed(tid_ctx *ctx, const void *keys, bool wide, int k, int64_t n, const PackSpec &ps,
                          tid_set *out) {
    OutCols oc{};
    for (int c = 0; c < out->k; ++c) oc.col[c] = out->col[c];
    if (wide) {
        PackedUniqueRow<unsigned long long> r{(const unsigned long long *)keys, ps, k};
        return launch_compact(ctx, r, n, out->k, oc, out->cap, out->d_rows, out->slot.dev);
    }
    PackedUniqueRow<uint32_t> r{(const uint32_t *)keys, ps, k};
    return launch_compact(ctx, r, n, out->k, oc, out->cap, out->d_rows, out->slot.dev);
}

}  // namespace tid
