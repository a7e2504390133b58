// K5 / K6: inner join of two tuple sets on all shared variables.
//
// Section 4.2 joins subquery result vectors by copying the related terms into
// key vectors, sorting them, and running a merge-join that returns pairs of
// matching positions, from which the remaining values are gathered; the
// relationship table lists the nine S/P/O position pairings a shared term can
// take, which here are simply the columns of the shared variables.
//
// Both algorithms follow the same three phases (the two-phase output sizing
// of He et al. that the paper cites): count matches per row, exclusive-scan
// the counts (one synchronisation reads the total to size the output), then
// write every output row with one thread -- the output is cut into tiles of equal
// work, and within a tile a running maximum over the rows' first output rows gives
// every output row its left row -- so a key with millions of matches is spread
// over as many threads (no per-row serial loops).
//
//  * runs: the right side leads with the key columns, so a key's rows are one run
//    of it, ordered by its other columns; each left row, whatever its order by
//    the key, finds its run and is written with it, which is canonical order --
//    no sort.  A run is found through a table over the range of the first key
//    column (a bucket's first and one-past-last right row), then by binary
//    search inside the bucket where it holds more than the one key.
//  * members: when one side holds a single key column and nothing else, the
//    join keeps the rows of the other side whose key is among its terms (one
//    bit per term): a row selection, no search and no count read-back.
//  * sort-merge (the right side does not lead with the key): both sides ordered
//    by the key (a radix-sorted permutation where it is no prefix); per left
//    row, lower/upper bound in the right keys.
//  * hash: the smaller side is grouped by key in an open-addressing table
//    (key -> [start, count) into a grouped row array, built with CAS inserts,
//    a scan and a scatter); the other side probes it.  A table of at most
//    2048 slots is copied into shared memory by every probing CTA.
// A key value 0 (unbound) never matches.  The output is sorted to canonical
// order unless it is written in that order already (both inputs lead with the
// shared variables); a join of two sets is a set, so no duplicate removal is
// needed.
//
// Left outer join (OPTIONAL; the library the paper used also offered outer and
// left joins, Section 4.2): sort-merge only; a left row without a match counts
// as one output row (its right range marked empty) and is written with the
// right side's other columns 0 (unbound).

#include <algorithm>

#include "lookback.cuh"
#include "ops.cuh"

namespace tid {

int set_rows_const(tid_set *set, int64_t n);

namespace {

struct Cols {
    const int32_t *c[TID_MAX_COLS];
};
struct MCols {
    int32_t *c[TID_MAX_COLS];
};

// Column loops run to TID_MAX_COLS with a guard: constant indices keep the
// column pointers in registers (a loop bounded by nk would copy the parameter
// arrays to local memory).
__device__ __forceinline__ int cmp_rows(const Cols &A, int64_t a, const Cols &B, int64_t b, int nk) {
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c) {
        if (c >= nk) break;
        const int32_t x = A.c[c][a], y = B.c[c][b];
        if (x != y) return x < y ? -1 : 1;
    }
    return 0;
}

__device__ __forceinline__ bool has_zero(const Cols &A, int64_t a, int nk) {
    bool z = false;
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c)
        if (c < nk) z = z || A.c[c][a] == 0;
    return z;
}

// Output row o of a join: L's kl columns of row lr, then R's other columns of
// row rr (rr < 0: unbound, 0).  outL / outR point at the output columns of
// each part, so every index here is a constant.
__device__ __forceinline__ void write_out(const Cols &L, int kl, const Cols &Rrest, int nrest, int64_t lr, int64_t rr,
                                          const MCols &outL, const MCols &outR, int64_t o) {
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c)
        if (c < kl) outL.c[c][o] = L.c[c][lr];
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c)
        if (c < nrest) outR.c[c][o] = rr < 0 ? 0 : Rrest.c[c][rr];
}

__device__ __forceinline__ void block_add_u64(unsigned long long v, unsigned long long *total) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(total, v);
}

// ---- sort-merge --------------------------------------------------------------
// [lo, hi) of the right keys equal to left key row l, searched inside [a0, b0)
__device__ __forceinline__ void eq_range(const Cols &RK, const Cols &LK, int64_t l, int nk, int64_t a0, int64_t b0,
                                         int64_t *lo, int64_t *hi) {
    int64_t a = a0, b = b0;  // lower bound
    while (a < b) {
        const int64_t m = (a + b) >> 1;
        if (cmp_rows(RK, m, LK, l, nk) < 0) a = m + 1;
        else b = m;
    }
    int64_t a2 = a, b2 = b0;  // upper bound
    while (a2 < b2) {
        const int64_t m = (a2 + b2) >> 1;
        if (cmp_rows(RK, m, LK, l, nk) <= 0) a2 = m + 1;
        else b2 = m;
    }
    *lo = a;
    *hi = a2;
}

// The left keys are sorted, so the right range of every left row of a warp
// lies between the lower bound of the warp's first row and the upper bound of
// its last: two searches over all of R per warp (lanes 0 and 31), then each
// lane searches only that bracket (a few cache lines, not DRAM at every level).
// first / last: the warp's first and last left rows (valid, first <= last).
__device__ __forceinline__ void warp_bracket(const Cols &RK, const Cols &LK, int nk, int64_t nr, int64_t first,
                                             int64_t last, int64_t *a0, int64_t *b0) {
    const unsigned lane = threadIdx.x & 31;
    int64_t lo = 0, hi = nr;
    if (lane == 0) {
        int64_t x, y;
        eq_range(RK, LK, first, nk, 0, nr, &x, &y);
        lo = x;
    } else if (lane == 31) {
        int64_t x, y;
        eq_range(RK, LK, last, nk, 0, nr, &x, &y);
        hi = y;
    }
    *a0 = __shfl_sync(0xffffffffu, lo, 0);
    *b0 = __shfl_sync(0xffffffffu, hi, 31);
}

constexpr uint32_t NO_MATCH = 0xFFFFFFFFu;  // left outer join: a left row written once, padded

// Where the right rows of a first-key term lie: bucket (order(term) - lo) >> shift
// holds rows [x, y) (x == y: none), for terms with order in [lo, lo + span].
// At most one bucket per right row, so the table is no
// larger than two columns of the right side and stays in L2 with it; IDs of a
// graph are dense, and the shift is then 0.
struct RunTable {
    uint2 *bucket;  // null: none (search the whole right side)
    uint32_t lo, span;
    int shift;
};

__device__ __forceinline__ uint32_t sort_order(int32_t x) { return (uint32_t)x ^ 0x80000000u; }

__global__ void __launch_bounds__(256) k_run_table(const int32_t *__restrict__ key, int64_t nr, RunTable t) {
    constexpr int U = 4;
    for (int64_t i0 = (int64_t)blockIdx.x * (256 * U) + threadIdx.x; i0 < nr; i0 += (int64_t)gridDim.x * (256 * U)) {
        int32_t x[U], y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = min(i0 + u * 256, nr - 1);
            x[u] = key[i];
            y[u] = key[i > 0 ? i - 1 : 0];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * 256;
            if (i >= nr) break;
            const uint32_t dx = sort_order(x[u]) - t.lo, dy = sort_order(y[u]) - t.lo;
            if (dx > t.span || dy > t.span) continue;  // outside the column's bounds: not a row of this column
            const uint32_t b = dx >> t.shift, p = dy >> t.shift;
            if (i == 0 || b != p) {
                t.bucket[b].x = (uint32_t)i;
                if (i > 0) t.bucket[p].y = (uint32_t)i;
            }
            if (i == nr - 1) t.bucket[b].y = (uint32_t)nr;
        }
    }
}

// cnt[l] right rows match left row l, from lo_out[l] on; exact: a bucket of the
// table holds the rows of one key.  A CTA takes a tile of the scan that follows and
// leaves its sum.
__global__ void __launch_bounds__(256) k_run_count(Cols LK, int64_t nl, Cols RK, int nk, bool left, RunTable t, bool exact,
                                                   uint32_t *__restrict__ cnt, uint32_t *__restrict__ lo_out,
                                                   unsigned long long *__restrict__ total,
                                                   uint32_t *__restrict__ sums) {
    constexpr int U = 4;  // rows per thread whose table reads are in flight together
    __shared__ unsigned s_sum[8];
    unsigned long long acc = 0;
    const int64_t begin = (int64_t)blockIdx.x * SCAN_TILE, end = min(begin + SCAN_TILE, nl);
    for (int64_t l0 = begin + threadIdx.x; l0 < end; l0 += 256 * U) {
        uint2 b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t l = min(l0 + u * 256, nl - 1);
            const int32_t x = LK.c[0][l];
            const uint32_t d = sort_order(x) - t.lo;
            b[u] = x != 0 && d <= t.span ? t.bucket[d >> t.shift] : make_uint2(0, 0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t l = l0 + u * 256;
            if (l >= nl) break;
            uint32_t c = b[u].y - b[u].x, lo = b[u].x;
            if (!exact && c) {
                int64_t a = 0, a2 = 0;
                if (!has_zero(LK, l, nk)) eq_range(RK, LK, l, nk, b[u].x, b[u].y, &a, &a2);
                lo = (uint32_t)a;
                c = (uint32_t)(a2 - a);
            }
            if (left && c == 0) {
                c = 1;
                lo = NO_MATCH;
            }
            cnt[l] = c;
            lo_out[l] = lo;
            acc += c;
        }
    }
    block_add_u64(acc, total);  // once per warp: one address takes these atomics one at a time
    const unsigned w = __reduce_add_sync(0xffffffffu, (unsigned)acc);
    if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = w;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned s = 0;
        for (int i = 0; i < 8; ++i) s += s_sum[i];
        sums[blockIdx.x] = s;
    }
}

// The same by binary search over all of the right keys; the left keys are sorted.
__global__ void k_sm_count(Cols LK, int64_t nl, Cols RK, int64_t nr, int nk, bool left, uint32_t *__restrict__ cnt,
                           uint32_t *__restrict__ lo_out, unsigned long long *__restrict__ total) {
    unsigned long long acc = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n_iter = ceil_div(nl, stride) * stride;
    for (int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; l < n_iter; l += stride) {
        const int64_t w0 = l - (threadIdx.x & 31);  // the warp's rows: w0 .. w0 + 31
        int64_t a0 = 0, b0 = nr;
        if (w0 < nl) warp_bracket(RK, LK, nk, nr, w0, min(w0 + 31, nl - 1), &a0, &b0);
        if (l < nl) {
            uint32_t c = 0, lo = 0;
            if (!has_zero(LK, l, nk)) {
                int64_t a, a2;
                eq_range(RK, LK, l, nk, a0, b0, &a, &a2);
                lo = (uint32_t)a;
                c = (uint32_t)(a2 - a);
            }
            if (left && c == 0) {
                c = 1;
                lo = NO_MATCH;
            }
            cnt[l] = c;
            lo_out[l] = lo;
            acc += c;
        }
    }
    block_add_u64(acc, total);  // once per warp: one address takes these atomics one at a time
}

// Output rows of probe rows: probe row l's matches are written at off[l] ..
// off[l + 1] - 1 (off the exclusive scan of the counts, total their sum).
// Load-balanced search (the merge-path partition of Odeh et al. applied to
// the sequences of row starts and output rows): CTA t takes items [t T, (t+1) T)
// of their merged order (row l before output o when off[l] <= o), i.e. some
// probe rows and the output rows next to them -- at most T items in all, so
// neither a long run of rows without matches nor one row with millions of
// matches makes a CTA's work unbounded.  The CTA stages its rows' offsets in
// shared memory and marks where each row's output begins; a running maximum then
// gives every output row its probe row (with a binary search per output row, a
// search per tile boundary by one thread and the scan's own sums, the join of 8M
// with 8M rows took 273 us, now 226).  Consecutive output rows go to consecutive
// threads (coalesced stores).
constexpr int JW_THREADS = 256;
constexpr int JW_ITEMS = 8;
constexpr int JW_TILE = JW_THREADS * JW_ITEMS;

// split[t] = rows among the first t JW_TILE items of the merged order, for every
// tile boundary: a warp each, 32 places tested at once (its own launch: a search
// inside the write kernel was some twenty dependent loads at the start of every CTA)
__global__ void __launch_bounds__(256) k_join_split(const uint32_t *__restrict__ off, int64_t nl, int64_t total,
                                                    int64_t tiles, uint32_t *__restrict__ split) {
    const int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (t > tiles) return;
    const unsigned lane = threadIdx.x & 31;
    const int64_t d = min(t * JW_TILE, nl + total);
    int64_t lo = max((int64_t)0, d - total), hi = min(d, nl);
    while (lo < hi) {  // row m is among the first d items if off[m] <= d - 1 - m; lane l tests the l-th part's end
        const int64_t part = (hi - lo + 31) / 32, m = lo + (lane + 1) * part - 1;
        const bool in = m < hi && (int64_t)off[m] <= d - 1 - m;
        lo += (int64_t)__popc(__ballot_sync(0xffffffffu, in)) * part;
        hi = min(hi, lo + part - 1);
    }
    if (lane == 0) split[t] = (uint32_t)min(lo, min(d, nl));
}

__global__ void __launch_bounds__(JW_THREADS) k_join_write(const uint32_t *__restrict__ off, int64_t nl,
                                                           const uint32_t *__restrict__ lo,
                                                           const int32_t *__restrict__ lperm,
                                                           const int32_t *__restrict__ rmap,
                                                           const int32_t *__restrict__ rperm, int64_t total, Cols L,
                                                           int kl, Cols Rrest, int nrest, MCols outL, MCols outR,
                                                           bool left_is_probe, const uint32_t *__restrict__ split,
                                                           int64_t *__restrict__ d_rows, int64_t *__restrict__ h_rows) {
    __shared__ uint32_t s_off[JW_TILE + 1], s_lo[JW_TILE + 1];  // of rows rb .. r1 - 1
    __shared__ __align__(16) uint16_t s_row[JW_TILE];  // output row o0 + i belongs to probe row rb + s_row[i]
    __shared__ unsigned s_wmax[JW_THREADS / 32];
    const int64_t d0 = (int64_t)blockIdx.x * JW_TILE, d1 = min(d0 + JW_TILE, nl + total);
    const int64_t r0 = split[blockIdx.x], r1 = split[blockIdx.x + 1];
    const int64_t o0 = d0 - r0, o1 = d1 - r1;
    if (d_rows && blockIdx.x == 0 && threadIdx.x == 0) {  // the result's row count
        *d_rows = total;
        *h_rows = total;
    }
    if (o0 >= o1) return;  // only rows here
    // the output rows [o0, o1) belong to rows rb .. r1 - 1: row r0 - 1 precedes
    // output o0 in the merged order (off[r0 - 1] <= o0), row r1 follows o1 - 1
    const int64_t rb = r0 > 0 ? r0 - 1 : 0;
    const int nr = (int)(r1 - rb);
    for (int i = threadIdx.x; i < nr; i += JW_THREADS) {
        s_off[i] = off[rb + i];
        s_lo[i] = lo[rb + i];
    }
    static_assert(JW_ITEMS == 8, "a thread scans eight 16-bit entries as one 16-byte word");
    reinterpret_cast<uint4 *>(s_row)[threadIdx.x] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    // The probe row of every output row: each row with output in the tile enters
    // itself at its first output row (of rows with one offset, the last has the
    // output; row 0 holds what was begun before the tile), then a running maximum.
    for (int i = threadIdx.x; i < nr; i += JW_THREADS) {
        const uint32_t f = s_off[i];
        if ((i + 1 == nr || s_off[i + 1] > f) && f >= (uint32_t)o0 && f < (uint32_t)o1) s_row[f - (uint32_t)o0] = (uint16_t)i;
    }
    __syncthreads();
    {
        const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        uint4 w = reinterpret_cast<const uint4 *>(s_row)[threadIdx.x];
        unsigned e[8] = {w.x & 0xFFFFu, w.x >> 16, w.y & 0xFFFFu, w.y >> 16, w.z & 0xFFFFu, w.z >> 16, w.w & 0xFFFFu, w.w >> 16};
#pragma unroll
        for (int q = 1; q < 8; ++q) e[q] = max(e[q], e[q - 1]);
        unsigned x = e[7];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, d);
            if ((int)lane >= d) x = max(x, y);
        }
        if (lane == 31) s_wmax[warp] = x;
        unsigned before = __shfl_up_sync(0xffffffffu, x, 1);
        if (lane == 0) before = 0;
        __syncthreads();
        for (unsigned v = 0; v < warp; ++v) before = max(before, s_wmax[v]);
#pragma unroll
        for (int q = 0; q < 8; ++q) e[q] = max(e[q], before);
        reinterpret_cast<uint4 *>(s_row)[threadIdx.x] =
            make_uint4(e[0] | e[1] << 16, e[2] | e[3] << 16, e[4] | e[5] << 16, e[6] | e[7] << 16);
    }
    __syncthreads();
    // every output row's left and right row first, then column by column, so
    // that a column's reads are in flight together
    int32_t lr[JW_ITEMS], rr[JW_ITEMS];
    const int64_t last = o1 - 1;
#pragma unroll
    for (int q = 0; q < JW_ITEMS; ++q) {
        const int64_t o = min(o0 + q * JW_THREADS + threadIdx.x, last);
        const int a = s_row[o - o0];
        lr[q] = (int32_t)(rb + a);
        // left outer join: a left row alone, right columns unbound (-1)
        rr[q] = s_lo[a] == NO_MATCH ? -1 : (int32_t)(s_lo[a] + (uint32_t)(o - s_off[a]));
    }
    if (!left_is_probe) {  // hash join built on the left: the probe rows are right rows, rr indexes grouped left rows
#pragma unroll
        for (int q = 0; q < JW_ITEMS; ++q) {
            const int32_t j = rmap[rr[q]];
            rr[q] = lr[q];
            lr[q] = j;
        }
    } else {
        if (lperm) {
#pragma unroll
            for (int q = 0; q < JW_ITEMS; ++q) lr[q] = lperm[lr[q]];
        }
        if (rmap) {
#pragma unroll
            for (int q = 0; q < JW_ITEMS; ++q) rr[q] = rr[q] < 0 ? -1 : rmap[rr[q]];
        }
        if (rperm) {
#pragma unroll
            for (int q = 0; q < JW_ITEMS; ++q) rr[q] = rr[q] < 0 ? -1 : rperm[rr[q]];
        }
    }
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c) {
        if (c >= kl) break;
        int32_t v[JW_ITEMS];
#pragma unroll
        for (int q = 0; q < JW_ITEMS; ++q) v[q] = L.c[c][lr[q]];
#pragma unroll
        for (int q = 0; q < JW_ITEMS; ++q) {
            const int64_t o = o0 + q * JW_THREADS + threadIdx.x;
            if (o < o1) outL.c[c][o] = v[q];
        }
    }
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c) {
        if (c >= nrest) break;
        int32_t v[JW_ITEMS];
#pragma unroll
        for (int q = 0; q < JW_ITEMS; ++q) v[q] = rr[q] < 0 ? 0 : Rrest.c[c][rr[q]];
#pragma unroll
        for (int q = 0; q < JW_ITEMS; ++q) {
            const int64_t o = o0 + q * JW_THREADS + threadIdx.x;
            if (o < o1) outR.c[c][o] = v[q];
        }
    }
}

// Single-pass sort-merge join of inputs that both lead with the key (so they
// are sorted by it) when one side holds only key columns: then every row of
// the other side matches at most one row, the output has at most
// (|other side|, + |L| for a left join) rows, and it can be written without a
// separate count pass.  A CTA takes a tile of MJ_TILE left rows (tickets in
// order); each thread finds the matching range of its rows in R (two binary
// searches), the block scans the counts, the decoupled look-back gives the
// tile's first output row, and the CTA writes its output rows in order --
// an output row finds its left row by binary search over the tile's scanned
// counts in shared memory, so a key with many matches is spread over all the
// CTA's threads.  The output is canonical as written.
constexpr int MJ_THREADS = 256;
constexpr int MJ_ITEMS = 4;
constexpr int MJ_TILE = MJ_THREADS * MJ_ITEMS;

__global__ void __launch_bounds__(MJ_THREADS)
k_merge_join(Cols LK, int64_t nl, Cols RK, int64_t nr, int nk, bool left, Cols L, int kl, Cols Rrest, int nrest,
             MCols outL, MCols outR, int64_t cap, int64_t *__restrict__ d_rows, int64_t *__restrict__ h_rows,
             Lookback lb) {
    __shared__ uint32_t s_excl[MJ_TILE + 1], s_lo[MJ_TILE];
    __shared__ uint32_t s_wsum[MJ_THREADS / 32];
    __shared__ unsigned s_tile;
    __shared__ long long s_prefix;
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = lb_ticket(lb);
    __syncthreads();
    const unsigned tile = s_tile;
    if (tile >= lb.num_tiles) return;
    const int64_t l0 = (int64_t)tile * MJ_TILE;
    const int rows = (int)min((int64_t)MJ_TILE, nl - l0);
    uint32_t c[MJ_ITEMS], sum = 0;
    // the warp's left rows are l0 + 128 w .. + 127: bracket their right ranges
    const int wf = (int)warp * 32 * MJ_ITEMS;
    int64_t a0 = 0, b0 = nr;
    if (wf < rows) warp_bracket(RK, LK, nk, nr, l0 + wf, l0 + min(wf + 32 * MJ_ITEMS, rows) - 1, &a0, &b0);
#pragma unroll
    for (int i = 0; i < MJ_ITEMS; ++i) {  // thread t: left rows l0 + 4t .. 4t + 3
        const int li = (int)threadIdx.x * MJ_ITEMS + i;
        const int64_t l = l0 + li;
        uint32_t cnt = 0, lo = 0;
        if (li < rows) {
            if (!has_zero(LK, l, nk)) {
                int64_t a, a2;
                eq_range(RK, LK, l, nk, a0, b0, &a, &a2);
                lo = (uint32_t)a;
                cnt = (uint32_t)(a2 - a);
            }
            if (left && cnt == 0) {
                cnt = 1;
                lo = NO_MATCH;
            }
            s_lo[li] = lo;
        }
        c[i] = cnt;
        sum += cnt;
    }
    uint32_t x = sum;  // block exclusive scan of the per-thread sums
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if ((int)lane >= d) x += y;
    }
    if (lane == 31) s_wsum[warp] = x;
    __syncthreads();
    uint32_t wb = 0, tot = 0;
    for (int w = 0; w < MJ_THREADS / 32; ++w) {
        if (w < (int)warp) wb += s_wsum[w];
        tot += s_wsum[w];
    }
    uint32_t run = wb + x - sum;
#pragma unroll
    for (int i = 0; i < MJ_ITEMS; ++i) {
        s_excl[threadIdx.x * MJ_ITEMS + i] = run;
        run += c[i];
    }
    if (threadIdx.x == 0) s_excl[MJ_TILE] = tot;
    if (warp == 0) {
        const long long excl = lb_exclusive_prefix(lb, tile, tot);
        if (lane == 0) {
            s_prefix = excl;
            if (tile == lb.num_tiles - 1 && excl >= 0) {
                *d_rows = excl + tot;
                *h_rows = excl + tot;
            }
        }
    }
    __syncthreads();
    const long long base = s_prefix;
    if (base < 0) return;
    for (uint32_t o = threadIdx.x; o < tot; o += MJ_THREADS) {
        int a = 0, b = rows;  // first local row whose exclusive count exceeds o
        while (a < b) {
            const int m = (a + b) >> 1;
            if (s_excl[m] <= o) a = m + 1;
            else b = m;
        }
        const int li = a - 1;
        const long long pos = base + o;
        if (pos >= cap) continue;
        const int64_t j = s_lo[li] == NO_MATCH ? -1 : (int64_t)s_lo[li] + (o - s_excl[li]);
        write_out(L, kl, Rrest, nrest, l0 + li, j, outL, outR, pos);
    }
}

// ---- hash ---------------------------------------------------------------------

constexpr unsigned long long EMPTY = ~0ull;
constexpr int SMEM_SLOTS = 2048;

__device__ __forceinline__ unsigned long long hash_key(const Cols &K, int64_t r, int nk) {
    unsigned long long h = 0x9E3779B97F4A7C15ull;
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c) {
        if (c < nk) {
            h ^= (unsigned long long)(uint32_t)K.c[c][r];
            h *= 0xFF51AFD7ED558CCDull;
            h ^= h >> 33;
            h *= 0xC4CEB9FE1A85EC53ull;
            h ^= h >> 29;
        }
    }
    return h;
}

__device__ __forceinline__ unsigned long long make_entry(unsigned long long h, int64_t row) {
    return ((h >> 32) << 32) | (unsigned long long)(uint32_t)row;
}

__global__ void k_hash_build(Cols BK, int64_t nb, int nk, unsigned long long *__restrict__ slots,
                             uint32_t *__restrict__ cnt, uint32_t mask, int *__restrict__ err) {
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += (int64_t)gridDim.x * blockDim.x) {
        if (has_zero(BK, b, nk)) continue;
        const unsigned long long h = hash_key(BK, b, nk);
        const unsigned long long e = make_entry(h, b);
        uint32_t idx = (uint32_t)h & mask;
        bool done = false;
        for (uint32_t probe = 0; probe <= mask && !done; ++probe) {
            unsigned long long cur = slots[idx];
            if (cur == EMPTY) {
                const unsigned long long old = atomicCAS(slots + idx, EMPTY, e);
                if (old == EMPTY) {
                    atomicAdd(cnt + idx, 1u);
                    done = true;
                    break;
                }
                cur = old;
            }
            if ((cur >> 32) == (e >> 32) && cmp_rows(BK, (int64_t)(uint32_t)cur, BK, b, nk) == 0) {
                atomicAdd(cnt + idx, 1u);
                done = true;
                break;
            }
            idx = (idx + 1) & mask;
        }
        if (!done) atomicExch(err, TID_ERR_CAPACITY);
    }
}

// slot of B row b's key (its key was inserted); -1 if absent
__device__ __forceinline__ int64_t find_slot(const unsigned long long *slots, uint32_t mask, const Cols &BK,
                                             const Cols &QK, int64_t q, int nk, unsigned long long h) {
    uint32_t idx = (uint32_t)h & mask;
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        const unsigned long long cur = slots[idx];
        if (cur == EMPTY) return -1;
        if ((cur >> 32) == (h >> 32) && cmp_rows(BK, (int64_t)(uint32_t)cur, QK, q, nk) == 0) return idx;
        idx = (idx + 1) & mask;
    }
    return -1;
}

__global__ void k_hash_scatter(Cols BK, int64_t nb, int nk, const unsigned long long *__restrict__ slots,
                               uint32_t mask, const uint32_t *__restrict__ start, uint32_t *__restrict__ cursor,
                               int32_t *__restrict__ grouped) {
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += (int64_t)gridDim.x * blockDim.x) {
        if (has_zero(BK, b, nk)) continue;
        const int64_t s = find_slot(slots, mask, BK, BK, b, nk, hash_key(BK, b, nk));
        if (s < 0) continue;
        const uint32_t pos = start[s] + atomicAdd(cursor + s, 1u);
        grouped[pos] = (int32_t)b;
    }
}

template <bool SMEM>
__global__ void k_hash_count(Cols QK, int64_t nq, Cols BK, int nk, const unsigned long long *__restrict__ g_slots,
                             const uint32_t *__restrict__ g_cnt, const uint32_t *__restrict__ g_start, uint32_t mask,
                             uint32_t *__restrict__ cnt, uint32_t *__restrict__ qstart,
                             unsigned long long *__restrict__ total) {
    __shared__ unsigned long long s_slots[SMEM ? SMEM_SLOTS : 1];
    __shared__ uint32_t s_cnt[SMEM ? SMEM_SLOTS : 1], s_start[SMEM ? SMEM_SLOTS : 1];
    const unsigned long long *slots = g_slots;
    const uint32_t *scnt = g_cnt, *sstart = g_start;
    if (SMEM) {
        for (uint32_t i = threadIdx.x; i <= mask; i += blockDim.x) {
            s_slots[i] = g_slots[i];
            s_cnt[i] = g_cnt[i];
            s_start[i] = g_start[i];
        }
        __syncthreads();
        slots = s_slots;
        scnt = s_cnt;
        sstart = s_start;
    }
    // HC_U probe rows per thread per step, hashed first so that their key
    // loads are in flight together
    constexpr int HC_U = 4;
    unsigned long long acc = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * HC_U;
    for (int64_t q0 = (int64_t)blockIdx.x * blockDim.x * HC_U + threadIdx.x; q0 < nq; q0 += stride) {
        unsigned long long h[HC_U];
        bool z[HC_U];
#pragma unroll
        for (int u = 0; u < HC_U; ++u) {
            const int64_t q = min(q0 + (int64_t)u * blockDim.x, nq - 1);
            h[u] = hash_key(QK, q, nk);
            z[u] = has_zero(QK, q, nk);
        }
#pragma unroll
        for (int u = 0; u < HC_U; ++u) {
            const int64_t q = q0 + (int64_t)u * blockDim.x;
            if (q >= nq) break;
            uint32_t c = 0, st = 0;
            if (!z[u]) {
                const int64_t s = find_slot(slots, mask, BK, QK, q, nk, h[u]);
                if (s >= 0) {
                    c = scnt[s];
                    st = sstart[s];
                }
            }
            cnt[q] = c;
            qstart[q] = st;
            acc += c;
        }
    }
    block_add_u64(acc, total);  // once per warp: one address takes these atomics one at a time
}

struct Scratch {
    tid_ctx *ctx;
    std::vector<void *> ptrs;
    explicit Scratch(tid_ctx *c) : ctx(c) {}
    ~Scratch() {
        for (void *p : ptrs) dev_free(ctx, p);
    }
    template <class T>
    int get(T **p, size_t count) {
        void *q = nullptr;
        TID_TRY(dev_alloc(ctx, &q, count * sizeof(T) + 16));
        ptrs.push_back(q);
        *p = (T *)q;
        return TID_OK;
    }
};

int read_u64(tid_ctx *ctx, const unsigned long long *d, unsigned long long *h) {
    TID_TRY_CUDA(cudaMemcpyAsync(h, d, 8, cudaMemcpyDeviceToHost, ctx->stream), "read count");
    TID_TRY_CUDA(cudaStreamSynchronize(ctx->stream), "read count");
    return check_ctx_error(ctx);
}

}  // namespace

int join_sets(tid_ctx *ctx, const tid_set *L, const tid_set *R, int algo, tid_set **out, bool sorted_out) {
    *out = nullptr;
    if (algo & TID_JOIN_RIGHT) return outer_join_sets(ctx, L, R, algo, out);
    const bool left = (algo & TID_JOIN_LEFT) != 0;
    algo &= ~TID_JOIN_LEFT;
    int64_t nl = 0, nr = 0;
    TID_TRY(set_rows_host(L, &nl));
    TID_TRY(set_rows_host(R, &nr));
    // schema: shared variables, R's other columns
    int lkey[TID_MAX_COLS], rkey[TID_MAX_COLS], rrest[TID_MAX_COLS];
    int nk = 0, nrest = 0;
    for (int c = 0; c < L->k; ++c)
        for (int d = 0; d < R->k; ++d)
            if (L->vars[c] == R->vars[d]) {
                lkey[nk] = c;
                rkey[nk] = d;
                ++nk;
            }
    for (int d = 0; d < R->k; ++d) {
        bool shared = false;
        for (int c = 0; c < L->k; ++c) shared = shared || L->vars[c] == R->vars[d];
        if (!shared) rrest[nrest++] = d;
    }
    const int kout = L->k + nrest;
    if (kout > TID_MAX_COLS) return fail(TID_ERR_ARG, "tid_join: output would have %d columns", kout);
    int8_t ovars[TID_MAX_COLS];
    for (int c = 0; c < L->k; ++c) ovars[c] = L->vars[c];
    for (int c = 0; c < nrest; ++c) ovars[L->k + c] = R->vars[rrest[c]];
    if (algo != TID_JOIN_AUTO && algo != TID_JOIN_SORT_MERGE && algo != TID_JOIN_HASH)
        return fail(TID_ERR_ARG, "tid_join: unknown algorithm %d", algo);

    if (left && algo == TID_JOIN_HASH)
        return fail(TID_ERR_ARG, "tid_join: a left outer join runs as a sort-merge join");
    if (left && nl > 0 && nr == 0) {  // every left row, unbound on the right
        tid_set *e = nullptr;
        TID_TRY(set_alloc(ctx, kout, ovars, nl, &e));
        int rc = TID_OK;
        for (int c = 0; c < kout && rc == TID_OK; ++c) {
            cudaError_t ce = c < L->k ? cudaMemcpyAsync(e->col[c], L->col[c], (size_t)nl * 4, cudaMemcpyDeviceToDevice,
                                                        ctx->stream)
                                      : cudaMemsetAsync(e->col[c], 0, (size_t)nl * 4, ctx->stream);
            if (ce != cudaSuccess) rc = fail_cuda(ce, "tid_join: left rows");
        }
        e->bounded = L->bounded;
        for (int c = 0; c < kout; ++c) {
            e->lo[c] = c < L->k ? L->lo[c] : 0x80000000u;
            e->hi[c] = c < L->k ? L->hi[c] : 0x80000000u;
        }
        if (rc == TID_OK) rc = set_rows_const(e, nl);
        if (rc == TID_OK) rc = set_ready(e);
        if (rc != TID_OK) {
            set_free(e);
            return rc;
        }
        *out = e;
        return TID_OK;
    }
    if (nl == 0 || nr == 0) {
        tid_set *e = nullptr;
        TID_TRY(set_alloc(ctx, kout, ovars, 0, &e));
        int rc = set_rows_const(e, 0);
        if (rc == TID_OK) rc = set_ready(e);
        if (rc != TID_OK) {
            set_free(e);
            return rc;
        }
        *out = e;
        return TID_OK;
    }
    bool lprefix = true, rprefix = true;
    for (int i = 0; i < nk; ++i) {
        lprefix = lprefix && lkey[i] == i;
        rprefix = rprefix && rkey[i] == i;
    }
    // runs (or members, or a merge of two sorted sides) need the right side alone
    // to lead with the key; a sort of the joined rows is what the hash join costs
    // (8M x 8M rows, 11.5M joined, on GB300: 2318 us by hash and sort, 226 us by
    // runs, bound by the table lookups' and the right rows' random reads in L2)
    if (algo == TID_JOIN_AUTO) algo = (nk == 0 || rprefix) ? TID_JOIN_SORT_MERGE : TID_JOIN_HASH;
    if (nk == 0 || left) algo = TID_JOIN_SORT_MERGE;  // cross product; left outer join
    if (!sorted_out && (algo != TID_JOIN_HASH || nk == 0 || left))
        return fail(TID_ERR_ARG, "join: unsorted output is for inner hash joins");

    cudaStream_t st = ctx->stream;
    Bounds b{};  // output columns keep their input's bounds
    for (int c = 0; c < L->k; ++c) {
        b.lo[c] = L->lo[c];
        b.hi[c] = L->hi[c];
    }
    for (int c = 0; c < nrest; ++c) {
        b.lo[L->k + c] = left ? std::min(R->lo[rrest[c]], 0x80000000u) : R->lo[rrest[c]];  // 0 pads
        b.hi[L->k + c] = left ? std::max(R->hi[rrest[c]], 0x80000000u) : R->hi[rrest[c]];
    }
    const bool bounded = L->bounded && R->bounded;
    auto finish = [&](tid_set *res) {
        res->bounded = bounded;
        for (int c = 0; c < kout && bounded; ++c) {
            res->lo[c] = b.lo[c];
            res->hi[c] = b.hi[c];
        }
        *out = res;
        return TID_OK;
    };
    if (algo == TID_JOIN_SORT_MERGE && !left && nk == 1 && lprefix && rprefix && (L->k == 1 || R->k == 1)) {
        // members: Q's rows whose key is among B's terms.  Q is read once, so not
        // when B is so small that its searches of Q cost less (the bits of B's
        // range are cleared and set first: at most as many bytes as both sides).
        // 0.5M keys against 8.2M rows: 127 us by k_merge_join (dependent searches),
        // 70 us as a selection
        const bool b_is_l = L->k == 1 && (R->k > 1 || nl <= nr);
        const tid_set *B = b_is_l ? L : R, *Q = b_is_l ? R : L;
        const int64_t nb = b_is_l ? nl : nr, nq = b_is_l ? nr : nl;
        const uint64_t w = B->bounded ? (uint64_t)B->hi[0] - B->lo[0] + 1 : ~0ull;
        if (w <= (uint64_t)(32 * (nl + nr)) && w <= 0xFFFFFFFFull && (!b_is_l || nq <= 64 * nb)) {
            Members m{};
            TID_TRY(member_bits(ctx, B->col[0], nb, B->lo[0], B->hi[0], &m));
            tid_set *res = nullptr;
            int rc = set_alloc(ctx, kout, ovars, nq, &res);
            if (rc == TID_OK) rc = compact_member(ctx, Q, nq, m, res);
            dev_free(ctx, (void *)m.bits);
            if (rc == TID_OK) rc = set_ready(res);
            if (rc != TID_OK) {
                if (res) set_free(res);
                return rc;
            }
            return finish(res);
        }
    }
    if (sorted_out && algo == TID_JOIN_SORT_MERGE && nk > 0 && lprefix && rprefix && (L->k == nk || R->k == nk)) {
        // single pass into a result sized by the bound on its rows
        const int64_t ub = (L->k == nk ? nr : nl) + (left && L->k == nk ? nl : 0);
        tid_set *res = nullptr;
        TID_TRY(set_alloc(ctx, kout, ovars, ub, &res));
        Cols LK{}, RK{}, Lc{}, Rc{};
        for (int i = 0; i < nk; ++i) {
            LK.c[i] = L->col[i];
            RK.c[i] = R->col[i];
        }
        MCols oL{}, oR{};
        for (int c = 0; c < L->k; ++c) {
            Lc.c[c] = L->col[c];
            oL.c[c] = res->col[c];
        }
        for (int c = 0; c < nrest; ++c) {
            Rc.c[c] = R->col[rrest[c]];
            oR.c[c] = res->col[L->k + c];
        }
        const unsigned tiles = (unsigned)ceil_div(nl, (int64_t)MJ_TILE);
        Lookback lb{};
        int rc = lookback_scratch(ctx, tiles, &lb);
        if (rc == TID_OK) {
            k_merge_join<<<tiles, MJ_THREADS, 0, st>>>(LK, nl, RK, nr, nk, left, Lc, L->k, Rc, nrest, oL, oR,
                                                      res->cap, res->d_rows, res->slot.dev, lb);
            rc = launch_check("k_merge_join");
        }
        if (rc == TID_OK) rc = set_ready(res);
        if (rc != TID_OK) {
            set_free(res);
            return rc;
        }
        return finish(res);
    }
    Scratch s(ctx);
    Cols Lall{}, Rrest{};
    for (int c = 0; c < L->k; ++c) Lall.c[c] = L->col[c];
    for (int c = 0; c < nrest; ++c) Rrest.c[c] = R->col[rrest[c]];
    unsigned long long *d_total = nullptr;
    TID_TRY(s.get(&d_total, 1));
    TID_TRY_CUDA(cudaMemsetAsync(d_total, 0, 8, st), "memset");

    uint32_t *off = nullptr, *lo = nullptr;
    const int32_t *lperm = nullptr, *rperm = nullptr, *rmap = nullptr;
    int64_t n_probe = nl;
    bool left_is_probe = true;
    // The rows come out already canonical (sorted, distinct) when L is walked in its
    // order and each left row's matches in R's, which lead with the shared
    // variables: the output is ordered by L's columns, then by R's other columns.
    // A hash join does the same when both inputs lead with the shared variables and
    // its build side holds only these (at most one match per probe row, the
    // output ordered as the probe side).  Then no output sort.
    bool canonical_out = false;

    // a few left rows in key order search the right side faster than a table of it is built
    const bool runs = algo == TID_JOIN_SORT_MERGE && nk > 0 && rprefix && !(lprefix && nl <= nr / 64);
    if (runs) {
        Cols LK{}, RK{};
        for (int i = 0; i < nk; ++i) {
            LK.c[i] = L->col[lkey[i]];
            RK.c[i] = R->col[i];
        }
        RunTable t{};
        t.lo = R->bounded ? R->lo[0] : 0u;
        t.span = R->bounded ? R->hi[0] - R->lo[0] : 0xFFFFFFFFu;
        while (((uint64_t)t.span >> t.shift) + 1 > (uint64_t)std::max<int64_t>(nr, 1024)) ++t.shift;
        const size_t nb = (size_t)(t.span >> t.shift) + 1;
        uint32_t *cnt = nullptr;
        TID_TRY(s.get(&t.bucket, nb));
        TID_TRY(s.get(&cnt, nl));
        TID_TRY(s.get(&lo, nl));
        TID_TRY(s.get(&off, nl));
        TID_TRY_CUDA(cudaMemsetAsync(t.bucket, 0, nb * sizeof(uint2), st), "run table");
        k_run_table<<<grid_for(nr, 1024, 8), 256, 0, st>>>(RK.c[0], nr, t);
        TID_TRY(launch_check("k_run_table"));
        uint32_t *sums = nullptr;
        TID_TRY(s.get(&sums, (size_t)ceil_div(nl, (int64_t)SCAN_TILE)));
        k_run_count<<<(unsigned)ceil_div(nl, (int64_t)SCAN_TILE), 256, 0, st>>>(
            LK, nl, RK, nk, left, t, nk == 1 && t.shift == 0, cnt, lo, d_total, sums);
        TID_TRY(launch_check("k_run_count"));
        TID_TRY(scan_exclusive_u32(ctx, cnt, off, nl, nullptr, sums));
        canonical_out = true;
    } else if (algo == TID_JOIN_SORT_MERGE) {
        Cols LK{}, RK{};
        // left keys in key order
        if (lprefix) {
            for (int i = 0; i < nk; ++i) LK.c[i] = L->col[i];
        } else {
            int32_t *p = nullptr;
            TID_TRY(s.get(&p, nl));
            const int32_t *kc[TID_MAX_COLS];
            for (int i = 0; i < nk; ++i) kc[i] = L->col[lkey[i]];
            TID_TRY(sort_perm(ctx, kc, nk, nl, p));
            int32_t *g[TID_MAX_COLS];
            for (int i = 0; i < nk; ++i) TID_TRY(s.get(&g[i], nl));
            TID_TRY(gather_cols(ctx, kc, nk, p, nl, g));
            for (int i = 0; i < nk; ++i) LK.c[i] = g[i];
            lperm = p;
        }
        if (rprefix) {
            for (int i = 0; i < nk; ++i) RK.c[i] = R->col[i];
        } else {
            int32_t *p = nullptr;
            TID_TRY(s.get(&p, nr));
            const int32_t *kc[TID_MAX_COLS];
            for (int i = 0; i < nk; ++i) kc[i] = R->col[rkey[i]];
            TID_TRY(sort_perm(ctx, kc, nk, nr, p));
            int32_t *g[TID_MAX_COLS];
            for (int i = 0; i < nk; ++i) TID_TRY(s.get(&g[i], nr));
            TID_TRY(gather_cols(ctx, kc, nk, p, nr, g));
            for (int i = 0; i < nk; ++i) RK.c[i] = g[i];
            rperm = p;
        }
        uint32_t *cnt = nullptr;
        TID_TRY(s.get(&cnt, nl));
        TID_TRY(s.get(&lo, nl));
        TID_TRY(s.get(&off, nl));
        canonical_out = lprefix && rprefix;
        k_sm_count<<<grid_for(nl, 256), 256, 0, st>>>(LK, nl, RK, nr, nk, left, cnt, lo, d_total);
        TID_TRY(launch_check("k_sm_count"));
        TID_TRY(scan_exclusive_u32(ctx, cnt, off, nl, nullptr));
    } else {
        // build on the smaller side
        const bool build_left = nl < nr;
        const tid_set *B = build_left ? L : R;
        const tid_set *Q = build_left ? R : L;
        const int *bkey = build_left ? lkey : rkey;
        const int *qkey = build_left ? rkey : lkey;
        const int64_t nb = build_left ? nl : nr, nq = build_left ? nr : nl;
        Cols BK{}, QK{};
        for (int i = 0; i < nk; ++i) {
            BK.c[i] = B->col[bkey[i]];
            QK.c[i] = Q->col[qkey[i]];
        }
        uint32_t T = 64;
        while ((int64_t)T < 2 * nb) T <<= 1;
        const uint32_t mask = T - 1;
        unsigned long long *slots = nullptr;
        uint32_t *scnt = nullptr, *sstart = nullptr, *cursor = nullptr, *cnt = nullptr;
        int32_t *grouped = nullptr;
        TID_TRY(s.get(&slots, T));
        TID_TRY(s.get(&scnt, T));
        TID_TRY(s.get(&sstart, T));
        TID_TRY(s.get(&cursor, T));
        TID_TRY(s.get(&grouped, nb));
        TID_TRY_CUDA(cudaMemsetAsync(slots, 0xFF, (size_t)T * 8, st), "memset");
        TID_TRY_CUDA(cudaMemsetAsync(scnt, 0, (size_t)T * 4, st), "memset");
        TID_TRY_CUDA(cudaMemsetAsync(cursor, 0, (size_t)T * 4, st), "memset");
        k_hash_build<<<grid_for(nb, 256), 256, 0, st>>>(BK, nb, nk, slots, scnt, mask, ctx->err_dev);
        TID_TRY(launch_check("k_hash_build"));
        TID_TRY(scan_exclusive_u32(ctx, scnt, sstart, T, nullptr));
        k_hash_scatter<<<grid_for(nb, 256), 256, 0, st>>>(BK, nb, nk, slots, mask, sstart, cursor, grouped);
        TID_TRY(launch_check("k_hash_scatter"));
        TID_TRY(s.get(&cnt, nq));
        TID_TRY(s.get(&lo, nq));
        TID_TRY(s.get(&off, nq));
        if (T <= (uint32_t)SMEM_SLOTS)
            k_hash_count<true><<<grid_for(nq, 256 * 4), 256, 0, st>>>(QK, nq, BK, nk, slots, scnt, sstart, mask, cnt, lo, d_total);
        else
            k_hash_count<false><<<grid_for(nq, 256 * 4), 256, 0, st>>>(QK, nq, BK, nk, slots, scnt, sstart, mask, cnt, lo, d_total);
        TID_TRY(launch_check("k_hash_count"));
        TID_TRY(scan_exclusive_u32(ctx, cnt, off, nq, nullptr));
        rmap = grouped;
        n_probe = nq;
        left_is_probe = !build_left;
        canonical_out = (lprefix && rprefix && B->k == nk) || !sorted_out;
    }

    unsigned long long total = 0;
    TID_TRY(read_u64(ctx, d_total, &total));
    if (total > (unsigned long long)INT32_MAX)
        return fail(TID_ERR_CAPACITY, "tid_join: %llu output rows exceed 2^31-1", total);
    uint32_t *split = nullptr;
    const int64_t jtiles = ceil_div(n_probe + (int64_t)total, (int64_t)JW_TILE);
    if (total > 0) {
        TID_TRY(s.get(&split, jtiles + 1));
        k_join_split<<<(unsigned)ceil_div(jtiles + 1, (int64_t)8), 256, 0, st>>>(off, n_probe, (int64_t)total, jtiles,
                                                                                  split);
        TID_TRY(launch_check("k_join_split"));
    }
    if (canonical_out) {  // write straight into the result set
        tid_set *res = nullptr;
        TID_TRY(set_alloc(ctx, kout, ovars, (int64_t)total, &res));
        MCols oL{}, oR{};
        for (int c = 0; c < L->k; ++c) oL.c[c] = res->col[c];
        for (int c = 0; c < nrest; ++c) oR.c[c] = res->col[L->k + c];
        int rc = TID_OK;
        if (total > 0) {
            k_join_write<<<(unsigned)jtiles, JW_THREADS, 0, st>>>(
                off, n_probe, lo, lperm, rmap, rperm, (int64_t)total, Lall, L->k, Rrest, nrest, oL, oR, left_is_probe,
                split, res->d_rows, res->slot.dev);
            rc = launch_check("k_join_write");
        }
        if (rc == TID_OK && total == 0) rc = set_rows_const(res, 0);
        res->rows_known = (int64_t)total;
        if (rc == TID_OK) rc = set_ready(res);
        if (rc != TID_OK) {
            set_free(res);
            return rc;
        }
        return finish(res);
    }
    // write, then sort to canonical order
    MCols oc{}, oL{}, oR{};
    for (int c = 0; c < kout; ++c) TID_TRY(s.get(&oc.c[c], total > 0 ? total : 1));
    for (int c = 0; c < L->k; ++c) oL.c[c] = oc.c[c];
    for (int c = 0; c < nrest; ++c) oR.c[c] = oc.c[L->k + c];
    if (total > 0) {
        k_join_write<<<(unsigned)jtiles, JW_THREADS, 0, st>>>(
            off, n_probe, lo, lperm, rmap, rperm, (int64_t)total, Lall, L->k, Rrest, nrest, oL, oR, left_is_probe,
                split, nullptr, nullptr);
        TID_TRY(launch_check("k_join_write"));
    }
    const int32_t *ocols[TID_MAX_COLS];
    for (int c = 0; c < kout; ++c) ocols[c] = oc.c[c];
    return canonicalize(ctx, ocols, kout, ovars, (int64_t)total, false, bounded ? &b : nullptr, out);
}

}  // namespace tid
