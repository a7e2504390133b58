// Union of canonical sets by merging (Section 4.1's union of subquery results,
// with Section 4.3's distinct final values).
//
// Two canonical sets whose columns keep their relative order in the union
// schema (absent variables padded with 0, which never reorders rows) are
// each sorted in the union schema, so their union is a merge followed by
// dropping adjacent duplicates -- no sort.  Merge path (Odeh, Green, Mwassi,
// Shmueli and Birk, "Merge Path - Parallel Merging Made Simple", IPDPSW 2012):
//  * k_merge_split: for every tile boundary d, the number of A rows among the
//    first d merged rows, by a search along the cross diagonal (A before B on
//    equal rows), a warp per boundary testing 32 places at once;
//  * rows whose columns fit 64 bits together (the usual case; a variable that one
//    branch lacks takes one more value than the other holds, its 0, rather than
//    the range from 0 to it): k_merge_mark packs a tile's rows as it loads them, so
//    a row is one word of shared memory and a comparison one instruction; a thread
//    merges 16 rows along its own diagonal and leaves two bits per merged row: from
//    A or B, and different from its predecessor (mark of select.cuh);
//    k_merge_expand writes the kept rows, reading A and B once more in order;
//  * wider rows: k_merge_unique merges columns in shared memory, 8 rows per
//    thread, tile offsets from the decoupled look-back.
// Bytes: every input row read twice (the second time partly from L2), every
// distinct row written once.  Measured on GB300, 23.6M (x, v) with 8.2M (x, y):
// k_merge_split 26 -> 19 us (a warp per boundary instead of a thread), merging
// 583 us by k_merge_unique, 416 us packed with a look-back (a tile waited for
// its predecessors three times as long as it worked, at three CTAs per SM),
// 162 us by k_merge_mark and 135 us by k_merge_expand.  Bound: the mark's
// shared-memory steps; the expansion's reads.

#include <algorithm>

#include "lookback.cuh"
#include "ops.cuh"
#include "select.cuh"

namespace tid {

namespace {

constexpr int MG_THREADS = 256;
constexpr int MG_WARPS = MG_THREADS / 32;
constexpr int MG_ITEMS = 8;
constexpr int MG_TILE = MG_THREADS * MG_ITEMS;  // merged rows per tile

struct PadCols {  // a set's columns in union-schema order; null = absent (reads as 0)
    const int32_t *c[TID_MAX_COLS];
};

__device__ __forceinline__ int32_t pval(const PadCols &A, int c, int64_t i) { return A.c[c] ? A.c[c][i] : 0; }

// a row of A vs a row of B: -1, 0, 1 in lexicographic int32 order (column loops
// run to TID_MAX_COLS with a guard so the pointers stay in registers)
__device__ __forceinline__ int cmp_pad(const PadCols &A, int64_t i, const PadCols &B, int64_t j, int nu) {
    int r = 0;
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c) {
        if (c < nu && r == 0) {
            const int32_t x = pval(A, c, i), y = pval(B, c, j);
            r = x == y ? 0 : (x < y ? -1 : 1);
        }
    }
    return r;
}

// A rows among the first d merged rows (a warp's search): A[mid] precedes
// B[d - 1 - mid] for every mid below the answer and for none from it on.
__device__ __forceinline__ int64_t warp_split(const PadCols &A, int64_t na, const PadCols &B, int64_t nb, int nu,
                                              int64_t d) {
    const unsigned lane = threadIdx.x & 31;
    int64_t lo = max((int64_t)0, d - nb), hi = min(d, na);
    while (lo < hi) {  // lane l tests the end of the l-th of 32 equal parts
        const int64_t part = (hi - lo + 31) / 32, mid = lo + (lane + 1) * part - 1;
        const bool below = mid < hi && cmp_pad(A, mid, B, d - 1 - mid, nu) <= 0;
        const int full = __popc(__ballot_sync(0xffffffffu, below));  // parts wholly below the answer
        lo += (int64_t)full * part;
        hi = min(hi, lo + part - 1);
    }
    return min(lo, min(d, na));
}

// Warp t: split[t] for the boundary before tile t (t <= tiles)
__global__ void __launch_bounds__(256) k_merge_split(PadCols A, int64_t na, PadCols B, int64_t nb, int nu, int64_t tiles,
                                                     int tile_rows, int64_t *__restrict__ split) {
    const int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (t > tiles) return;
    const int64_t s = warp_split(A, na, B, nb, nu, min(t * tile_rows, na + nb));
    if ((threadIdx.x & 31) == 0) split[t] = s;
}

typedef unsigned long long u64;

constexpr int MP_THREADS = 256;
// Merged rows per thread: 16, or 4 where 16 would leave SMs without a tile (a tile's
// time is then its chain of loads, search and merge steps).
template <int ITEMS>
constexpr int mp_tile() {
    return MP_THREADS * ITEMS;
}

// One column's field of a packed row; zero: 0 is the field 0 and the values from
// min + 1 (sort order) up follow it.
__device__ __forceinline__ u64 pack_field(const MergePack &mp, int c, int32_t x) {
    const uint32_t f = ((mp.zero >> c) & 1u) && x == 0 ? 0u : ((uint32_t)x ^ 0x80000000u) - mp.ps.min[c];
    return (u64)f << mp.ps.shift[c];
}
__device__ __forceinline__ u64 pack_one(const MergePack &mp, const PadCols &A, int nu, int64_t i) {
    u64 key = 0;
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c)
        if (c < nu && mp.ps.mask[c]) key |= pack_field(mp, c, pval(A, c, i));
    return key;
}

// Merged rows: the selection's scratch, and per step the bits "from A" (32 words)
// and the first A row.
struct MergeBits {
    SelScratch sc;
    uint32_t *take;
    uint32_t *first_a;
};

template <int MP_ITEMS>
__global__ void __launch_bounds__(MP_THREADS, 4)
k_merge_mark(PadCols A, int64_t na, PadCols B, int64_t nb, int nu, MergePack mp, const int64_t *__restrict__ split,
             MergeBits mb, int64_t *__restrict__ d_rows, int64_t *__restrict__ h_rows) {
    constexpr int MP_TILE = mp_tile<MP_ITEMS>();
    constexpr int STEP_THREADS = SEL_STEP / MP_ITEMS;  // threads whose rows make a step
    constexpr int WORD_THREADS = 32 / MP_ITEMS;        // and a word
    __shared__ u64 s_key[MP_TILE];
    __shared__ u64 s_before;  // the merged row before the tile
    __shared__ int64_t s_split[2];
    __shared__ unsigned s_cnt[MP_THREADS / 32];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tile = blockIdx.x;
    const int64_t d0 = tile * MP_TILE, d1 = min(d0 + MP_TILE, na + nb);
    if (!split) {  // a few tiles: their own searches cost less than a launch for them
        if (warp < 2) {
            const int64_t s = warp_split(A, na, B, nb, nu, warp == 0 ? d0 : d1);
            if (lane == 0) s_split[warp] = s;
        }
        __syncthreads();
    }
    const int64_t a0 = split ? split[tile] : s_split[0], a1 = split ? split[tile + 1] : s_split[1], b0 = d0 - a0;
    const int la = (int)(a1 - a0), len = (int)(d1 - d0);
    {  // pack the tile's rows, A's first
        u64 k[MP_ITEMS];
#pragma unroll
        for (int q = 0; q < MP_ITEMS; ++q) k[q] = 0;
#pragma unroll
        for (int c = 0; c < TID_MAX_COLS; ++c) {
            if (c >= nu) break;
            if (!mp.ps.mask[c]) continue;
            int32_t x[MP_ITEMS];
#pragma unroll
            for (int q = 0; q < MP_ITEMS; ++q) {
                const int r = q * MP_THREADS + threadIdx.x;
                x[q] = 0;
                if (r < la) {
                    if (A.c[c]) x[q] = A.c[c][a0 + r];
                } else if (r < len) {
                    if (B.c[c]) x[q] = B.c[c][b0 + (r - la)];
                }
            }
#pragma unroll
            for (int q = 0; q < MP_ITEMS; ++q) k[q] |= pack_field(mp, c, x[q]);
        }
#pragma unroll
        for (int q = 0; q < MP_ITEMS; ++q) {
            const int r = q * MP_THREADS + threadIdx.x;
            if (r < len) s_key[r] = k[q];
        }
    }
    if (threadIdx.x == 0 && d0 > 0) {
        u64 v = 0;
        if (a0 > 0) v = pack_one(mp, A, nu, a0 - 1);
        if (b0 > 0) v = max(v, pack_one(mp, B, nu, b0 - 1));
        s_before = v;
    }
    __syncthreads();
    // this thread's diagonal: local merged rows [dt, dt + MP_ITEMS)
    const int dt = min((int)threadIdx.x * MP_ITEMS, len), lb_ = len - la;
    int lo = max(0, dt - lb_), hi = min(dt, la);
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (s_key[mid] <= s_key[la + dt - 1 - mid]) lo = mid + 1;
        else hi = mid;
    }
    int i = lo, j = la + dt - lo;  // next A row, next B row
    // the merged row before the diagonal: the larger of the two before it
    u64 prev = 0;
    bool has_prev = true;
    if (i > 0) prev = s_key[i - 1];
    if (j > la) prev = max(prev, s_key[j - 1]);
    if (i == 0 && j == la) {  // the tile's first row
        has_prev = d0 > 0;
        prev = has_prev ? s_before : 0;
    }
    const int64_t step = tile * (MP_TILE / SEL_STEP) + threadIdx.x / STEP_THREADS;
    if (threadIdx.x % STEP_THREADS == 0 && step < mb.sc.steps) mb.first_a[step] = (uint32_t)(a0 + i);
    u64 ka = i < la ? s_key[i] : 0, kb = j < len ? s_key[j] : 0;
    unsigned keep = 0, take = 0;
#pragma unroll
    for (int e = 0; e < MP_ITEMS; ++e) {
        if (dt + e >= len) break;
        const bool take_a = j >= len || (i < la && ka <= kb);
        const u64 v = take_a ? ka : kb;
        if (!has_prev || v != prev) keep |= 1u << e;
        has_prev = true;
        prev = v;
        if (take_a) {
            take |= 1u << e;
            ++i;
            ka = i < la ? s_key[i] : 0;
        } else {
            ++j;
            kb = j < len ? s_key[j] : 0;
        }
    }
    const unsigned c = __reduce_add_sync(0xffffffffu, __popc(keep));
    keep <<= MP_ITEMS * (lane % WORD_THREADS);
    take <<= MP_ITEMS * (lane % WORD_THREADS);
#pragma unroll
    for (int d = 1; d < WORD_THREADS; d <<= 1) {
        keep |= __shfl_xor_sync(0xffffffffu, keep, d);
        take |= __shfl_xor_sync(0xffffffffu, take, d);
    }
    if (lane % WORD_THREADS == 0 && step < mb.sc.steps) {
        const size_t w = (size_t)step * 32 + (threadIdx.x % STEP_THREADS) / WORD_THREADS;
        mb.sc.bits[w] = keep;
        mb.take[w] = take;
    }
    if (lane == 0) s_cnt[warp] = c;
    __syncthreads();
    if (threadIdx.x % STEP_THREADS == 0 && step < mb.sc.steps) {
        unsigned n = 0;
        for (int w = 0; w < STEP_THREADS / 32; ++w) n += s_cnt[warp + w];
        mb.sc.cnt[step] = n;
    }
    sel_finish(mb.sc, c, d_rows, h_rows);
}

template <int K>
__global__ void __launch_bounds__(SEL_THREADS, K <= 3 ? 4 : 2)
k_merge_expand(PadCols A, PadCols B, int nu, MergeBits mb, OutCols out, int64_t cap) {
    const unsigned lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
    constexpr int UX = 4;  // rows per lane read together
    // a range is four steps or one, a step per warp: two or eight ranges per CTA
    const unsigned warp = threadIdx.x >> 5, per = mb.sc.per;
    const unsigned range = blockIdx.x * (SEL_WARPS / per) + warp / per;
    if (range >= mb.sc.ranges) return;
    sel_walk(mb.sc, range, warp % per, per, [&](unsigned step, uint32_t word, unsigned xo, unsigned, unsigned long long o0) {
        const uint32_t take = mb.take[(size_t)step * 32 + lane];
        const unsigned pc = __popc(take);
        unsigned tx = pc;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, tx, d);
            if ((int)lane >= d) tx += y;
        }
        tx -= pc;
        const uint32_t as = mb.first_a[step], bs = step * SEL_STEP - as;
#pragma unroll 1
        for (int w0 = 0; w0 < 32; w0 += UX) {
            int32_t v[UX][K];
            unsigned bw[UX];
#pragma unroll
            for (int u = 0; u < UX; ++u) {
                const int w = w0 + u;
                bw[u] = __shfl_sync(0xffffffffu, word, w);
                const uint32_t tw = __shfl_sync(0xffffffffu, take, w), at = __shfl_sync(0xffffffffu, tx, w);
                const bool from_a = (tw >> lane) & 1u;
                const uint32_t r = from_a ? as + at + __popc(tw & lt) : bs + (w * 32 - at) + __popc(~tw & lt);
                if ((bw[u] >> lane) & 1u) {
#pragma unroll
                    for (int c = 0; c < K; ++c) {
                        if (c >= nu) break;
                        const int32_t *p = from_a ? A.c[c] : B.c[c];
                        v[u][c] = p ? p[r] : 0;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < UX; ++u) {
                const unsigned long long pos = o0 + __shfl_sync(0xffffffffu, xo, w0 + u) + __popc(bw[u] & lt);
                if (((bw[u] >> lane) & 1u) && pos < (unsigned long long)cap) {
#pragma unroll
                    for (int c = 0; c < K; ++c)
                        if (c < nu) out.col[c][pos] = v[u][c];
                }
            }
        }
    });
}

// shared-memory rows: column c of local row r at s_rows[c * (MG_TILE + 1) + r];
// rows [0, la) are A's, [la, la + lb) B's, row MG_TILE the tile's predecessor
__device__ __forceinline__ bool rows_equal(const int32_t *s_rows, int nu, int r1, int r2) {
    bool eq = true;
    for (int c = 0; c < nu; ++c) eq = eq && s_rows[c * (MG_TILE + 1) + r1] == s_rows[c * (MG_TILE + 1) + r2];
    return eq;
}

__device__ __forceinline__ int cmp_local(const int32_t *s_rows, int nu, int r1, int r2) {
    for (int c = 0; c < nu; ++c) {
        const int32_t x = s_rows[c * (MG_TILE + 1) + r1], y = s_rows[c * (MG_TILE + 1) + r2];
        if (x != y) return x < y ? -1 : 1;
    }
    return 0;
}

__global__ void __launch_bounds__(MG_THREADS)
k_merge_unique(PadCols A, int64_t na, PadCols B, int64_t nb, int nu, const int64_t *__restrict__ split, OutCols out,
               int64_t cap, int64_t *__restrict__ d_rows, int64_t *__restrict__ h_rows, Lookback lb) {
    extern __shared__ int32_t s_rows[];  // nu x (MG_TILE + 1)
    __shared__ uint16_t s_order[MG_TILE];
    __shared__ unsigned s_off[MG_ITEMS * MG_WARPS];
    __shared__ unsigned s_tile;
    __shared__ long long s_prefix;
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = lb_ticket(lb);
    __syncthreads();
    const unsigned tile = s_tile;
    if (tile >= lb.num_tiles) return;
    const int64_t d0 = (int64_t)tile * MG_TILE;
    const int64_t d1 = min(d0 + MG_TILE, na + nb);
    const int64_t a0 = split[tile], a1 = split[tile + 1];
    const int64_t b0 = d0 - a0, b1 = d1 - a1;
    const int la = (int)(a1 - a0), lb_ = (int)(b1 - b0), len = la + lb_;
#pragma unroll
    for (int c = 0; c < TID_MAX_COLS; ++c) {
        if (c >= nu) continue;
        int32_t *col = s_rows + c * (MG_TILE + 1);
        for (int r = threadIdx.x; r < len; r += MG_THREADS)
            col[r] = r < la ? pval(A, c, a0 + r) : pval(B, c, b0 + (r - la));
    }
    // the merged row before the tile: the later (larger) of A[a0 - 1] and B[b0 - 1]
    if (threadIdx.x == 0 && d0 > 0) {
        const bool from_b = a0 == 0 || (b0 > 0 && cmp_pad(A, a0 - 1, B, b0 - 1, nu) <= 0);
#pragma unroll
        for (int c = 0; c < TID_MAX_COLS; ++c)
            if (c < nu) s_rows[c * (MG_TILE + 1) + MG_TILE] = from_b ? pval(B, c, b0 - 1) : pval(A, c, a0 - 1);
    }
    __syncthreads();
    // this thread's diagonal: local merged rows [dt, dt + 8)
    const int dt = min((int)threadIdx.x * MG_ITEMS, len);
    int lo = max(0, dt - lb_), hi = min(dt, la);
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (cmp_local(s_rows, nu, mid, la + dt - 1 - mid) <= 0) lo = mid + 1;
        else hi = mid;
    }
    int i = lo, j = dt - lo;  // next A row, next B row (local)
    for (int e = 0; e < MG_ITEMS && dt + e < len; ++e) {
        const bool take_a = j >= lb_ || (i < la && cmp_local(s_rows, nu, i, la + j) <= 0);
        s_order[dt + e] = (uint16_t)(take_a ? i++ : la + j++);
    }
    __syncthreads();
    // striped: drop a row equal to its predecessor in merged order
    const unsigned lt = (1u << lane) - 1u;
    unsigned keep = 0, wpre[MG_ITEMS];
#pragma unroll
    for (int q = 0; q < MG_ITEMS; ++q) {
        const int p = q * MG_THREADS + threadIdx.x;
        bool kp = false;
        if (p < len) {
            const int prev = p > 0 ? s_order[p - 1] : MG_TILE;
            kp = (d0 + p == 0) || !rows_equal(s_rows, nu, s_order[p], prev);
        }
        keep |= (unsigned)kp << q;
        const unsigned b = __ballot_sync(0xffffffffu, kp);
        wpre[q] = __popc(b & lt);
        if (lane == 0) s_off[q * MG_WARPS + warp] = __popc(b);
    }
    __syncthreads();
    if (warp == 0) {
        const unsigned x0 = s_off[2 * lane], x1 = s_off[2 * lane + 1];
        unsigned x = x0 + x1;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, d);
            if ((int)lane >= d) x += y;
        }
        const unsigned ex = x - x0 - x1;
        s_off[2 * lane] = ex;
        s_off[2 * lane + 1] = ex + x0;
        const unsigned total = __shfl_sync(0xffffffffu, x, 31);
        const long long excl = lb_exclusive_prefix(lb, tile, total);
        if (lane == 0) {
            s_prefix = excl;
            if (tile == lb.num_tiles - 1 && excl >= 0) {
                *d_rows = excl + total;
                *h_rows = excl + total;
            }
        }
    }
    __syncthreads();
    const long long prefix = s_prefix;
    if (prefix < 0) return;
#pragma unroll
    for (int q = 0; q < MG_ITEMS; ++q) {
        if (!((keep >> q) & 1u)) continue;
        const int p = q * MG_THREADS + threadIdx.x;
        const long long pos = prefix + s_off[q * MG_WARPS + warp] + wpre[q];
        if (pos >= cap) continue;
        const int r = s_order[p];
#pragma unroll
        for (int c = 0; c < TID_MAX_COLS; ++c)
            if (c < nu) out.col[c][pos] = s_rows[c * (MG_TILE + 1) + r];
    }
}

struct Scratch {
    tid_ctx *ctx;
    void *p = nullptr;
    explicit Scratch(tid_ctx *c) : ctx(c) {}
    ~Scratch() {
        if (p) dev_free(ctx, p);
    }
};

}  // namespace

int merge_unique(tid_ctx *ctx, const int32_t *const *acols, int64_t na, const int32_t *const *bcols, int64_t nb,
                 int nu, const MergePack *mp, tid_set *out) {
    if (nu < 1 || nu > TID_MAX_COLS) return fail(TID_ERR_ARG, "merge: %d columns", nu);
    cudaStream_t st = ctx->stream;
    if (na + nb == 0) return set_rows_const(out, 0);
    if (nb == 0) {  // one sorted side with all its columns: its distinct rows
        bool all = true;
        for (int c = 0; c < nu; ++c) all = all && acols[c];
        if (all) return compact_unique(ctx, acols, nu, nullptr, na, out);
    }
    PadCols A{}, B{};
    for (int c = 0; c < nu; ++c) {
        A.c[c] = acols[c];
        B.c[c] = bcols[c];
    }
    OutCols oc{};
    for (int c = 0; c < nu; ++c) oc.col[c] = out->col[c];
    const bool few = na + nb < (int64_t)sm_count() * 2 * mp_tile<16>();
    const int tile_rows = !mp ? MG_TILE : few ? mp_tile<4>() : mp_tile<16>();
    const int64_t tiles = ceil_div(na + nb, (int64_t)tile_rows);
    Scratch s(ctx);
    int64_t *split = nullptr;
    if (!mp || !few) {
        TID_TRY(dev_alloc(ctx, &s.p, sizeof(int64_t) * (tiles + 1)));
        split = (int64_t *)s.p;
        k_merge_split<<<(unsigned)ceil_div(tiles + 1, 8), 256, 0, st>>>(A, na, B, nb, nu, tiles, tile_rows, split);
        TID_TRY(launch_check("k_merge_split"));
    }
    if (mp) {
        MergeBits mb{};
        const size_t steps = (size_t)ceil_div(na + nb, (int64_t)SEL_STEP);
        void *blk = nullptr, *extra = nullptr;
        TID_TRY(sel_scratch(ctx, na + nb, 1, steps * 33 * 4, &mb.sc, &blk, &extra, tile_rows / SEL_STEP));
        mb.take = (uint32_t *)extra;
        mb.first_a = mb.take + steps * 32;
        if (few)
            k_merge_mark<4><<<(unsigned)tiles, MP_THREADS, 0, st>>>(A, na, B, nb, nu, *mp, split, mb, out->d_rows,
                                                                   out->slot.dev);
        else
            k_merge_mark<16><<<(unsigned)tiles, MP_THREADS, 0, st>>>(A, na, B, nb, nu, *mp, split, mb, out->d_rows,
                                                                    out->slot.dev);
        int rc = launch_check("k_merge_mark");
        if (rc == TID_OK) {
            const unsigned grid = (unsigned)ceil_div(mb.sc.ranges, (int64_t)(SEL_WARPS / mb.sc.per));
            if (nu <= 3) k_merge_expand<3><<<grid, SEL_THREADS, 0, st>>>(A, B, nu, mb, oc, out->cap);
            else k_merge_expand<TID_MAX_COLS><<<grid, SEL_THREADS, 0, st>>>(A, B, nu, mb, oc, out->cap);
            rc = launch_check("k_merge_expand");
        }
        dev_free(ctx, blk);
        return rc;
    }
    Lookback lb{};
    TID_TRY(lookback_scratch(ctx, (unsigned)tiles, &lb));
    const size_t smem = sizeof(int32_t) * nu * (MG_TILE + 1);
    static bool opted = false;
    if (!opted) {
        TID_TRY_CUDA(cudaFuncSetAttribute(k_merge_unique, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)(sizeof(int32_t) * TID_MAX_COLS * (MG_TILE + 1))),
                     "k_merge_unique smem");
        opted = true;
    }
    k_merge_unique<<<(unsigned)tiles, MG_THREADS, smem, st>>>(A, na, B, nb, nu, split, oc, out->cap, out->d_rows,
                                                              out->slot.dev, lb);
    return launch_check("k_merge_unique");
}

}  // namespace tid
