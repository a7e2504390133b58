// K2: several triple patterns in one pass over the store.
//
// Section 4.1 extends the search to a key array holding the keys of all
// subqueries: every triple is compared with each key and marked with the list
// of subqueries it answers (a triple may answer several, as in the paper's
// second union example).  Here the marks become one ascending index list per
// pattern by mark and expand (select.cuh): k2_mark loads the union of the
// patterns' bound columns once per step and tests every pattern on the loaded
// values, leaving one hit bit per triple and pattern; k_scan_ranges scans each
// pattern's range totals; k2_expand writes the lists.
// Bytes per launch: 4 * |union of bound columns| * n read + 4 * sum of hits written
// (+ n/8 per pattern of bitmap written and read, mostly in L2).  Measured on GB300,
// three patterns over two columns of 200M triples, 32.3M hits: k2_mark 251 us
// (6.4 TB/s), k_scan_ranges 12 us, k2_expand 95 us; before, chunks in shared memory
// with one look-back chain per pattern took 483 us, and 88 us at 1M triples, where
// they gave four CTAs work.

#include <algorithm>

#include "select.cuh"

namespace tid {

namespace {

struct MultiArgs {
    int m;
    int32_t key[TID_MAX_MULTI][3];
    int32_t *out[TID_MAX_MULTI];
    int64_t cap[TID_MAX_MULTI];
    int64_t *d_rows[TID_MAX_MULTI];
    int64_t *h_rows[TID_MAX_MULTI];
};

// list j's part of the scratch of several lists
__device__ __forceinline__ SelScratch list_of(const SelScratch &all, int j) {
    SelScratch sc = all;
    sc.bits += (size_t)j * all.steps * 32;
    sc.cnt += (size_t)j * all.steps;
    sc.tot += (size_t)j * all.ranges;
    sc.off += (size_t)j * all.ranges;
    return sc;
}

template <int U, bool VEC>
__global__ void __launch_bounds__(SEL_THREADS)
k2_mark(const int32_t *__restrict__ S, const int32_t *__restrict__ P, const int32_t *__restrict__ O, int64_t n,
        const __grid_constant__ MultiArgs args, SelScratch sc) {
    __shared__ unsigned s_kept[TID_MAX_MULTI][SEL_WARPS];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned r0 = blockIdx.x * sc.per, r1 = min(r0 + sc.per, sc.steps);
    const int m = args.m;
    for (int j = (int)lane; j < m; j += 32) s_kept[j][warp] = 0;
    __syncwarp();
    for (unsigned step = r0 + warp; step < r1; step += SEL_WARPS) {
        int4 v[3][8];
        load_step<U, VEC>(S, P, O, n, step, v);
        // triples past n: a pattern binds at least one column of U or none at all
        // (then it matches every triple of the store, and only those)
        const int64_t left = n - ((int64_t)step * SEL_STEP + lane * 4);
#pragma unroll 1
        for (int j = 0; j < m; ++j) {
            const int32_t ks = args.key[j][0], kp = args.key[j][1], ko = args.key[j][2];
            unsigned k4[8], any = 0;
#pragma unroll
            for (int g = 0; g < 8; ++g) k4[g] = 0xFu;
            if ((U & 1) && ks) {
#pragma unroll
                for (int g = 0; g < 8; ++g) k4[g] &= eq4(v[0][g], ks);
            }
            if ((U & 2) && kp) {
#pragma unroll
                for (int g = 0; g < 8; ++g) k4[g] &= eq4(v[1][g], kp);
            }
            if ((U & 4) && ko) {
#pragma unroll
                for (int g = 0; g < 8; ++g) k4[g] &= eq4(v[2][g], ko);
            }
            if ((ks | kp | ko) == 0 && (int64_t)(step + 1) * SEL_STEP > n) {
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    const int64_t l = left - g * 128;
                    k4[g] = l >= 4 ? 0xFu : (l <= 0 ? 0u : (1u << l) - 1u);
                }
            }
#pragma unroll
            for (int g = 0; g < 8; ++g) any |= k4[g];
            unsigned c = 0;
            if (__any_sync(0xffffffffu, any)) {  // a step without a hit writes its count alone
                const uint32_t word = sel_word(k4);
                __stcg(sc.bits + ((size_t)j * sc.steps + step) * 32 + sel_word_index(), word);
                c = __reduce_add_sync(0xffffffffu, __popc(word));
            }
            if (lane == 0) {
                __stcg(sc.cnt + (size_t)j * sc.steps + step, c);
                s_kept[j][warp] += c;
            }
        }
    }
    __syncthreads();
    if ((int)threadIdx.x < m) {
        unsigned t = 0;
        for (int w = 0; w < SEL_WARPS; ++w) t += s_kept[threadIdx.x][w];
        sc.tot[(size_t)threadIdx.x * sc.ranges + blockIdx.x] = t;
    }
}

// CTA j: the first output row of each of list j's ranges, and its row count
__global__ void __launch_bounds__(SEL_THREADS) k_scan_ranges(const __grid_constant__ MultiArgs args, SelScratch all) {
    const SelScratch sc = list_of(all, blockIdx.x);
    const unsigned long long n = sel_scan_totals(sc.tot, sc.off, sc.ranges);
    if (threadIdx.x == 0) {
        *args.d_rows[blockIdx.x] = (int64_t)n;
        *args.h_rows[blockIdx.x] = (int64_t)n;
    }
}

__global__ void __launch_bounds__(SEL_THREADS) k2_expand(const __grid_constant__ MultiArgs args, SelScratch all) {
    const SelScratch sc = list_of(all, blockIdx.y);
    sel_expand_index(sc, args.out[blockIdx.y], args.cap[blockIdx.y]);
}

template <int U>
int launch_vec(bool vec, tid_ctx *ctx, const int32_t *S, const int32_t *P, const int32_t *O, int64_t n,
               const MultiArgs &a) {
    SelScratch sc{};
    void *blk = nullptr;
    TID_TRY(sel_scratch(ctx, n, a.m, 0, &sc, &blk, nullptr));
    cudaStream_t st = ctx->stream;
    if (vec) k2_mark<U, true><<<sc.ranges, SEL_THREADS, 0, st>>>(S, P, O, n, a, sc);
    else k2_mark<U, false><<<sc.ranges, SEL_THREADS, 0, st>>>(S, P, O, n, a, sc);
    int rc = launch_check("k2_mark");
    if (rc == TID_OK) {
        k_scan_ranges<<<a.m, SEL_THREADS, 0, st>>>(a, sc);
        rc = launch_check("k_scan_ranges");
    }
    if (rc == TID_OK) {
        k2_expand<<<dim3(sel_index_grid(sc), a.m), SEL_THREADS, 0, st>>>(a, sc);
        rc = launch_check("k2_expand");
    }
    dev_free(ctx, blk);
    return rc;
}

}  // namespace

}  // namespace tid

using namespace tid;

extern "C" int tid_match_multi(tid_ctx *ctx, const tid_store *st, const tid_pattern *pats, int m, tid_set **outs) {
    clear_error();
    tid::Range nvtx_range("tid_match_multi");
    if (!ctx || !st || !pats || !outs) return fail(TID_ERR_ARG, "tid_match_multi: null argument");
    if (m < 1 || m > TID_MAX_MULTI) return fail(TID_ERR_ARG, "tid_match_multi: m = %d (1..%d)", m, TID_MAX_MULTI);
    if (st->ctx != ctx) return fail(TID_ERR_ARG, "tid_match_multi: store belongs to another context");
    for (int j = 0; j < m; ++j) {
        outs[j] = nullptr;
        if (pats[j].s < 0 || pats[j].p < 0 || pats[j].o < 0)
            return fail(TID_ERR_ID, "tid_match_multi: negative ID in pattern %d", j);
    }
    CallGuard g(ctx);
    const int64_t n = st->n;
    int U = 0;
    for (int j = 0; j < m; ++j) U |= (pats[j].s != 0) | ((pats[j].p != 0) << 1) | ((pats[j].o != 0) << 2);
    MultiArgs a{};
    a.m = m;
    int rc = TID_OK;
    const int8_t var = -1;
    for (int j = 0; j < m && rc == TID_OK; ++j) {
        rc = set_alloc(ctx, 1, &var, n, &outs[j]);
        if (rc != TID_OK) break;
        a.key[j][0] = pats[j].s;
        a.key[j][1] = pats[j].p;
        a.key[j][2] = pats[j].o;
        a.out[j] = outs[j]->col[0];
        a.cap[j] = outs[j]->cap;
        a.d_rows[j] = outs[j]->d_rows;
        a.h_rows[j] = outs[j]->slot.dev;
    }
    if (rc == TID_OK) {
        if (n == 0 || U == 0) {
            // nothing bound anywhere: every list is 0..n-1 (tid_match handles it)
            for (int j = 0; j < m && rc == TID_OK; ++j) {
                LbScratch none{};
                rc = launch_match(ctx->stream, st->s, st->p, st->o, n, st->aligned16, 0, 0, 0, outs[j]->col[0],
                                  outs[j]->cap, outs[j]->d_rows, outs[j]->slot.dev, none);
            }
        } else {
            const bool v = st->aligned16;
            switch (U) {
                case 1: rc = launch_vec<1>(v, ctx, st->s, st->p, st->o, n, a); break;
                case 2: rc = launch_vec<2>(v, ctx, st->s, st->p, st->o, n, a); break;
                case 3: rc = launch_vec<3>(v, ctx, st->s, st->p, st->o, n, a); break;
                case 4: rc = launch_vec<4>(v, ctx, st->s, st->p, st->o, n, a); break;
                case 5: rc = launch_vec<5>(v, ctx, st->s, st->p, st->o, n, a); break;
                case 6: rc = launch_vec<6>(v, ctx, st->s, st->p, st->o, n, a); break;
                default: rc = launch_vec<7>(v, ctx, st->s, st->p, st->o, n, a); break;
            }
        }
    }
    for (int j = 0; j < m && rc == TID_OK; ++j) rc = set_ready(outs[j]);
    if (rc != TID_OK) {
        for (int j = 0; j < m; ++j) {
            set_free(outs[j]);
            outs[j] = nullptr;
        }
    }
    return rc;
}
