// Device side of "mark and expand": a kernel tests every row of a long input and
// leaves one keep bit per row (mark), the next one writes the kept rows, in order
// (expand).  Used by the searches (match.cu, multi.cu) and by the row selections
// of the tuple-set operators (compact.cu).
//
// The rows go in steps of 1024, one warp at a time; a CTA owns a range of steps.
// It leaves the steps' keep words and counts and its range's total; the totals
// are scanned (by the last CTA of the mark kernel, or by k_scan_ranges for several
// lists), which gives every range its first output row.  No CTA waits for another.
// A CTA per range rather than a resident grid: the hardware hands out the ranges
// as SMs come free, and SMs stream at different speeds.
#pragma once

#include "tid_internal.cuh"

namespace tid {

constexpr int SEL_THREADS = 256;
constexpr int SEL_WARPS = SEL_THREADS / 32;
constexpr int SEL_STEP = 1024;         // rows per step
// Kept rows from which a step is written word by word (32 rounds of its words); a
// step that keeps fewer puts its positions in shared memory first, and its rounds
// then have every lane at work (a third of the rows kept: 10 rounds for 32).
constexpr unsigned SEL_DENSE = 640;

struct SelScratch {           // of one list; list j of several follows at j * (steps, ranges)
    uint32_t *bits;           // 32 keep words per step (bit b of word w: row 1024 step + 32 w + b)
    uint32_t *cnt;            // kept rows per step
    unsigned *done;           // CTAs that have finished (0 between launches)
    uint32_t *tot;            // kept rows per range
    unsigned long long *off;  // first output row per range
    unsigned steps, per, ranges;  // range b owns steps [b per, (b + 1) per)
};

// Scratch for `lists` selections over n rows from the context's pool (*block is
// freed by the caller; `extra` further bytes at *extra_at).  The finished-CTA
// counter is the context's (under capture the graph's own): the last CTA of a mark
// kernel sets it back to 0.
// per: steps per range (0: chosen by n).
int sel_scratch(tid_ctx *ctx, int64_t n, int lists, size_t extra, SelScratch *sc, void **block, void **extra_at,
                unsigned per = 0);

// 4-bit masks of a lane's rows (m[g], bits e: row 128 g + 4 lane + e of the step)
// to the step's keep words: lane 8k + g returns word 4g + k.
__device__ __forceinline__ uint32_t sel_word(const unsigned *m) {
    const unsigned sub = threadIdx.x & 7u;
    uint32_t word = 0;
#pragma unroll
    for (int g = 0; g < 8; ++g) {  // eight lanes merge their masks
        uint32_t v = m[g] << (4 * sub);
        v |= __shfl_xor_sync(0xffffffffu, v, 1);
        v |= __shfl_xor_sync(0xffffffffu, v, 2);
        v |= __shfl_xor_sync(0xffffffffu, v, 4);
        if (sub == (unsigned)g) word = v;
    }
    return word;
}
__device__ __forceinline__ unsigned sel_word_index() {  // of the word sel_word returns
    return (threadIdx.x & 7u) * 4 + ((threadIdx.x & 31u) >> 3);
}

// Exclusive scan of the range totals by one CTA; returns their sum.
__device__ __forceinline__ unsigned long long sel_scan_totals(const uint32_t *tot, unsigned long long *off,
                                                              unsigned ranges) {
    __shared__ unsigned long long s_w[SEL_WARPS];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned chunk = (ranges + SEL_THREADS - 1) / SEL_THREADS;  // consecutive ranges per thread
    const unsigned b0 = min(threadIdx.x * chunk, ranges), b1 = min(b0 + chunk, ranges);
    unsigned long long sum = 0;
#pragma unroll 8
    for (unsigned b = b0; b < b1; ++b) sum += __ldcg(tot + b);
    unsigned long long x = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, d);
        if ((int)lane >= d) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    unsigned long long run = x - sum, all = 0;
    for (int w = 0; w < SEL_WARPS; ++w) {
        if (w < (int)warp) run += s_w[w];
        all += s_w[w];
    }
#pragma unroll 8
    for (unsigned b = b0; b < b1; ++b) {
        off[b] = run;
        run += __ldcg(tot + b);
    }
    return all;
}

// End of a mark CTA with one list: `kept` is its warp's kept rows.  Writes the
// range's total; the last CTA scans the totals and writes the row count.
__device__ __forceinline__ void sel_finish(const SelScratch &sc, unsigned kept, int64_t *d_rows, int64_t *h_rows) {
    __shared__ unsigned s_kept[SEL_WARPS], s_last;
    if ((threadIdx.x & 31) == 0) s_kept[threadIdx.x >> 5] = kept;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned t = 0;
        for (int w = 0; w < SEL_WARPS; ++w) t += s_kept[w];
        __stcg(sc.tot + blockIdx.x, t);
        __threadfence();
        s_last = atomicAdd(sc.done, 1u) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    const unsigned long long all = sel_scan_totals(sc.tot, sc.off, sc.ranges);
    if (threadIdx.x == 0) {
        *d_rows = (int64_t)all;
        *h_rows = (int64_t)all;
        *sc.done = 0;
    }
}

// Walks a range in an expand kernel: body(step, word, word_prefix, kept, first
// row) for every step with kept rows, the steps dealt out to `warps` warps, of
// which this is number `warp`; lane l holds keep word l and the kept rows of the
// words before it.
template <class Body>
__device__ __forceinline__ void sel_walk(const SelScratch &sc, unsigned range, unsigned warp, unsigned warps, Body body) {
    const unsigned lane = threadIdx.x & 31;
    const unsigned r0 = range * sc.per, r1 = min(r0 + sc.per, sc.steps);
    unsigned long long run = sc.off[range];
    for (unsigned q0 = r0; q0 < r1; q0 += 32) {
        const unsigned here = min(32u, r1 - q0);
        const unsigned cnt = lane < here ? sc.cnt[q0 + lane] : 0u;
        // this warp's steps that have kept rows, and the first one's words
        unsigned todo = __ballot_sync(0xffffffffu, cnt != 0 && lane % warps == warp);
        uint32_t next = todo ? sc.bits[(size_t)(q0 + __ffs(todo) - 1) * 32 + lane] : 0u;
        unsigned first = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, first, d);
            if ((int)lane >= d) first += y;
        }
        const unsigned kept = __shfl_sync(0xffffffffu, first, 31);
        first -= cnt;  // of step q0 + lane
        while (todo) {
            const unsigned li = __ffs(todo) - 1;
            todo &= todo - 1;
            const uint32_t word = next;
            if (todo) next = sc.bits[(size_t)(q0 + __ffs(todo) - 1) * 32 + lane];
            const unsigned sn = __shfl_sync(0xffffffffu, cnt, li);
            const unsigned long long o0 = run + __shfl_sync(0xffffffffu, first, li);
            const unsigned pc = __popc(word);
            unsigned xo = pc;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, xo, d);
                if ((int)lane >= d) xo += y;
            }
            body(q0 + li, word, xo - pc, sn, o0);
        }
        run += kept;
    }
}

// Positions (within their step) of a sparse step's kept rows, in order, to
// stage[0 .. kept); kept < SEL_DENSE.
__device__ __forceinline__ void sel_stage(uint32_t word, unsigned at, uint16_t *stage) {
    const unsigned lane = threadIdx.x & 31;
    while (word) {
        stage[at++] = (uint16_t)(lane * 32 + __ffs(word) - 1);
        word &= word - 1;
    }
    __syncwarp();
}

// ---- expand of a search: the kept rows' numbers -------------------------------

// A long range (32 steps) is two warps', so that the thousands of ranges of a large
// store, most of them without a hit, are few CTAs (one warp left too few in flight
// where hits are many: 23.6M of 200M triples 67 us, two 58).  A short one is a CTA's.
constexpr unsigned SEL_RANGE_WARPS = 2;
__device__ __forceinline__ void sel_expand_index(const SelScratch &sc, int32_t *out, int64_t cap) {
    __shared__ uint16_t s_stage[SEL_WARPS][SEL_DENSE];
    const unsigned lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
    uint16_t *stage = s_stage[threadIdx.x >> 5];
    const bool long_range = sc.per > SEL_WARPS;
    const unsigned warp = threadIdx.x >> 5, warps = long_range ? SEL_RANGE_WARPS : SEL_WARPS;
    const unsigned range = blockIdx.x * (SEL_WARPS / warps) + warp / warps;
    if (range >= sc.ranges || sc.tot[range] == 0) return;
    sel_walk(sc, range, warp % warps, warps, [&](unsigned step, uint32_t word, unsigned xo, unsigned sn, unsigned long long o0) {
        const int32_t base = (int32_t)(step * SEL_STEP);
        if (sn >= SEL_DENSE) {
#pragma unroll 8
            for (int w = 0; w < 32; ++w) {
                const uint32_t bw = __shfl_sync(0xffffffffu, word, w);
                const unsigned long long pos = o0 + __shfl_sync(0xffffffffu, xo, w) + __popc(bw & lt);
                if (((bw >> lane) & 1u) && pos < (unsigned long long)cap) out[pos] = base + w * 32 + (int32_t)lane;
            }
        } else {
            sel_stage(word, xo, stage);
            for (unsigned e = lane; e < sn; e += 32)
                if (o0 + e < (unsigned long long)cap) out[o0 + e] = base + stage[e];
            __syncwarp();  // the stage is rewritten by the next step
        }
    });
}

inline unsigned sel_index_grid(const SelScratch &sc) {
    constexpr unsigned in_cta = SEL_WARPS / SEL_RANGE_WARPS;
    return sc.per > SEL_WARPS ? (sc.ranges + in_cta - 1) / in_cta : sc.ranges;
}

// ---- streaming loads of store columns ------------------------------------------

__device__ __forceinline__ int4 ld_stream_v4(const int32_t *p) {
    int4 v;
    asm("ld.global.nc.L1::no_allocate.L2::256B.v4.s32 {%0,%1,%2,%3}, [%4];"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "l"(p));
    return v;
}

__device__ __forceinline__ int32_t ld_stream(const int32_t *p) {
    int32_t v;
    asm("ld.global.nc.L1::no_allocate.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// four consecutive elements e0..e0+3 of a column; elements at or past n read as 0
template <bool VEC>
__device__ __forceinline__ int4 load4(const int32_t *__restrict__ c, int64_t e0, int64_t n) {
    if (VEC && e0 + 3 < n) return ld_stream_v4(c + e0);
    int4 v = make_int4(0, 0, 0, 0);
    if (e0 < n) v.x = ld_stream(c + e0);
    if (e0 + 1 < n) v.y = ld_stream(c + e0 + 1);
    if (e0 + 2 < n) v.z = ld_stream(c + e0 + 2);
    if (e0 + 3 < n) v.w = ld_stream(c + e0 + 3);
    return v;
}

__device__ __forceinline__ unsigned eq4(int4 v, int32_t k) {
    return (unsigned)(v.x == k) | ((unsigned)(v.y == k) << 1) |
           ((unsigned)(v.z == k) << 2) | ((unsigned)(v.w == k) << 3);
}

// A lane's 32 triples of a step, the columns in U (bit 0 s, 1 p, 2 o): v[c][g] holds
// triples 1024 step + 128 g + 4 lane + (0..3); those past n read as 0.
template <int U, bool VEC>
__device__ __forceinline__ void load_step(const int32_t *__restrict__ S, const int32_t *__restrict__ P,
                                          const int32_t *__restrict__ O, int64_t n, unsigned step, int4 (*v)[8]) {
    const int64_t base = (int64_t)step * SEL_STEP + (threadIdx.x & 31) * 4;
    auto four = [](const int32_t *p) {
        if (VEC) return ld_stream_v4(p);
        return make_int4(ld_stream(p), ld_stream(p + 1), ld_stream(p + 2), ld_stream(p + 3));
    };
    if ((int64_t)(step + 1) * SEL_STEP <= n) {
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            if (U & 1) v[0][g] = four(S + base + g * 128);
            if (U & 2) v[1][g] = four(P + base + g * 128);
            if (U & 4) v[2][g] = four(O + base + g * 128);
        }
    } else {
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            if (U & 1) v[0][g] = load4<VEC>(S, base + g * 128, n);
            if (U & 2) v[1][g] = load4<VEC>(P, base + g * 128, n);
            if (U & 4) v[2][g] = load4<VEC>(O, base + g * 128, n);
        }
    }
}

}  // namespace tid
