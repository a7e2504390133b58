// tid_entail: RDFS entailment rules as two searches and a join (Section 5,
// Table "RDFS Entailment rules" and the Rule-11 walk-through).
//
//  1. search the schema premise (?a TERM ?b) -- K1 -- and extract its result
//     vector (a, b) -- K3/K4;
//  2. its distinct terms at the join position (the paper's keys of the second
//     GPUSearch) -- a projection with DISTINCT -- are the key set (keys.cuh);
//  3. one pass over the store marks the triples of the other premise whose term
//     at the join position is a key (k_key_mark: their number, the keys among
//     them, and the range of the conclusion's term).  When both premises search
//     the same predicate, the pass is over the first search's result vector.
//  4. the join on the shared term, the conclusion's terms kept with DISTINCT:
//      * a pair of terms, one from each premise, whose bit matrix (rank of the
//        schema term by data term - min) is small: every marked triple sets the
//        bits of its pairs, and the set bits, read in order, are the distinct
//        pairs in canonical order.  Nothing is extracted, joined or sorted;
//      * a schema premise with one row per key (a class with one superclass): the
//        joined rows are the marked triples with the key's term replaced, so they
//        are extracted that way and sorted once;
//      * otherwise: extraction, hash join, and one sort of the conclusion's terms, by
//        the bounds that the extraction leaves (R9 over 20M triples whose classes have
//        three superclasses each: 2.2 ms; 3.8 with a pass for the bounds and a second
//        sort that puts the fixed predicate in, 3.2 with one and copied columns).
// Measured on GB300, 200M triples and their schema, the six rules: 21.6 -> 12.4 ms.
// Kernel times by rule: R2 2.9 -> 1.7, R3 1.7 -> 1.1, R5 0.4 -> 0.2, R7 5.4 -> 3.4, R9
// 7.5 -> 3.9, R11 0.5 -> 0.3 ms; k_key_mark 268 us over one column of 200M triples, 359
// over two (a third column of loads at once, 80 registers, took 430 and 627 us)
// (before: every rule extracted its marked rows, R7 and R9 materialised the hash
// join's rows).  Bound: R2 and R3 by the matrix's random L2 reads, R7 and R9 by the
// digit passes of their sort.
#include <algorithm>
#include <vector>

#include "keys.cuh"
#include "ops.cuh"

namespace tid {
int bind_set(tid_ctx *ctx, const tid_store *st, const tid_pattern &pat, const tid_set *idx, const tid_pred *preds,
             int n_preds, tid_set **out, const VarMember *mem = nullptr, int n_mem = 0);
}  // namespace tid

using namespace tid;

namespace {

enum Term { NONE = -1, TYPE = 0, DOMAIN, RANGE, SUBPROP, SUBCLASS };

// variable ids used inside the evaluation (a and b of the schema premise, then
// the data premise's own variables)
constexpr int8_t VA = 10, VB = 11, VC = 12, VD = 13;

struct Rule {
    int schema;          // the schema premise is (?a schema ?b), a = VA, b = VB
    int8_t on;           // join variable: VA or VB
    int data_fixed;      // data premise: fixed predicate term, or NONE
    int key_slot;        // slot of the join variable in the data premise
    int8_t data_var[3];  // data premise variables per slot (-1: the fixed term or unused)
    int8_t then_var[3];  // conclusion per slot: a variable, or -1 for then_term
    int then_term;       // the conclusion's fixed predicate (slot 1), or NONE
};

bool rule_of(int id, Rule *r) {
    switch (id) {
        case TID_RULE_R2: *r = Rule{DOMAIN, VA, NONE, 1, {VC, VA, -1}, {VC, -1, VB}, TYPE}; return true;
        case TID_RULE_R3: *r = Rule{RANGE, VA, NONE, 1, {-1, VA, VC}, {VC, -1, VB}, TYPE}; return true;
        case TID_RULE_R5: *r = Rule{SUBPROP, VB, SUBPROP, 0, {VB, -1, VC}, {VA, -1, VC}, SUBPROP}; return true;
        case TID_RULE_R7: *r = Rule{SUBPROP, VA, NONE, 1, {VC, VA, VD}, {VC, VB, VD}, NONE}; return true;
        case TID_RULE_R9: *r = Rule{SUBCLASS, VA, TYPE, 2, {VC, -1, VA}, {VC, -1, VB}, TYPE}; return true;
        case TID_RULE_R11: *r = Rule{SUBCLASS, VB, SUBCLASS, 0, {VB, -1, VC}, {VA, -1, VC}, SUBCLASS}; return true;
        default: return false;
    }
}

__global__ void k_fill_i32(int32_t *__restrict__ out, int64_t n, int32_t v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = v;
}

constexpr int BM_THREADS = 256;

__device__ __forceinline__ uint32_t sort_order(int32_t x) { return (uint32_t)x ^ 0x80000000u; }
inline uint32_t sort_order_host(int32_t x) { return (uint32_t)x ^ 0x80000000u; }

// What a keyed pass finds besides its marks.
struct KeyStats {
    unsigned long long keys;  // keys that occur in the marked rows (the paper's #Dist2)
    uint32_t lo, hi;          // range of the marked rows' conclusion term, in sort order
};

constexpr unsigned KM_SMEM_KEYS = 16384;  // keys whose flags are kept in shared memory, a byte each, if there are no more

// Marks the scan's kept rows (mark of select.cuh).  flags gets one bit per key
// number that occurs; when term is not null, st->lo / st->hi its range over the
// kept rows (preset to ~0 and 0).  16 rows per lane at a time, their key tests side
// by side; the key column is read only where a group of 128 rows holds the fixed
// term at all, the term column only where one is kept.
__global__ void __launch_bounds__(SEL_THREADS)
k_key_mark(const __grid_constant__ KeyedScan ks, SelScratch sc, int64_t *__restrict__ d_rows,
           int64_t *__restrict__ h_rows, uint32_t *__restrict__ flags, unsigned numbers,
           const int32_t *__restrict__ term, KeyStats *__restrict__ st) {
    extern __shared__ uint8_t s_seen[];  // per key number, when there are at most KM_SMEM_KEYS
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool in_smem = numbers <= KM_SMEM_KEYS;
    if (in_smem) {
        for (unsigned w = threadIdx.x; w < numbers; w += SEL_THREADS) s_seen[w] = 0;
        __syncthreads();
    }
    auto column = [&](int slot) { return slot == 0 ? ks.col[0] : (slot == 1 ? ks.col[1] : ks.col[2]); };
    const int32_t *key = column(ks.key_slot), *fixed = ks.fixed_slot >= 0 ? column(ks.fixed_slot) : nullptr;
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    auto seen = [&](int h) {
        if (in_smem) {
            s_seen[h] = 1;
        } else {  // set a bit only while it is clear
            const uint32_t b = 1u << (h & 31);
            if (!(__ldcg(flags + (h >> 5)) & b)) atomicOr(flags + (h >> 5), b);
        }
    };
    auto four = [&](const int32_t *p) { return ks.vec ? ld_stream_v4(p) : make_int4(p[0], p[1], p[2], p[3]); };
    const unsigned r0 = blockIdx.x * sc.per, r1 = min(r0 + sc.per, sc.steps);
    unsigned kept = 0;
    for (unsigned step = r0 + warp; step < r1; step += SEL_WARPS) {
        const int64_t base = (int64_t)step * SEL_STEP + lane * 4;
        unsigned m[8];
        if ((int64_t)(step + 1) * SEL_STEP <= ks.n) {
#pragma unroll
            for (int h = 0; h < 8; h += 4) {
                int32_t x[16];
                unsigned want = 0xFFFFu;  // bit i: row i may be kept
                auto load = [&](const int32_t *p, int g) {
                    const int4 v = four(p + base + (h + g) * 128);
                    x[4 * g] = v.x, x[4 * g + 1] = v.y, x[4 * g + 2] = v.z, x[4 * g + 3] = v.w;
                };
#pragma unroll
                for (int g = 0; g < 4; ++g) load(fixed ? fixed : key, g);
                if (fixed) {
                    want = 0;
#pragma unroll
                    for (int i = 0; i < 16; ++i) want |= (unsigned)(x[i] == ks.fixed_val) << i;
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                        if (__any_sync(0xffffffffu, (want >> (4 * g)) & 0xFu)) load(key, g);
                }
                unsigned r = 0;
                if (ks.keys.bits) {
                    uint32_t word[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const uint32_t d = sort_order(x[i]) - ks.keys.lo;
                        word[i] = 0;
                        if (((want >> i) & 1u) && d < ks.keys.w && x[i] != 0) word[i] = __ldg(ks.keys.bits + (d >> 5));
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const uint32_t d = sort_order(x[i]) - ks.keys.lo;
                        if ((word[i] >> (d & 31)) & 1u) {
                            r |= 1u << i;
                            seen((int)d);
                        }
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const int k = ((want >> i) & 1u) ? key_number(ks.keys, x[i]) : -1;
                        if (k >= 0) {
                            r |= 1u << i;
                            seen(k);
                        }
                    }
                }
#pragma unroll
                for (int g = 0; g < 4; ++g) m[h + g] = (r >> (4 * g)) & 0xFu;
                if (term) {
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                        if (__any_sync(0xffffffffu, m[h + g])) load(term, g);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        if (!((r >> i) & 1u)) continue;
                        lo = min(lo, sort_order(x[i]));
                        hi = max(hi, sort_order(x[i]));
                    }
                }
            }
        } else {  // ragged last step
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                unsigned r = 0;
                for (int e = 0; e < 4; ++e) {
                    const int64_t i = base + g * 128 + e;
                    if (i >= ks.n || (fixed && fixed[i] != ks.fixed_val)) continue;
                    const int k = key_number(ks.keys, key[i]);
                    if (k < 0) continue;
                    seen(k);
                    r |= 1u << e;
                    if (term) {
                        lo = min(lo, sort_order(term[i]));
                        hi = max(hi, sort_order(term[i]));
                    }
                }
                m[g] = r;
            }
        }
        __syncwarp();
        const uint32_t word = sel_word(m);
        sc.bits[(size_t)step * 32 + sel_word_index()] = word;
        const unsigned c = __reduce_add_sync(0xffffffffu, __popc(word));
        if (lane == 0) sc.cnt[step] = c;
        kept += c;
    }
    if (term) {
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0 && lo <= hi) {  // skip an atomic that cannot widen the range
            if (lo < __ldcg(&st->lo)) atomicMin(&st->lo, lo);
            if (hi > __ldcg(&st->hi)) atomicMax(&st->hi, hi);
        }
    }
    if (in_smem) {
        __syncthreads();
        for (unsigned k0 = warp * 32; k0 < numbers; k0 += SEL_THREADS) {
            const unsigned k = k0 + lane;
            const uint32_t w = __ballot_sync(0xffffffffu, k < numbers && s_seen[k]);
            if (lane == 0 && (w & ~__ldcg(flags + (k0 >> 5)))) atomicOr(flags + (k0 >> 5), w);
        }
    }
    sel_finish(sc, kept, d_rows, h_rows);
}

// The conclusion's distinct pairs as the set bits of a matrix.  A marked row
// (join term, term t) joined with the schema rows of that join term gives the pairs
// (r, t) for A's other terms r.  r is ranked among A's distinct values of that
// term (ascending) and t is taken as d = order(t) - vmin.  Rows of the matrix
// follow the conclusion's first term and are 2^lg bits wide (the second term's span
// rounded up to a power of two): the pair is bit (r << lg) + d when A's term comes
// first, (d << lg) + r when t does.  The set bits in ascending order are the
// canonical distinct rows.
struct PairBits {
    const int32_t *key, *val;  // the scan's key column and conclusion term
    KeySet keys;
    const uint32_t *off;    // key number h: A's ranks are rank[off[h] .. off[h + 1])
    const uint32_t *rank;
    const uint32_t *kmask;  // key number h: the same ranks as a mask (t first, 2^lg <= 32)
    uint32_t vmin;
    int lg;
    int a_first;
    uint32_t *bits;
};

// Sets the pairs of U rows per lane (h[u] < 0: no row); all lanes take part.
// MASK: t first and rows of at most 32 bits, so a row's ranks are one mask within
// one word; lanes holding consecutive rows of the same word OR their masks (a
// segmented scan across the warp) and the last lane of each run writes it.  The U
// words are read together: a word that has the bits already costs no atomic (a
// stale read only costs the atomic).  Without the read, 58.7M rows whose terms are
// skewed queue on the popular words: 1658 us against 499.
// Otherwise one atomic OR per (row, rank) whose bit is clear; a lane skips a row
// equal, in key and term, to the previous lane's.
template <bool MASK, int U>
__device__ __forceinline__ void set_pairs(const PairBits &P, const int *h, const int32_t *t) {
    const unsigned lane = threadIdx.x & 31;
    if (MASK) {
        const unsigned le = lane == 31 ? 0xFFFFFFFFu : (2u << lane) - 1u;  // lanes <= this one
        uint64_t word[U];
        uint32_t acc[U], cur[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t g = (uint64_t)(sort_order(t[u]) - P.vmin) << P.lg;
            word[u] = h[u] >= 0 ? g >> 5 : ~0ull;
            acc[u] = h[u] >= 0 ? P.kmask[h[u]] << (g & 31) : 0u;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t wp = __shfl_up_sync(0xffffffffu, word[u], 1);
            const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || wp != word[u]);
            if (heads != 0xFFFFFFFFu) {  // some neighbours share a word
                const int start = 31 - __clz(heads & le);
#pragma unroll
                for (int s = 1; s < 32; s <<= 1) {
                    const uint32_t o = __shfl_up_sync(0xffffffffu, acc[u], s);
                    if ((int)lane - s >= start) acc[u] |= o;
                }
                if (lane < 31 && !((heads >> (lane + 1)) & 1u)) word[u] = ~0ull;  // the run's last lane writes
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) cur[u] = word[u] != ~0ull ? __ldcg(P.bits + word[u]) : 0xFFFFFFFFu;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if ((cur[u] & acc[u]) != acc[u]) atomicOr(P.bits + word[u], acc[u]);
    } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t d = sort_order(t[u]) - P.vmin;
            const int hp = __shfl_up_sync(0xffffffffu, h[u], 1);
            const uint32_t dp = __shfl_up_sync(0xffffffffu, d, 1);
            if (h[u] < 0 || (lane > 0 && hp == h[u] && dp == d)) continue;
            for (uint32_t j = P.off[h[u]]; j < P.off[h[u] + 1]; ++j) {
                const uint64_t r = P.rank[j];
                const uint64_t g = P.a_first ? (r << P.lg) + d : ((uint64_t)d << P.lg) + r;
                const uint32_t b = 1u << (g & 31);
                if (!(__ldcg(P.bits + (g >> 5)) & b)) atomicOr(P.bits + (g >> 5), b);
            }
        }
    }
}

template <bool MASK>
__global__ void __launch_bounds__(SEL_THREADS) k_pair_bits(const __grid_constant__ PairBits P, SelScratch sc) {
    __shared__ uint16_t s_stage[SEL_WARPS][SEL_DENSE];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int U = 4;  // rows per lane whose loads are in flight together
    uint16_t *stage = s_stage[warp];
    sel_walk(sc, blockIdx.x, warp, SEL_WARPS, [&](unsigned step, uint32_t word, unsigned xo, unsigned sn,
                                                   unsigned long long) {
        const int64_t base = (int64_t)step * SEL_STEP;
        const bool dense = sn >= SEL_DENSE;
        if (!dense) sel_stage(word, xo, stage);
        const unsigned rounds = dense ? 32 : (sn + 31) / 32;
#pragma unroll 1
        for (unsigned q0 = 0; q0 < rounds; q0 += U) {
            int32_t x[U], t[U];
            int h[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned q = q0 + u;
                int64_t r = -1;
                if (dense) {
                    if ((__shfl_sync(0xffffffffu, word, q) >> lane) & 1u) r = base + q * 32 + lane;
                } else if (q * 32 + lane < sn) {
                    r = base + stage[q * 32 + lane];
                }
                x[u] = r >= 0 ? P.key[r] : 0;
                t[u] = r >= 0 ? P.val[r] : 0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) h[u] = key_number(P.keys, x[u]);  // -1 without a row
            set_pairs<MASK, U>(P, h, t);
        }
        __syncwarp();  // the stage is rewritten by the next step
    });
}

// Reading the matrix out: segment s is words [s R 32, (s + 1) R 32), R rounds
// of 32 words, one warp per segment (a round's words one per lane).
__device__ __forceinline__ int64_t seg_of_warp() { return (int64_t)blockIdx.x * (BM_THREADS / 32) + (threadIdx.x >> 5); }

// counts[s] = set bits of segment s
__global__ void __launch_bounds__(BM_THREADS) k_seg_bits(const uint32_t *__restrict__ bits, int64_t nwords, int R,
                                                         int64_t nseg, uint32_t *__restrict__ counts) {
    const int64_t s = seg_of_warp();
    if (s >= nseg) return;
    const unsigned lane = threadIdx.x & 31;
    const int64_t w0 = s * R * 32 + lane;
    uint32_t c = 0;
#pragma unroll 8
    for (int r = 0; r < R; ++r) {
        const int64_t w = w0 + (int64_t)r * 32;
        c += w < nwords ? __popc(bits[w]) : 0u;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
    if (lane == 0) counts[s] = c;
}

// offs[s] = sum of counts[0, s) (64-bit), *total = sum of all.  One CTA steps
// through the counts 8192 at a time (eight consecutive ones per thread) with a
// carry.
__global__ void __launch_bounds__(1024) k_scan_segs(const uint32_t *__restrict__ counts, int64_t nseg,
                                                    unsigned long long *__restrict__ offs,
                                                    unsigned long long *__restrict__ total) {
    __shared__ unsigned long long s_w[32];
    __shared__ unsigned long long s_chunk;
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long carry = 0;
    for (int64_t base = 0; base < nseg; base += 1024 * 8) {
        const int64_t e0 = base + (int64_t)threadIdx.x * 8;
        uint32_t c[8];
        unsigned long long s = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            c[j] = e0 + j < nseg ? counts[e0 + j] : 0u;
            s += c[j];
        }
        unsigned long long x = s;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, d);
            if ((int)lane >= d) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        if (warp == 0) {
            const unsigned long long v = s_w[lane];
            unsigned long long y = v;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned long long z = __shfl_up_sync(0xffffffffu, y, d);
                if ((int)lane >= d) y += z;
            }
            s_w[lane] = y - v;
            if (lane == 31) s_chunk = y;
        }
        __syncthreads();
        unsigned long long run = carry + s_w[warp] + x - s;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (e0 + j < nseg) offs[e0 + j] = run;
            run += c[j];
        }
        carry += s_chunk;
        __syncthreads();  // s_w and s_chunk are rewritten by the next chunk
    }
    if (threadIdx.x == 0) *total = carry;
}

struct PairOut {  // decoding a set bit into the conclusion's row
    const int32_t *rankval;  // A's distinct terms, ascending
    uint32_t vmin;
    int lg;
    int a_first;
    int32_t *out0, *out1;
    __device__ __forceinline__ void put(uint64_t g, uint64_t pos) const {
        const uint64_t hi = g >> lg, lo = g & ((1ull << lg) - 1ull);
        const uint64_t r = a_first ? hi : lo, d = a_first ? lo : hi;
        const int32_t a = rankval[r], t = (int32_t)((vmin + (uint32_t)d) ^ 0x80000000u);
        out0[pos] = a_first ? a : t;
        out1[pos] = a_first ? t : a;
    }
};

// The set bits of each segment, in order, as rows at the segment's offset.  A
// round whose words hold few bits (at most two each) is written lane by lane,
// the lanes' rows being consecutive; a denser round word by word, the word's
// bits one per lane, so the stores are coalesced either way.
__global__ void __launch_bounds__(BM_THREADS) k_emit_pairs(const uint32_t *__restrict__ bits, int64_t nwords, int R,
                                                           int64_t nseg, const unsigned long long *__restrict__ offs,
                                                           PairOut O) {
    const int64_t s = seg_of_warp();
    if (s >= nseg) return;
    const unsigned lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    uint64_t pos = offs[s];
    constexpr int AHEAD = 8;  // rounds whose words are loaded together
    for (int r0 = 0; r0 < R; r0 += AHEAD) {
        uint32_t va[AHEAD];
#pragma unroll
        for (int q = 0; q < AHEAD; ++q) {
            const int64_t w = (s * R + r0 + q) * 32 + lane;
            va[q] = r0 + q < R && w < nwords ? bits[w] : 0u;
        }
#pragma unroll
        for (int q = 0; q < AHEAD; ++q) {
            const int64_t wb = (s * R + r0 + q) * 32;  // the round's first word
            if (r0 + q >= R || wb >= nwords) break;
            const int64_t w = wb + lane;
            uint32_t v = va[q];
            const uint32_t c = __popc(v);
            uint32_t x = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
                if ((int)lane >= d) x += y;
            }
            const uint64_t mine = pos + x - c;
            const uint32_t tot = __shfl_sync(0xffffffffu, x, 31);
            if (__any_sync(0xffffffffu, c > 2)) {
                unsigned nz = __ballot_sync(0xffffffffu, v != 0);
                while (nz) {
                    const int L = __ffs(nz) - 1;
                    nz &= nz - 1;
                    const uint32_t wv = __shfl_sync(0xffffffffu, v, L);
                    const uint64_t b0 = __shfl_sync(0xffffffffu, mine, L);
                    if ((wv >> lane) & 1u) O.put((uint64_t)(wb + L) * 32 + lane, b0 + __popc(wv & lt));
                }
            } else {
                uint64_t at = mine;
                while (v) {
                    const int b = __ffs(v) - 1;
                    v &= v - 1;
                    O.put((uint64_t)w * 32 + b, at++);
                }
            }
            pos += tot;
        }
    }
}

// *count = set bits of words[0, n) (one CTA)
__global__ void __launch_bounds__(1024) k_count_bits(const uint32_t *__restrict__ words, int64_t n,
                                                     unsigned long long *__restrict__ count) {
    __shared__ unsigned long long s_w[32];
    unsigned long long c = 0;
    for (int64_t i = threadIdx.x; i < n; i += 1024) c += (unsigned)__popc(words[i]);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x < 32) {
        c = s_w[threadIdx.x];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
        if (threadIdx.x == 0) *count = c;
    }
}

struct Sets {  // frees what it holds
    std::vector<tid_set *> v;
    ~Sets() {
        for (tid_set *s : v) set_free(s);
    }
    tid_set *keep(tid_set *s) {
        v.push_back(s);
        return s;
    }
};

int rows_of(tid_set *s, int64_t *n) { return set_rows_host(s, n); }

struct Buf {  // a device allocation freed on scope exit
    tid_ctx *c;
    void *p = nullptr;
    ~Buf() {
        if (p) dev_free(c, p);
    }
};

constexpr int64_t PAIR_MAX_SCHEMA_ROWS = 1 << 22;  // schema rows ranked on the host
constexpr int64_t MAP_MAX_SCHEMA_ROWS = 1 << 18;   // or made a map there, for R7's conclusion
// A matrix of up to 64 MiB stays mostly in L2 and is always taken; a larger
// one only up to 4 bytes per data-premise row: beyond L2 every pair's bit is a
// random DRAM read-modify-write, and joining and sorting the rows costs less
// (R9 at 200M: a 1.28 GB matrix took 4.8 ms to fill and read out).
constexpr uint64_t PAIR_MIN_BYTES = 64ull << 20;
constexpr uint64_t PAIR_BYTES_PER_ROW = 4;
constexpr uint64_t PAIR_MAX_BYTES = 4ull << 30;

// The schema premise's rows by key: (key number, other term), sorted.
struct SchemaRows {
    std::vector<std::pair<uint32_t, int32_t>> rows;
    bool one_each = true;  // one row per key
};

// One column of a set of pairs, from its rows on the host.
struct KeyTable {
    KeySet set{};
    uint32_t numbers = 0;              // key numbers lie in [0, numbers)
    std::vector<uint32_t> bits;        // direct: a bit per term of the range
    std::vector<int32_t> table;        // or the open-addressing table
    int64_t number(int32_t key) const {
        if (key == 0) return -1;
        if (table.empty()) {
            const uint32_t d = ((uint32_t)key ^ 0x80000000u) - set.lo;
            return d < set.w && ((bits[d >> 5] >> (d & 31)) & 1u) ? (int64_t)d : -1;
        }
        uint32_t h = home_slot(key, set.tbits);
        for (uint32_t probe = 0; probe < numbers; ++probe, h = (h + 1) & (numbers - 1)) {
            if (table[h] == key) return h;
            if (table[h] == 0) return -1;
        }
        return -1;
    }
};

// A key's arrays (flags, ranks, map) are indexed by number: a direct range of up to
// 2^20 terms costs at most a few MB of them and one bit test per triple in place
// of a hash probe.
constexpr uint64_t KEY_DIRECT = 1ull << 20;

void build_keys(const std::vector<int32_t> &keys, KeyTable *kt) {  // distinct, ascending
    uint32_t lo = 0xFFFFFFFFu, hi = 0;
    size_t n = 0;
    for (int32_t k : keys) {
        if (k == 0) continue;  // 0 never joins
        const uint32_t o = (uint32_t)k ^ 0x80000000u;
        lo = std::min(lo, o);
        hi = std::max(hi, o);
        ++n;
    }
    if (n == 0 || (uint64_t)hi - lo < KEY_DIRECT) {
        kt->set.lo = n ? lo : 0u;
        kt->set.w = n ? hi - lo + 1 : 1u;
        kt->numbers = kt->set.w;
        kt->bits.assign((kt->set.w + 31) / 32, 0u);
        for (int32_t k : keys) {
            const uint32_t d = ((uint32_t)k ^ 0x80000000u) - kt->set.lo;
            if (k != 0) kt->bits[d >> 5] |= 1u << (d & 31);
        }
        return;
    }
    kt->set.tbits = 4;
    while ((1ull << kt->set.tbits) < 2 * (uint64_t)n) ++kt->set.tbits;
    kt->numbers = 1u << kt->set.tbits;
    kt->table.assign(kt->numbers, 0);
    for (int32_t k : keys) {
        if (k == 0) continue;
        uint32_t h = home_slot(k, kt->set.tbits);
        while (kt->table[h] != 0) h = (h + 1) & (kt->numbers - 1);
        kt->table[h] = k;
    }
}

// The conclusion as the bit matrix of its distinct pairs (PairBits), when the
// matrix is small enough; *out stays null when it is not.  a_pos: which of the two
// conclusion terms is A's; O: the three-column result, pair columns at slots pos[2].
int conclude_pairs(tid_ctx *ctx, const KeyedScan &ks, const SelScratch &sc, const KeyTable &kt, const SchemaRows &sr,
                   const KeyStats &st, int64_t res2, const int32_t *term, int a_pos, const int *pos, int fixed_pos,
                   int32_t fixed_term, tid_set **out) {
    cudaStream_t stream = ctx->stream;
    // A's other terms ranked; the matrix's size decides the form
    std::vector<int32_t> vals;
    vals.reserve(sr.rows.size());
    for (const auto &r : sr.rows) vals.push_back(r.second);
    std::sort(vals.begin(), vals.end());
    vals.erase(std::unique(vals.begin(), vals.end()), vals.end());
    const uint64_t na = vals.size(), w = (uint64_t)(st.hi - st.lo) + 1;
    const uint64_t nrows = a_pos == 0 ? na : w, width = a_pos == 0 ? w : na;  // matrix rows, bits per row
    int lg = 0;
    while ((1ull << lg) < width) ++lg;
    int lr = 0;
    while ((1ull << lr) < nrows) ++lr;
    if (lg + lr > 40) return TID_OK;  // far beyond the size limit below
    const uint64_t nwords = ((nrows << lg) + 31) / 32, bytes = nwords * sizeof(uint32_t);
    if (bytes > std::max(PAIR_MIN_BYTES, PAIR_BYTES_PER_ROW * (uint64_t)res2) || bytes > PAIR_MAX_BYTES) return TID_OK;

    const bool use_mask = a_pos == 1 && lg <= 5;  // a row's ranks fit one word
    // layout: rank values (na) | off (numbers + 1) | ranks | masks (numbers, when used)
    const uint32_t nk = kt.numbers;
    std::vector<uint32_t> meta(na + nk + 1 + sr.rows.size() + (use_mask ? nk : 0), 0u);
    uint32_t *m_off = meta.data() + na, *m_rank = m_off + nk + 1, *m_mask = m_rank + sr.rows.size();
    for (uint64_t r = 0; r < na; ++r) meta[r] = (uint32_t)vals[r];
    for (size_t j = 0; j < sr.rows.size(); ++j) {
        const uint32_t rank = (uint32_t)(std::lower_bound(vals.begin(), vals.end(), sr.rows[j].second) - vals.begin());
        m_off[sr.rows[j].first + 1]++;
        m_rank[j] = rank;
        if (use_mask) m_mask[sr.rows[j].first] |= 1u << rank;
    }
    for (uint32_t h = 0; h < nk; ++h) m_off[h + 1] += m_off[h];
    Buf mb{ctx};
    TID_TRY(dev_alloc(ctx, &mb.p, meta.size() * sizeof(uint32_t)));
    TID_TRY_CUDA(cudaMemcpyAsync(mb.p, meta.data(), meta.size() * sizeof(uint32_t), cudaMemcpyHostToDevice, stream),
                 "pair ranks");
    const uint32_t *d_meta = (const uint32_t *)mb.p;

    // the matrix's bits, then its set bits in order as rows
    Buf bb{ctx};
    TID_TRY(dev_alloc(ctx, &bb.p, bytes));
    uint32_t *bits = (uint32_t *)bb.p;
    TID_TRY_CUDA(cudaMemsetAsync(bits, 0, bytes, stream), "pair bits");
    const PairBits P{ks.col[ks.key_slot], term, ks.keys, d_meta + na, d_meta + na + nk + 1,
                     use_mask ? d_meta + na + nk + 1 + sr.rows.size() : nullptr, st.lo, lg, a_pos == 0 ? 1 : 0, bits};
    if (use_mask) k_pair_bits<true><<<sc.ranges, SEL_THREADS, 0, stream>>>(P, sc);
    else k_pair_bits<false><<<sc.ranges, SEL_THREADS, 0, stream>>>(P, sc);
    TID_TRY(launch_check("k_pair_bits"));
    // segments of R rounds of 32 words, at most 2^16 of them (one warp each)
    const int rounds = (int)std::max<int64_t>(8, ceil_div((int64_t)nwords, (int64_t)32 << 16));
    const int64_t nseg = ceil_div((int64_t)nwords, (int64_t)rounds * 32);
    const unsigned seg_ctas = (unsigned)ceil_div(nseg, BM_THREADS / 32);
    const int64_t cpad = (nseg + 1) & ~(int64_t)1;
    Buf sb{ctx};
    TID_TRY(dev_alloc(ctx, &sb.p, sizeof(uint32_t) * cpad + sizeof(unsigned long long) * (nseg + 1)));
    uint32_t *counts = (uint32_t *)sb.p;
    unsigned long long *offs = (unsigned long long *)(counts + cpad), *d_total = offs + nseg;
    k_seg_bits<<<seg_ctas, BM_THREADS, 0, stream>>>(bits, (int64_t)nwords, rounds, nseg, counts);
    TID_TRY(launch_check("k_seg_bits"));
    k_scan_segs<<<1, 1024, 0, stream>>>(counts, nseg, offs, d_total);
    TID_TRY(launch_check("k_scan_segs"));
    unsigned long long total = 0;
    TID_TRY_CUDA(cudaMemcpyAsync(&total, d_total, sizeof total, cudaMemcpyDeviceToHost, stream), "pair rows");
    TID_TRY_CUDA(cudaStreamSynchronize(stream), "pair rows");
    const int8_t ovars[3] = {0, 1, 2};
    tid_set *O = nullptr;
    TID_TRY(set_alloc(ctx, 3, ovars, (int64_t)total, &O));
    int rc = TID_OK;
    if (total > 0) {
        const PairOut E{(const int32_t *)d_meta, st.lo, lg, a_pos == 0 ? 1 : 0, O->col[pos[0]], O->col[pos[1]]};
        k_emit_pairs<<<seg_ctas, BM_THREADS, 0, stream>>>(bits, (int64_t)nwords, rounds, nseg, offs, E);
        rc = launch_check("k_emit_pairs");
        if (rc == TID_OK) {
            k_fill_i32<<<grid_for((int64_t)total, 256, 8), 256, 0, stream>>>(O->col[fixed_pos], (int64_t)total, fixed_term);
            rc = launch_check("k_fill_i32");
        }
    }
    if (rc == TID_OK) rc = set_rows_const(O, (int64_t)total);
    if (rc == TID_OK) {
        // valid bounds (sort order) of each column
        O->bounded = true;
        O->lo[pos[a_pos]] = sort_order_host(vals.front());
        O->hi[pos[a_pos]] = sort_order_host(vals.back());
        O->lo[pos[1 - a_pos]] = st.lo;
        O->hi[pos[1 - a_pos]] = st.hi;
        O->lo[fixed_pos] = O->hi[fixed_pos] = sort_order_host(fixed_term);
        rc = set_ready(O);
    }
    if (rc != TID_OK) {
        set_free(O);
        return rc;
    }
    *out = O;
    return TID_OK;
}

}  // namespace

extern "C" int tid_entail(tid_ctx *ctx, const tid_store *st, int rule, const tid_rdfs_vocab *vocab, tid_set **out,
                          tid_entail_stats *stats) {
    clear_error();
    tid::Range nvtx_range("tid_entail");
    if (!ctx || !st || !vocab || !out) return fail(TID_ERR_ARG, "tid_entail: null argument");
    *out = nullptr;
    if (st->ctx != ctx) return fail(TID_ERR_ARG, "tid_entail: store belongs to another context");
    Rule R;
    if (!rule_of(rule, &R)) return fail(TID_ERR_ARG, "tid_entail: unknown rule %d", rule);
    const int32_t term[5] = {vocab->type, vocab->domain, vocab->range, vocab->sub_property_of, vocab->sub_class_of};
    for (int t = 0; t < 5; ++t)
        if (term[t] <= 0) return fail(TID_ERR_ID, "tid_entail: vocabulary ID %d is not positive", term[t]);
    CallGuard g(ctx);
    cudaStream_t stream = ctx->stream;
    tid_entail_stats sx{};
    Sets hold;

    // 1) schema premise (?a TERM ?b) -> (a, b)
    tid_pattern sp{};
    sp.p = term[R.schema];
    sp.var[0] = VA;
    sp.var[1] = -1;
    sp.var[2] = VB;
    tid_set *idx1 = nullptr, *A = nullptr;
    TID_TRY(tid_match(ctx, st, sp, &idx1));
    hold.keep(idx1);
    TID_TRY(rows_of(idx1, &sx.res1));
    TID_TRY(bind_set(ctx, st, sp, idx1, nullptr, 0, &A));
    hold.keep(A);

    // 2) its distinct join terms -> key set
    tid_set *K = nullptr;
    TID_TRY(project_set(ctx, A, &R.on, 1, &K));
    hold.keep(K);
    TID_TRY(rows_of(K, &sx.dist1));
    std::vector<int32_t> keys((size_t)sx.dist1);
    if (sx.dist1 > 0) {
        int64_t got = 0;
        TID_TRY(tid_set_to_host(K, keys.data(), sx.dist1, &got));
    }
    KeyTable kt;
    build_keys(keys, &kt);
    Buf kb{ctx};
    const size_t kbytes = kt.table.empty() ? kt.bits.size() * 4 : kt.table.size() * 4;
    TID_TRY(dev_alloc(ctx, &kb.p, kbytes));
    TID_TRY_CUDA(cudaMemcpyAsync(kb.p, kt.table.empty() ? (const void *)kt.bits.data() : (const void *)kt.table.data(), kbytes,
                                 cudaMemcpyHostToDevice, stream),
                 "key set");
    if (kt.table.empty()) kt.set.bits = (const uint32_t *)kb.p;
    else kt.set.table = (const int32_t *)kb.p;

    // 3) the data premise's triples whose join term is a key.  Both premises on
    //    the same predicate: the first search found the data premise's triples too
    KeyedScan ks{};
    const bool same = R.data_fixed != NONE && term[R.data_fixed] == term[R.schema];
    ks.col[0] = same ? A->col[0] : st->s;
    ks.col[1] = st->p;
    ks.col[2] = same ? A->col[1] : st->o;
    ks.n = same ? sx.res1 : st->n;
    ks.fixed_slot = same || R.data_fixed == NONE ? -1 : 1;
    ks.fixed_val = R.data_fixed == NONE ? 0 : term[R.data_fixed];
    ks.key_slot = R.key_slot;
    ks.keys = kt.set;
    ks.vec = same || st->aligned16;
    // the conclusion's terms: their slots, and where each comes from
    const int8_t other = R.on == VA ? VB : VA;  // A's term that is not the join term
    int pos[3], kc = 0, a_pos = -1, fixed_pos = -1;
    int8_t src[3];  // data slot of conclusion term i; 3: A's other term
    for (int slot = 0; slot < 3; ++slot) {
        if (R.then_var[slot] < 0) {
            fixed_pos = slot;
            continue;
        }
        if (R.then_var[slot] == other) {
            a_pos = kc;
            src[kc] = 3;
        } else {
            for (int d = 0; d < 3; ++d)
                if (R.data_var[d] == R.then_var[slot]) src[kc] = (int8_t)d;
        }
        pos[kc++] = slot;
    }
    const bool pair = kc == 2;
    const int32_t *pair_term = pair ? ks.col[src[1 - a_pos]] : nullptr;
    const int8_t one = 0;
    tid_set *count = nullptr;  // holds the number of marked rows
    TID_TRY(set_alloc(ctx, 1, &one, 0, &count));
    hold.keep(count);
    SelScratch sc{};
    Buf scb{ctx}, fb{ctx};
    KeyStats ss{0, 0xFFFFFFFFu, 0u};
    if (sx.dist1 > 0 && ks.n > 0) {
        TID_TRY(sel_scratch(ctx, ks.n, 1, 0, &sc, &scb.p, nullptr));
        const uint32_t fwords = (kt.numbers + 31) / 32;
        TID_TRY(dev_alloc(ctx, &fb.p, sizeof(KeyStats) + sizeof(uint32_t) * fwords));
        KeyStats *d_ss = (KeyStats *)fb.p;
        uint32_t *flags = (uint32_t *)(d_ss + 1);
        TID_TRY_CUDA(cudaMemcpyAsync(d_ss, &ss, sizeof ss, cudaMemcpyHostToDevice, stream), "key stats");
        TID_TRY_CUDA(cudaMemsetAsync(flags, 0, sizeof(uint32_t) * fwords, stream), "key flags");
        const size_t smem = kt.numbers <= KM_SMEM_KEYS ? kt.numbers : 0;
        k_key_mark<<<sc.ranges, SEL_THREADS, smem, stream>>>(ks, sc, count->d_rows, count->slot.dev, flags, kt.numbers, pair_term,
                                                             d_ss);
        TID_TRY(launch_check("k_key_mark"));
        k_count_bits<<<1, 1024, 0, stream>>>(flags, fwords, &d_ss->keys);
        TID_TRY(launch_check("k_count_bits"));
        TID_TRY_CUDA(cudaMemcpyAsync(&ss, d_ss, sizeof ss, cudaMemcpyDeviceToHost, stream), "key stats");
    } else {
        TID_TRY(set_rows_const(count, 0));
    }
    TID_TRY(set_ready(count));
    // the schema premise's rows (synchronises: the statistics are on the host too)
    SchemaRows sr;
    if (sx.res1 <= (pair ? PAIR_MAX_SCHEMA_ROWS : MAP_MAX_SCHEMA_ROWS)) {
        std::vector<int32_t> arows((size_t)sx.res1 * 2);
        int64_t got = 0;
        TID_TRY(tid_set_to_host(A, arows.data(), sx.res1, &got));
        const int ak = A->vars[0] == R.on ? 0 : 1;
        sr.rows.reserve((size_t)got);
        for (int64_t i = 0; i < got; ++i) {
            const int64_t h = kt.number(arows[(size_t)i * 2 + ak]);
            if (h >= 0) sr.rows.emplace_back((uint32_t)h, arows[(size_t)i * 2 + 1 - ak]);
        }
        std::sort(sr.rows.begin(), sr.rows.end());
        sr.rows.erase(std::unique(sr.rows.begin(), sr.rows.end()), sr.rows.end());
        for (size_t i = 1; i < sr.rows.size(); ++i) sr.one_each = sr.one_each && sr.rows[i].first != sr.rows[i - 1].first;
    }
    TID_TRY_CUDA(cudaStreamSynchronize(stream), "key stats");
    TID_TRY(rows_of(count, &sx.res2));
    sx.dist2 = (int64_t)ss.keys;

    // 4) the conclusion, labelled (s, p, o); a fixed predicate is its middle
    //    column, whose one value keeps the canonical order
    const int8_t ovars[3] = {0, 1, 2};
    const int32_t fixed_term = R.then_term == NONE ? 0 : term[R.then_term];
    tid_set *O = nullptr;
    if (sx.res2 == 0) {
        TID_TRY(set_alloc(ctx, 3, ovars, 0, &O));
        int rc = set_rows_const(O, 0);
        if (rc == TID_OK) rc = set_ready(O);
        if (rc != TID_OK) {
            set_free(O);
            return rc;
        }
    } else if (pair && !sr.rows.empty()) {
        TID_TRY(conclude_pairs(ctx, ks, sc, kt, sr, ss, sx.res2, pair_term, a_pos, pos, fixed_pos, fixed_term, &O));
    }
    if (!O) {
        // the joined rows' conclusion terms, in any order, then sorted with DISTINCT
        tid_set *J = nullptr;
        const int32_t *ccols[3];
        Bounds cb{};
        int64_t nj = 0;
        if (!sr.rows.empty() && sr.one_each) {
            int8_t jvars[3] = {0, 1, 2};
            TID_TRY(set_alloc(ctx, kc, jvars, sx.res2, &J));
            hold.keep(J);
            std::vector<int32_t> map(kt.numbers, 0);
            for (const auto &r : sr.rows) map[r.first] = r.second;
            Buf mapb{ctx};
            TID_TRY(dev_alloc(ctx, &mapb.p, map.size() * 4));
            int32_t *d_map = (int32_t *)mapb.p;
            TID_TRY_CUDA(cudaMemcpyAsync(d_map, map.data(), map.size() * 4, cudaMemcpyHostToDevice, stream), "key map");
            BoundsOut mm{};
            if (!pair) TID_TRY(bounds_out(J, &mm));
            TID_TRY(expand_keyed(ctx, ks, sc, src, d_map, J, mm));
            TID_TRY_CUDA(cudaStreamSynchronize(stream), "conclusion range");  // (and the host copy of the map)
            if (pair) {  // the data term's range is known; A's terms are on the host
                cb.lo[1 - a_pos] = ss.lo;
                cb.hi[1 - a_pos] = ss.hi;
                cb.lo[a_pos] = 0xFFFFFFFFu;
                for (const auto &r : sr.rows) {
                    cb.lo[a_pos] = std::min(cb.lo[a_pos], sort_order_host(r.second));
                    cb.hi[a_pos] = std::max(cb.hi[a_pos], sort_order_host(r.second));
                }
            } else {
                read_bounds(J, kc, cb.lo, cb.hi);
            }
            for (int i = 0; i < kc; ++i) ccols[i] = J->col[i];
            nj = sx.res2;
        } else {
            // the data premise's rows in store order, joined with the schema side
            // (the small one) as the hash table
            int8_t bvars[3], bsrc[3];
            int nb = 0;
            for (int slot = 0; slot < 3; ++slot) {
                if (R.data_var[slot] < 0) continue;
                bvars[nb] = R.data_var[slot];
                bsrc[nb++] = (int8_t)slot;
            }
            tid_set *B = nullptr;
            TID_TRY(set_alloc(ctx, nb, bvars, sx.res2, &B));
            hold.keep(B);
            BoundsOut mm{};
            TID_TRY(bounds_out(B, &mm));
            TID_TRY(expand_keyed(ctx, ks, sc, bsrc, nullptr, B, mm));
            TID_TRY(set_rows_const(B, sx.res2));
            TID_TRY(set_ready(B));
            TID_TRY(join_sets(ctx, A, B, TID_JOIN_HASH, &J, false));
            hold.keep(J);
            TID_TRY(rows_of(J, &nj));
            // the join has waited for its row count, so B's bounds are on the host; a
            // joined column keeps its side's (A, a bound result with rows, has them)
            read_bounds(B, nb, B->lo, B->hi);
            for (int i = 0; i < kc; ++i) {
                const int8_t v = R.then_var[pos[i]];
                int c = 0, a = 0, b = 0;
                while (J->vars[c] != v) ++c;
                ccols[i] = J->col[c];
                while (a < A->k && A->vars[a] != v) ++a;
                while (b < nb && bvars[b] != v) ++b;
                cb.lo[i] = a < A->k ? A->lo[a] : B->lo[b];
                cb.hi[i] = a < A->k ? A->hi[a] : B->hi[b];
            }
        }
        if (!pair) {
            TID_TRY(canonicalize(ctx, ccols, 3, ovars, nj, true, &cb, &O));
        } else {
            // a column of one value has no field in the packed rows (two columns
            // always fit them) and is not read
            const int32_t *o3[3];
            Bounds ob{};
            for (int i = 0; i < 2; ++i) {
                o3[pos[i]] = ccols[i];
                ob.lo[pos[i]] = cb.lo[i];
                ob.hi[pos[i]] = cb.hi[i];
            }
            o3[fixed_pos] = ccols[0];
            ob.lo[fixed_pos] = ob.hi[fixed_pos] = sort_order_host(fixed_term);
            TID_TRY(canonicalize(ctx, o3, 3, ovars, nj, true, &ob, &O));
        }
    }
    hold.keep(O);
    TID_TRY(rows_of(O, &sx.all));
    hold.v.pop_back();
    if (stats) *stats = sx;
    *out = O;
    return TID_OK;
}
