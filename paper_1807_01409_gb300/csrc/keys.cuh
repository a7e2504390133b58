// A set of join terms on the device, each with a number: the entailment's second
// search asks of every triple whether its term is one of them, and which.
#pragma once

#include "ops.cuh"
#include "select.cuh"

namespace tid {

// Terms that lie in a short range (predicates, classes) are numbered by their
// place in it and held as one bit each; others by their slot in an open-addressing
// table, at most half full (0 = empty).  0 (unbound) is never in the set.
struct KeySet {
    const uint32_t *bits;  // null: the table
    uint32_t lo, w;        // range in sort order (int32 ^ 0x80000000)
    const int32_t *table;
    int tbits;             // log2 of the table size
};

constexpr uint32_t KEY_HASH = 0x9E3779B1u;  // multiplicative (Knuth) hash: the top bits depend on every bit of the key

__host__ __device__ __forceinline__ uint32_t home_slot(int32_t key, int tbits) {
    return ((uint32_t)key * KEY_HASH) >> (32 - tbits);
}

// number of `key`, -1 if it is not in the set
__device__ __forceinline__ int key_number(const KeySet &s, int32_t key) {
    if (key == 0) return -1;
    if (s.bits) {
        const uint32_t d = ((uint32_t)key ^ 0x80000000u) - s.lo;
        return d < s.w && ((__ldg(s.bits + (d >> 5)) >> (d & 31)) & 1u) ? (int)d : -1;
    }
    const uint32_t mask = (1u << s.tbits) - 1u;
    uint32_t h = home_slot(key, s.tbits);
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        const int32_t t = __ldg(s.table + h);
        if (t == key) return (int)h;
        if (t == 0) return -1;
        h = (h + 1) & mask;
    }
    return -1;
}

// Rows (triples as three columns) of which those are kept whose fixed_slot holds
// fixed_val (fixed_slot -1: any) and whose key_slot term is a key.
struct KeyedScan {
    const int32_t *col[3];
    int64_t n;
    int fixed_slot;
    int32_t fixed_val;
    int key_slot;
    KeySet keys;
    int vec;  // the columns are 16-byte aligned
};

// The kept rows of a marked scan, in order, into out's columns: column c is slot
// src[c], or (src[c] == 3) map[number of the row's key].
int expand_keyed(tid_ctx *ctx, const KeyedScan &ks, const SelScratch &sc, const int8_t *src, const int32_t *map,
                 tid_set *out, const BoundsOut &mm);

}  // namespace tid
