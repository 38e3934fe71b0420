// Lookup of a mode's hottest rows in shared memory: a table of buckets of two
// (row, slot) pairs, one hash, one 16-byte load per lookup.
#pragma once
#include "internal.h"

namespace blco {
namespace {

__device__ __forceinline__ uint32_t hot_hash(uint32_t row, int log2n) {
    return log2n > 0 ? (row * 0x9E3779B1u) >> (32 - log2n) : 0u;
}

// Fills the table with rows 0..kw-1 of hot_rows (by decreasing count), all
// threads at once: thread i ranks row i among the hotter rows of its bucket; a
// third one stays out and is simply a cold row. `ids` is scratch of kw words.
// Ends with the table complete for the whole CTA.
template <int THREADS>
__device__ __forceinline__ void fill_hot_table(uint4 *table, int nb, int log2nb, const uint32_t *hot_rows, int kw,
                                               uint32_t *ids) {
    for (int i = threadIdx.x; i < nb; i += THREADS) table[i] = make_uint4(kNoRow, 0u, kNoRow, 0u);
    for (int i = threadIdx.x; i < kw; i += THREADS) ids[i] = __ldg(hot_rows + i);
    __syncthreads();
    for (int i = threadIdx.x; i < kw; i += THREADS) {
        const uint32_t row = ids[i], b = hot_hash(row, log2nb);
        int before = 0;
        for (int j = 0; j < i; ++j) before += hot_hash(ids[j], log2nb) == b;
        if (before < 2) reinterpret_cast<uint2 *>(table + b)[before] = make_uint2(row, (uint32_t)i);
    }
    __syncthreads();
}

}  // namespace
}  // namespace blco
