// Where a tile's ranks stand in shared memory.
#pragma once
#include "internal.h"

namespace blco {
namespace {

// Staged ranks: every subgroup's P ranks are followed by one unused entry, so
// that the subgroups of a warp, which read P entries apart, hit different
// banks (without it every record read is a 4-way conflict).
template <int P>
__host__ __device__ constexpr int staged() {
    return kTile + kTile / P;
}
template <int P>
__device__ __forceinline__ uint32_t staged_at(uint32_t r) {
    return r + r / P;
}

}  // namespace
}  // namespace blco
