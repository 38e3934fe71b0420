// The order inside tiles (built once with a resident store): for every mode,
// the nonzeros of each tile of kTile consecutive store positions, stably
// ranked by their target row. Kept per mode: for every store position its rank
// inside the tile (10 bits) and its target row's place among the mode's
// hottest rows (6 bits), and one bit per rank for the last nonzero of a run of
// equal target rows; float64 stores also keep one for the last of a fiber
// (equal target and partner rows, the partner being the longest other mode).
// 2.13 bytes per nonzero and mode (2.25 for float64), next to the store's 12,
// for the modes where run_end_share() is low.
//
// Why: a kernel that orders 32 nonzeros at a time spends 152 of its 410 warp
// instructions per 32 nonzeros on that, and ends a run at 0.34-0.65 of the
// nonzeros (3-mode Zipf shape); in tiles of 1024 runs end at 0.21-0.35 of
// them, fibers at 0.47-0.71, and the order costs the kernel one 2-byte read
// per nonzero (mttkrp_tiled.cuh). Tiles of 4096 would give 0.18-0.22 and
// 0.44-0.64 for four times the staging. Within a run the nonzeros stay in ALTO
// order, which already groups equal partner rows: sorting them by the partner
// as well changed float32 by nothing and float64 by 5 %, putting longer runs
// first gained 0-3 %, and the two took the sort from 3.2 to 11.8 ms for 100M
// nonzeros of three modes.
//
// One warp sorts one tile in registers, 32 words (target | position) per lane,
// by a bitonic network whose strides below 32 stay inside the lane; 32-bit
// words where the mode has at most 2^22 rows (one min or max per compare),
// 64-bit words otherwise. Lane L ends with ranks [32 L, 32 L + 32), which is
// one word of a bit mask. Bound by instruction issue.
#include <algorithm>
#include <cstring>

#include "hot_rows.cuh"
#include "internal.h"

namespace blco {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kOrderWarps = 4;
constexpr int kPosBits = 10;
static_assert(kTile == 1 << kPosBits, "a tile position takes kPosBits bits");
constexpr int kHotLog2 = 7;  // two buckets per hot row
constexpr int kHotBuckets = 1 << kHotLog2;

struct OrderArgs {
    int N;
    int bits[MAXN];
    int partner[MAXN];
    const uint32_t *hot[MAXN];  // hottest rows, by decreasing count
    int nhot[MAXN];             // at most kOrderCold
};

template <typename W>
__device__ __forceinline__ void order2(W &a, W &b, bool up) {
    const W lo = a < b ? a : b, hi = a < b ? b : a;
    a = up ? lo : hi;
    b = up ? hi : lo;
}

// strides 16..1 of a bitonic merge inside each lane
template <typename W>
__device__ __forceinline__ void merge_lane(W (&w)[32], bool up) {
#pragma unroll
    for (int j = 16; j >= 1; j >>= 1)
#pragma unroll
        for (int r = 0; r < 32; ++r)
            if ((r & j) == 0) order2(w[r], w[r | j], up);
}

// ascending bitonic sort of kTile words, element lane * 32 + r in w[r]
template <typename W>
__device__ __forceinline__ void sort_tile(W (&w)[32], int lane) {
#pragma unroll
    for (int k = 2; k <= 16; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j >= 1; j >>= 1)
#pragma unroll
            for (int r = 0; r < 32; ++r)
                if ((r & j) == 0) order2(w[r], w[r | j], (r & k) == 0);
    merge_lane(w, (lane & 1) == 0);
#pragma unroll 1
    for (int k = 2; k <= 32; k <<= 1) {  // lanes per sorted sequence after this step
        const bool up = (lane & k) == 0;
#pragma unroll 1
        for (int j = k >> 1; j >= 1; j >>= 1) {
            const bool keep_min = ((lane & j) == 0) == up;
#pragma unroll
            for (int r = 0; r < 32; ++r) {
                const W o = __shfl_xor_sync(kFull, w[r], j);
                const W lo = o < w[r] ? o : w[r], hi = o < w[r] ? w[r] : o;
                w[r] = keep_min ? lo : hi;
            }
        }
        merge_lane(w, up);
    }
}

// The tile's positions in rank order: lane's ranks 32 L + r. Positions past
// the end (their row is the largest word) sort last, in order.
template <typename W>
__device__ __forceinline__ void rank_tile(const uint32_t *srow, int lane, int nvalid, uint32_t (&pos)[32]) {
    W w[32];
#pragma unroll
    for (int r = 0; r < 32; ++r) {
        const int p = r * 32 + lane;
        w[r] = ((p < nvalid ? (W)srow[p] : ~(W)0) << kPosBits) | (W)p;
    }
    sort_tile(w, lane);
#pragma unroll
    for (int r = 0; r < 32; ++r) pos[r] = (uint32_t)w[r] & (kTile - 1);
}

// Bits of the lane's ranks whose successor has another row in `s`, or none.
__device__ __forceinline__ uint32_t change_bits(const uint32_t (&pos)[32], const uint32_t *s, int lane, int nvalid) {
    uint32_t bits = 0, t = s[pos[0]];
    const uint32_t tn = __shfl_down_sync(kFull, t, 1);
#pragma unroll
    for (int r = 0; r < 32; ++r) {
        const uint32_t t1 = r < 31 ? s[pos[r < 31 ? r + 1 : r]] : tn;
        if (t1 != t || lane * 32 + r == nvalid - 1) bits |= 1u << r;
        t = t1;
    }
    const int live = nvalid - lane * 32;  // none among the positions past the end
    return bits & (live >= 32 ? kFull : (live <= 0 ? 0u : ((1u << live) - 1u)));
}

__global__ void __launch_bounds__(kOrderWarps * 32, 4) k_tile_order(const StoreView sv, const OrderArgs a,
                                                                    const TileOrder to) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint4 *tables = reinterpret_cast<uint4 *>(smem);  // kHotBuckets buckets of two (row, slot) pairs per mode
    uint32_t *rows = reinterpret_cast<uint32_t *>(tables + a.N * kHotBuckets);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t *srow = rows + (size_t)wid * (kTile + kTile / 2);
    uint16_t *srank = reinterpret_cast<uint16_t *>(srow + kTile);
    for (int n = 0; n < a.N; ++n)
        fill_hot_table<kOrderWarps * 32>(tables + n * kHotBuckets, kHotBuckets, kHotLog2, a.hot[n], a.nhot[n], rows);
    const int64_t ntiles = (sv.end + kTile - 1) / kTile;
    for (int64_t tile = (int64_t)blockIdx.x * kOrderWarps + wid; tile < ntiles;
         tile += (int64_t)gridDim.x * kOrderWarps) {
        const int64_t base = tile * kTile;
        const int nvalid = sv.end - base < kTile ? (int)(sv.end - base) : kTile;
        // rows of mode m by position into srow
        const auto stage_rows = [&](int m) {
            __syncwarp();
#pragma unroll 8
            for (int r = 0; r < 32; ++r) {
                const int p = r * 32 + lane;
                uint32_t t = 0;
                if (p < nvalid) {
                    const int64_t q = base + p;
                    t = (uint32_t)((sv.keys[q] >> sv.shift[m]) & sv.mask[m]);
                    if (!sv.single_block) {
                        uint32_t b = sv.tile_block[q >> 5];
                        while (q >= sv.bstart[b + 1]) ++b;
                        t += sv.bbase[(size_t)b * MAXN + m];
                    }
                }
                srow[p] = t;
            }
            __syncwarp();
        };
        for (int n = 0; n < a.N; ++n) {
            if (!to.rank[n]) continue;
            uint32_t pos[32];
            stage_rows(n);
            if (a.bits[n] + kPosBits <= 32)
                rank_tile<uint32_t>(srow, lane, nvalid, pos);
            else
                rank_tile<uint64_t>(srow, lane, nvalid, pos);
            const uint32_t ends = change_bits(pos, srow, lane, nvalid);
            to.ends[n][tile * (kTile / 32) + lane] = ends;
            const uint4 *tb = tables + n * kHotBuckets;
#pragma unroll
            for (int r = 0; r < 32; ++r) {
                const uint32_t t = srow[pos[r]];
                const uint4 bk = tb[hot_hash(t, kHotLog2)];
                const uint32_t slot = bk.x == t ? bk.y : (bk.z == t ? bk.w : (uint32_t)kOrderCold);
                srank[pos[r]] = (uint16_t)((slot << kPosBits) | (uint32_t)(lane * 32 + r));
            }
            if (to.fends[n]) {
                stage_rows(a.partner[n]);
                to.fends[n][tile * (kTile / 32) + lane] = ends | change_bits(pos, srow, lane, nvalid);
            }
            __syncwarp();
            uint32_t *dst = reinterpret_cast<uint32_t *>(to.rank[n] + base);
            const uint32_t *src = reinterpret_cast<const uint32_t *>(srank);
            for (int i = lane; i < kTile / 2; i += 32) dst[i] = src[i];
        }
    }
}

// Distinct rows of mode blockIdx.y in every `step`-th tile (the run ends its order
// would have), added to count[mode]: one CTA per tile and mode, a hash table in
// shared memory four times the tile.
constexpr int kEndsThreads = 256;
constexpr int kEndsSlots = 4 * kTile;
__global__ void __launch_bounds__(kEndsThreads) k_run_ends(const StoreView sv, int64_t step, unsigned long long *count) {
    __shared__ uint32_t seen[kEndsSlots];
    for (int i = threadIdx.x; i < kEndsSlots; i += kEndsThreads) seen[i] = kNoRow;
    __syncthreads();
    const int n = blockIdx.y;
    const int64_t base = (int64_t)blockIdx.x * step * kTile;
    int distinct = 0;
    for (int p = threadIdx.x; p < kTile; p += kEndsThreads) {
        const int64_t q = base + p;
        if (q >= sv.end) break;
        uint32_t t = (uint32_t)((sv.keys[q] >> sv.shift[n]) & sv.mask[n]);
        if (!sv.single_block) {
            uint32_t b = sv.tile_block[q >> 5];
            while (q >= sv.bstart[b + 1]) ++b;
            t += sv.bbase[(size_t)b * MAXN + n];
        }
        uint32_t at = (t * 0x9E3779B1u) >> 20;  // the top 12 bits; the table is never more than a quarter full
        static_assert(kEndsSlots == 1 << 12, "a hash of 12 bits");
        for (;;) {
            const uint32_t was = atomicCAS(&seen[at], kNoRow, t);
            if (was == kNoRow) ++distinct;
            if (was == kNoRow || was == t) break;
            at = (at + 1) & (kEndsSlots - 1);
        }
    }
    distinct = __reduce_add_sync(kFull, distinct);
    if ((threadIdx.x & 31) == 0 && distinct) atomicAdd(count + n, (unsigned long long)distinct);
}

constexpr int64_t kSampleTiles = 512;

size_t mode_bytes(int64_t tiles, bool fibers) {
    return (size_t)tiles * (kTile * sizeof(uint16_t) + (fibers ? 2 : 1) * (kTile / 32) * sizeof(uint32_t));
}

}  // namespace

// The longest other mode (the lowest of equal ones).
int order_partner(const int64_t *dims, int N, int mode) {
    int m = -1;
    for (int k = 0; k < N; ++k)
        if (k != mode && (m < 0 || dims[k] > dims[m])) m = k;
    return m;
}

bool tile_order_supported(const Layout &L) {
    if (L.N < 2) return false;
    for (int n = 0; n < L.N; ++n)
        if (L.dims[n] > ((int64_t)1 << 31)) return false;  // a staged row and its slot share a word
    return true;
}

size_t tile_order_bytes(int64_t nnz, int modes, bool fibers) {
    return (size_t)modes * mode_bytes((nnz + kTile - 1) / kTile, fibers);
}

TileOrder tile_order_view(void *buf, int64_t nnz, const bool *modes, bool fibers) {
    const int64_t tiles = (nnz + kTile - 1) / kTile;
    TileOrder to;
    char *p = static_cast<char *>(buf);
    for (int n = 0; n < MAXN; ++n) {
        if (!modes[n]) continue;
        to.rank[n] = reinterpret_cast<uint16_t *>(p);
        to.ends[n] = reinterpret_cast<uint32_t *>(p + tiles * kTile * sizeof(uint16_t));
        if (fibers) to.fends[n] = to.ends[n] + tiles * (kTile / 32);
        p += mode_bytes(tiles, fibers);
    }
    return to;
}

// Run ends per mode in at most kSampleTiles whole tiles, for run_end_share().
cudaError_t sample_run_ends(const StoreView &sv, unsigned long long *count, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long) * MAXN, s);
    const int64_t tiles = sv.end / kTile;
    if (e != cudaSuccess || tiles == 0) return e;
    const int64_t step = (tiles + kSampleTiles - 1) / kSampleTiles;
    k_run_ends<<<dim3((unsigned)(tiles / step), (unsigned)sv.N), kEndsThreads, 0, s>>>(sv, step, count);
    return cudaGetLastError();
}

// Run ends per nonzero in the sample: whether a mode's runs in tiles are long
// enough for the order to pay. Speed of the tiled kernels over those that order 32
// nonzeros at a time by that share (random shapes of 2 to 8 modes, uniform and
// Zipf, from 2^20 nonzeros, R = 16 / 32 / 64): below 0.3 1.29 / 1.23 / 1.18,
// 0.7-0.8 1.16 / 1.15 / 1.12, 0.96-0.98 1.12 / 1.12 / 1.07, above 1.00 / 0.96 /
// 0.99 (0.83 on 30M uniform nonzeros of 2^22 x 3M x 100k): there nothing merges,
// and the rows gathered in store order share more with their neighbours. So the
// order is kept below 0.98; the same in float64 (1.03 / 1.00 / 0.96 above it) and
// for all modes of a 5-mode store in one pass (0.93 / 0.96 / 0.99), which needs
// every mode's ranks. Float64 below 2^20 nonzeros: 0.7 (from 200k on 1.0-1.3 below
// it, 0.93-1.0 above).
float run_end_share(unsigned long long run_ends, int64_t nnz) {
    const int64_t tiles = nnz / kTile;
    if (tiles == 0) return 1.f;
    const int64_t step = (tiles + kSampleTiles - 1) / kSampleTiles;
    return (float)((double)run_ends / (double)(tiles / step * kTile));
}

cudaError_t build_tile_order(const StoreView &sv, const Layout &L, const HotRows *hot, const TileOrder &to,
                             cudaStream_t s) {
    if (sv.end <= 0 || sv.N < 2) return cudaSuccess;
    OrderArgs a;
    memset(&a, 0, sizeof(a));
    a.N = sv.N;
    for (int n = 0; n < sv.N; ++n) {
        a.bits[n] = L.bits[n];
        a.partner[n] = order_partner(sv.dims, sv.N, n);
        a.hot[n] = hot[n].rows;
        a.nhot[n] = std::min(hot[n].count, kOrderCold);
    }
    const size_t shm = (size_t)sv.N * kHotBuckets * sizeof(uint4) + (size_t)kOrderWarps * kTile * 6;
    cudaError_t e = allow_smem((const void *)k_tile_order, shm);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (sv.end + kTile - 1) / kTile;
    const int64_t grid = std::min<int64_t>((tiles + kOrderWarps - 1) / kOrderWarps, (int64_t)sm_count() * 4);
    k_tile_order<<<(unsigned)grid, kOrderWarps * 32, shm, s>>>(sv, a, to);
    return cudaGetLastError();
}

}  // namespace blco
