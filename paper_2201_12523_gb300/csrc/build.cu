// BLCO construction on the GPU (Section 4, and the construction pipeline of
// Section 6 -- linearize, sort, block, re-encode -- moved from the host CPU
// to the device):
//   k_linearize   ALTO linear index of every nonzero (Section 4.1, Fig. 6a),
//                 range check of every coordinate;
//   radix sort    stable LSD sort of (linear index, input position), 8-bit
//                 digits; per-tile digit counts, one exclusive scan, and a
//                 stable per-tile scatter ranked with warp votes;
//   k_respread    per stored nonzero: the sorted linear index's bits moved to
//                 the in-block key = concatenated per-mode low fields, mode 0
//                 lowest (Fig. 6b), and to the packed block key = bits above
//                 the line; value gathered by input position. Linear indices
//                 of more than 64 bits take k_reencode, which forms the same
//                 from the coordinates;
//   runs/blocks   block boundaries where the block key changes (Section 4.2),
//                 compacted on the device, split at the cap on the host.
#include <cuda.h>

#include <algorithm>
#include <cstring>

#include "internal.h"

namespace blco {

// ---------------------------------------------------------------------------
// host: layout
// ---------------------------------------------------------------------------
bool plan_layout(Layout &L, std::string &why) {
    if (L.N < 1 || L.N > MAXN) {
        why = "order N must be in 1..8";
        return false;
    }
    int maxb = 0;
    L.B = 0;
    for (int n = 0; n < L.N; ++n) {
        if (L.dims[n] < 1 || L.dims[n] > 0xFFFFFFFFll) {
            why = "mode lengths must be in 1..2^32-1";
            return false;
        }
        int b = 0;
        while (b < 32 && ((int64_t)1 << b) < L.dims[n]) ++b;
        L.bits[n] = b;
        L.B += b;
        maxb = std::max(maxb, b);
    }
    if (L.B > 128) {
        why = "more than 128 index bits";
        return false;
    }
    if (L.line < 1 || L.line > 64) {
        why = "line_bits must be in 1..64";
        return false;
    }
    if (L.B - L.line > 64) {
        why = "more than 64 bits above the encoding line";
        return false;
    }
    int pos = 0;
    for (int n = 0; n < L.N; ++n) L.kbits[n] = 0;
    for (int l = 0; l < maxb; ++l)
        for (int n = 0; n < L.N; ++n)
            if (L.bits[n] > l) {
                L.keypos[n][l] = (uint8_t)pos;
                if (pos >= L.line) L.kbits[n]++;
                ++pos;
            }
    int off = 0, boff = 0;
    for (int n = 0; n < L.N; ++n) {
        L.width[n] = L.bits[n] - L.kbits[n];
        L.shift[n] = off;
        off += L.width[n];
        L.boff[n] = boff;
        boff += L.kbits[n];
    }
    return true;
}

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

struct LinArgs {
    int N;
    uint32_t dims_m1[MAXN];  // I_n - 1
    int bits[MAXN];
    int table[MAXN];         // first byte table of mode n
    int ntables;
    uint8_t keypos[MAXN][32];
};

// ---------------------------------------------------------------------------
// ALTO key of every nonzero; lo = key bits 0..63, hi = bits 64..127 (WIDE).
//
// The key is an OR over the bytes of the coordinates: a shared-memory table
// per byte holds where its 8 bits go. Moving the bits one by one took 670 warp
// instructions per 32 nonzeros and 2.7 ms for 100M nonzeros of three modes (54
// bits), bound by the integer pipes; the tables take 0.53 ms,
// bound by their shared-memory reads.
// ---------------------------------------------------------------------------
template <bool WIDE>
__global__ void __launch_bounds__(256) k_linearize(const uint32_t *__restrict__ coords, int64_t nnz, const LinArgs a,
                                                   uint64_t *__restrict__ lo, uint64_t *__restrict__ hi,
                                                   unsigned long long *__restrict__ first_bad) {
    extern __shared__ uint64_t tab[];  // [ntables][256] low words, then high words (WIDE)
    for (int i = threadIdx.x; i < a.ntables * 256; i += blockDim.x) {
        const int t = i >> 8, v = i & 255;
        int n = 0;
        while (n + 1 < a.N && t >= a.table[n + 1]) ++n;
        const int first = (t - a.table[n]) * 8;
        uint64_t l = 0, h = 0;
        for (int k = 0; k < 8 && first + k < a.bits[n]; ++k) {
            const uint64_t bit = (v >> k) & 1;
            const int p = a.keypos[n][first + k];
            if (p < 64)
                l |= bit << p;
            else
                h |= bit << (p - 64);
        }
        tab[i] = l;
        if (WIDE) tab[a.ntables * 256 + i] = h;
    }
    __syncthreads();
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nnz; j += (int64_t)gridDim.x * blockDim.x) {
        uint64_t l = 0, h = 0;
        bool bad = false;
#pragma unroll
        for (int n = 0; n < MAXN; ++n) {
            if (n < a.N) {
                const uint32_t c = coords[j * a.N + n];
                bad |= c > a.dims_m1[n];
                const uint64_t *t = tab + a.table[n] * 256;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    if (b * 8 < a.bits[n]) {
                        const uint32_t v = b * 256 + ((c >> (b * 8)) & 255u);
                        l |= t[v];
                        if (WIDE) h |= t[a.ntables * 256 + v];
                    }
                }
            }
        }
        if (bad) atomicMin(first_bad, (unsigned long long)j);
        lo[j] = l;
        if (WIDE) hi[j] = h;
    }
}

// ---------------------------------------------------------------------------
// exclusive scan of uint32 (in place), any length, recursive over tile sums
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *sh, uint32_t &total) {
    // warp inclusive scan
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t s = lane < (int)(blockDim.x / 32) ? sh[lane] : 0u;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, s, d);
            if (lane >= d) s += y;
        }
        if (lane < (int)(blockDim.x / 32)) sh[lane] = s;
    }
    __syncthreads();
    const uint32_t before = w > 0 ? sh[w - 1] : 0u;
    total = sh[blockDim.x / 32 - 1];
    __syncthreads();
    return before + x - v;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const uint32_t *__restrict__ d, int64_t n,
                                                              uint32_t *__restrict__ sums) {
    __shared__ uint32_t sh[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    uint32_t s = 0;
    for (int i = 0; i < kScanItems; ++i) {
        const int64_t p = base + (int64_t)i * kScanThreads + threadIdx.x;
        if (p < n) s += d[p];
    }
    uint32_t total;
    block_exclusive_scan(s, sh, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_down(uint32_t *__restrict__ d, int64_t n,
                                                            const uint32_t *__restrict__ offs) {
    __shared__ uint32_t sh[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    // blocked arrangement: thread t owns items [t*16, t*16+16)
    uint32_t v[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int64_t p = base + (int64_t)threadIdx.x * kScanItems + i;
        v[i] = p < n ? d[p] : 0u;
        s += v[i];
    }
    uint32_t total;
    uint32_t run = block_exclusive_scan(s, sh, total) + (offs ? offs[blockIdx.x] : 0u);
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int64_t p = base + (int64_t)threadIdx.x * kScanItems + i;
        if (p < n) d[p] = run;
        run += v[i];
    }
}

cudaError_t scan_exclusive(uint32_t *d, int64_t n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int64_t tiles = (n + kScanTile - 1) / kScanTile;
    if (tiles == 1) {
        k_scan_down<<<1, kScanThreads, 0, s>>>(d, n, nullptr);
        return cudaGetLastError();
    }
    uint32_t *sums = nullptr;
    cudaError_t e = cudaMallocAsync(&sums, sizeof(uint32_t) * tiles, s);
    if (e != cudaSuccess) return e;
    k_scan_reduce<<<(unsigned)tiles, kScanThreads, 0, s>>>(d, n, sums);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = scan_exclusive(sums, tiles, s);
    if (e == cudaSuccess) {
        k_scan_down<<<(unsigned)tiles, kScanThreads, 0, s>>>(d, n, sums);
        e = cudaGetLastError();
    }
    cudaFreeAsync(sums, s);
    return e;
}

// ---------------------------------------------------------------------------
// stable LSD radix sort of (key, uint32 value) pairs, 8-bit digits
// ---------------------------------------------------------------------------
constexpr int kRsThreads = 256;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsRounds = 16;
constexpr int kRsTile = kRsThreads * kRsRounds;  // 4096 items

// Lanes with the same 8-bit digit, among the valid ones: one vote per digit bit.
// __match_any_sync takes a time that grows with the number of distinct values:
// with it the scatter of 100M keys took 0.64-0.83 ms by digit, with the votes
// 0.63-0.70.
__device__ __forceinline__ unsigned same_digit(uint32_t dg, bool valid) {
    unsigned peers = __ballot_sync(kFull, valid);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool bit = (dg >> b) & 1u;
        const unsigned v = __ballot_sync(kFull, bit);
        peers &= bit ? v : ~v;
    }
    return peers;
}

// Digit counts of a tile: integer atomics on a histogram per warp, which take a
// cycle per lane with the same digit (grouping the lanes by votes first costs
// 24 instructions for every 32 keys: 0.31 ms for 100M keys, this 0.20).
template <typename K>
__global__ void __launch_bounds__(kRsThreads) k_rs_count(const K *__restrict__ keys, int64_t n, int shift,
                                                         uint32_t *__restrict__ counts, int64_t ntiles) {
    __shared__ uint32_t hist[kRsWarps][256];
    for (int i = threadIdx.x; i < kRsWarps * 256; i += kRsThreads) (&hist[0][0])[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kRsTile;
    uint32_t *h = hist[threadIdx.x >> 5];
#pragma unroll 8
    for (int r = 0; r < kRsRounds; ++r) {
        const int64_t p = base + (int64_t)r * kRsThreads + threadIdx.x;
        if (p < n) atomicAdd(&h[(uint32_t)(keys[p] >> shift) & 0xFFu], 1u);
    }
    __syncthreads();
    uint32_t t = 0;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) t += hist[w][threadIdx.x];
    counts[(int64_t)threadIdx.x * ntiles + blockIdx.x] = t;
}

// Bound by latency, so by the warps in flight: with every item's key, value
// and rank in registers (143 of them) one CTA fitted an SM, and a pass over
// 100M (8 + 4)-byte items took 1.9 ms; with values read only where they are
// staged and two ranks per register three CTAs fit: 0.64-0.83 ms by digit, and
// 0.63-0.70 with the votes of same_digit().
template <typename K>
__global__ void __launch_bounds__(kRsThreads, 3) k_rs_scatter(const K *__restrict__ kin,
                                                              const uint32_t *__restrict__ vin, K *__restrict__ kout,
                                                              uint32_t *__restrict__ vout, int64_t n, int shift,
                                                              const uint32_t *__restrict__ offs, int64_t ntiles) {
    extern __shared__ __align__(16) unsigned char smem[];
    K *sk = reinterpret_cast<K *>(smem);
    uint32_t *sv = reinterpret_cast<uint32_t *>(sk + kRsTile);
    uint32_t *whist = sv + kRsTile;            // [kRsWarps][256]
    uint32_t *tbase = whist + kRsWarps * 256;  // [256]
    uint32_t *gbase = tbase + 256;             // [256] global offset of the digit's run minus tbase
    uint32_t *tmp = gbase + 256;               // [32]

    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * kRsTile;
    const int tile_n = n - base < kRsTile ? (int)(n - base) : kRsTile;
    // warp w ranks items [w*512, w*512+512) of the tile, 32 at a time, in order
    const int it0 = w * (kRsTile / kRsWarps) + lane;
    K kr[kRsRounds];
#pragma unroll
    for (int r = 0; r < kRsRounds; ++r) kr[r] = it0 + r * 32 < tile_n ? kin[base + it0 + r * 32] : (K)0;
    for (int i = threadIdx.x; i < kRsWarps * 256; i += kRsThreads) whist[i] = 0;
    __syncthreads();

    uint32_t rr[kRsRounds / 2];  // ranks, two per word
#pragma unroll
    for (int r = 0; r < kRsRounds; ++r) {
        const bool valid = it0 + r * 32 < tile_n;
        const uint32_t dg = (uint32_t)((kr[r] >> shift) & 0xFFu);
        const unsigned peers = same_digit(dg, valid);
        const int leader = __ffs(peers) - 1;
        const uint32_t prev = whist[w * 256 + dg];
        __syncwarp();
        if (valid && lane == leader) whist[w * 256 + dg] = prev + (uint32_t)__popc(peers);
        __syncwarp();
        const uint32_t rank = prev + (uint32_t)__popc(peers & ((1u << lane) - 1u));
        rr[r / 2] = (r & 1) ? rr[r / 2] | (rank << 16) : rank;
    }
    __syncthreads();
    // per digit: exclusive over warps, and the tile total
    uint32_t total_d;
    {
        const int d = threadIdx.x;  // 256 threads, one per digit
        uint32_t run = 0;
        for (int ww = 0; ww < kRsWarps; ++ww) {
            const uint32_t t = whist[ww * 256 + d];
            whist[ww * 256 + d] = run;
            run += t;
        }
        total_d = run;
    }
    const uint32_t goff = offs[(int64_t)threadIdx.x * ntiles + blockIdx.x];
    __syncthreads();
    uint32_t all;
    const uint32_t excl = block_exclusive_scan(total_d, tmp, all);
    tbase[threadIdx.x] = excl;
    gbase[threadIdx.x] = goff - excl;  // positions are below 2^32; the difference wraps
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRsRounds; ++r) {
        const int it = it0 + r * 32;
        if (it < tile_n) {
            const uint32_t dg = (uint32_t)((kr[r] >> shift) & 0xFFu);
            const uint32_t lp = tbase[dg] + whist[w * 256 + dg] + ((rr[r / 2] >> ((r & 1) * 16)) & 0xFFFFu);
            sk[lp] = kr[r];
            sv[lp] = vin ? vin[base + it] : (uint32_t)(base + it);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < tile_n; i += kRsThreads) {
        const K k = sk[i];
        const uint32_t gp = gbase[(uint32_t)((k >> shift) & 0xFFu)] + (uint32_t)i;
        kout[gp] = k;
        vout[gp] = sv[i];
    }
}

template <typename K>
size_t rs_scatter_smem() {
    return sizeof(K) * kRsTile + sizeof(uint32_t) * kRsTile + sizeof(uint32_t) * (kRsWarps * 256 + 512 + 32);
}

int rs_passes(int nbits) { return (nbits + 7) / 8; }

// Sorts (key, value) pairs by key bits [0, nbits), at least one, in
// rs_passes(nbits) passes that alternate between the two pairs of buffers; the
// result ends in (keys, vals). The keys are read from `keys` after an even
// number of passes' worth, else from `kalt`: key_source() says which. With
// vals_in NULL the values are the positions 0..n-1. `counts` is scratch of
// 256 * ceil(n / kRsTile) words.
template <typename K>
K *key_source(K *keys, K *kalt, int nbits) {
    return (rs_passes(nbits) & 1) ? kalt : keys;
}
template <typename K>
cudaError_t radix_sort_pairs(K *keys, uint32_t *vals, K *kalt, uint32_t *valt, const uint32_t *vals_in, int64_t n,
                             int nbits, uint32_t *counts, cudaStream_t s) {
    const int64_t ntiles = (n + kRsTile - 1) / kRsTile;
    const size_t shm = rs_scatter_smem<K>();
    cudaError_t e = allow_smem((const void *)k_rs_scatter<K>, shm);
    const int passes = rs_passes(nbits);
    K *ki = key_source(keys, kalt, nbits);
    const uint32_t *vi = vals_in;
    for (int i = 0; i < passes && e == cudaSuccess; ++i) {
        const bool to_main = ((passes - i) & 1) != 0;
        K *ko = to_main ? keys : kalt;
        uint32_t *vo = to_main ? vals : valt;
        k_rs_count<K><<<(unsigned)ntiles, kRsThreads, 0, s>>>(ki, n, 8 * i, counts, ntiles);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = scan_exclusive(counts, 256 * ntiles, s);
        if (e == cudaSuccess) {
            k_rs_scatter<K><<<(unsigned)ntiles, kRsThreads, shm, s>>>(ki, vi, ko, vo, n, 8 * i, counts, ntiles);
            e = cudaGetLastError();
        }
        ki = ko;
        vi = vo;
    }
    return e;
}

// ---------------------------------------------------------------------------
// gathers and re-encoding
// ---------------------------------------------------------------------------
__global__ void k_gather_u64(const uint64_t *__restrict__ src, const uint32_t *__restrict__ idx, int64_t n,
                             uint64_t *__restrict__ dst) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
        dst[j] = src[idx[j]];
}

struct EncArgs {
    int N;
    int has_blocks;
    uint32_t lowmask[MAXN];
    int shift[MAXN];
    int width[MAXN];
    int boff[MAXN];
};

__global__ void k_reencode(const uint32_t *__restrict__ coords, const float *__restrict__ vals,
                           const uint32_t *__restrict__ perm, int64_t nnz, const EncArgs a,
                           uint64_t *__restrict__ skeys, float *__restrict__ svals,
                           uint64_t *__restrict__ bkey) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nnz;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = perm[j];
        uint64_t key = 0, bk = 0;
#pragma unroll
        for (int n = 0; n < MAXN; ++n) {
            if (n < a.N) {
                const uint32_t c = coords[p * a.N + n];
                key |= (uint64_t)(c & a.lowmask[n]) << a.shift[n];
                if (a.has_blocks) bk |= (a.width[n] >= 32 ? 0ull : (uint64_t)(c >> a.width[n])) << a.boff[n];
            }
        }
        skeys[j] = key;
        svals[j] = vals ? vals[p] : 0.f;  // no float32 values: a float64 store gathers its own
        if (a.has_blocks) bkey[j] = bk;
    }
}

// Where the bits of a linear index of at most 64 bits go: byte b's tables are
// key[b][256], and, for stores with block-key bits, bkey[b][256].
struct SpreadArgs {
    int nbytes;
    int has_blocks;
    uint8_t to[64];  // destination of linear-index bit p: key bit, or 64 + block-key bit
};

// In-block key, block key and value of every stored nonzero from the sorted
// linear indices (`lin` may be `skeys`). Reading the coordinates by input
// position instead (k_reencode) took 4.4 ms for 100M nonzeros of three modes,
// a random 12-byte read each; this takes 2.1, most of it the values'.
template <bool BLOCKS>
__global__ void __launch_bounds__(256) k_respread(const uint64_t *lin, const float *__restrict__ vals,
                                                  const uint32_t *__restrict__ perm, int64_t nnz, const SpreadArgs a,
                                                  uint64_t *skeys, float *__restrict__ svals,
                                                  uint64_t *__restrict__ bkey) {
    extern __shared__ uint64_t tab[];
    for (int i = threadIdx.x; i < a.nbytes * 256; i += blockDim.x) {
        uint64_t k = 0, b = 0;
        for (int j = 0; j < 8; ++j) {
            const int to = a.to[((i >> 8) * 8 + j) & 63];
            const uint64_t bit = (i >> j) & 1;
            if (to < 64)
                k |= bit << to;
            else if (to < 128)
                b |= bit << (to - 64);
        }
        tab[i] = k;
        if (BLOCKS) tab[a.nbytes * 256 + i] = b;
    }
    __syncthreads();
    // four elements per thread in flight: the values are random reads
    constexpr int U = 4;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j0 < nnz; j0 += U * step) {
        uint64_t l[U];
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t j = j0 + u * step;
            l[u] = j < nnz ? lin[j] : 0ull;
            v[u] = j < nnz && vals ? vals[perm[j]] : 0.f;  // no float32 values: a float64 store gathers its own
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t j = j0 + u * step;
            uint64_t key = 0, bk = 0;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                if (b < a.nbytes) {
                    const int t = b * 256 + (int)((l[u] >> (8 * b)) & 255u);
                    key |= tab[t];
                    if (BLOCKS) bk |= tab[a.nbytes * 256 + t];
                }
            }
            if (j < nnz) {
                skeys[j] = key;
                svals[j] = v[u];
                if (BLOCKS) bkey[j] = bk;
            }
        }
    }
}

__global__ void k_gather_f64(const double *__restrict__ src, const uint32_t *__restrict__ perm, int64_t nnz,
                             double *__restrict__ dst) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nnz; j += (int64_t)gridDim.x * blockDim.x)
        dst[j] = src[perm[j]];
}

__global__ void k_run_flags(const uint64_t *__restrict__ bkey, int64_t n, uint32_t *__restrict__ flags) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
        flags[j] = (j == 0 || bkey[j] != bkey[j - 1]) ? 1u : 0u;
}

__global__ void k_run_compact(const uint64_t *__restrict__ bkey, const uint32_t *__restrict__ scanned,
                              int64_t n, int64_t *__restrict__ starts, uint64_t *__restrict__ keys_out) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        if (j == 0 || bkey[j] != bkey[j - 1]) {
            const uint32_t r = scanned[j];
            starts[r] = j;
            keys_out[r] = bkey[j];
        }
    }
}

__global__ void k_tile_block(const int64_t *__restrict__ bstart, int64_t nblocks, int64_t ntiles,
                             uint32_t *__restrict__ tb) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ntiles; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t pos = t * 32;
        // last block b with bstart[b] <= pos
        int64_t lo = 0, hi = nblocks - 1;
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (bstart[mid] <= pos)
                lo = mid;
            else
                hi = mid - 1;
        }
        tb[t] = (uint32_t)lo;
    }
}

// Row counts of one mode over a systematic sample of the store: every
// `stride`-th 32-nonzero tile (all tiles when stride is 1), one warp per
// sampled tile. The counts only rank rows for on-chip accumulation, so a
// sample of tens of millions of nonzeros is enough to find the heavy rows.
// Short modes (SMEM) count in shared memory first: a 2048-row mode of 100M
// nonzeros took 1.6 ms with all atomics on the same few rows in L2, 0.27 so.
constexpr int kHistRows = 8192;

template <bool SMEM>
__global__ void k_histogram(const StoreView sv, int mode, int64_t stride, uint32_t *__restrict__ counts) {
    extern __shared__ uint32_t local[];
    const int nrows = (int)sv.dims[mode];  // used where SMEM: at most kHistRows
    if (SMEM) {
        for (int i = threadIdx.x; i < nrows; i += blockDim.x) local[i] = 0;
        __syncthreads();
    }
    const int64_t ntiles = (sv.end - sv.begin + 31) >> 5;
    const int64_t nsamp = (ntiles + stride - 1) / stride;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // the loop bound is uniform over the warp, so whole warps iterate together
    for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < nsamp; j += nwarps) {
        const int64_t pos = sv.begin + j * stride * 32 + lane;
        const bool live = pos < sv.end;
        uint32_t row = 0;
        if (live) {
            const uint64_t key = sv.keys[pos - sv.key_origin];
            uint32_t base = 0;
            if (!sv.single_block) {
                uint32_t b = sv.tile_block[pos >> 5];
                while (pos >= sv.bstart[b + 1]) ++b;
                base = sv.bbase[(size_t)b * MAXN + mode];
            }
            row = (uint32_t)((key >> sv.shift[mode]) & sv.mask[mode]) + base;
        }
        const unsigned lanes = __ballot_sync(0xFFFFFFFFu, live);
        if (live) {
            const unsigned peers = __match_any_sync(lanes, row);
            if (lane == __ffs(peers) - 1) atomicAdd(SMEM ? &local[row] : &counts[row], (uint32_t)__popc(peers));
        }
    }
    if (SMEM) {
        __syncthreads();
        for (int i = threadIdx.x; i < nrows; i += blockDim.x)
            if (local[i]) atomicAdd(&counts[i], local[i]);
    }
}

__global__ void k_complement(const uint32_t *__restrict__ counts, int64_t I, uint32_t *__restrict__ key) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < I; i += (int64_t)gridDim.x * blockDim.x)
        key[i] = ~counts[i];  // ascending sort of ~count = descending count
}

unsigned grid_for(int64_t n, int threads) {
    int64_t g = (n + threads - 1) / threads;
    const int64_t cap = (int64_t)sm_count() * 16;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (unsigned)g;
}

// Grid of a kernel whose CTAs begin by filling byte tables: few enough CTAs
// that each has many elements to amortize that over.
unsigned table_grid(int64_t n) {
    const int64_t need = (n + 2047) / 2048;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)sm_count() * 8));
}

}  // namespace

// ---------------------------------------------------------------------------
// Scratch of one construction. It goes back without waiting for other streams'
// work, as cudaFree would: a program that builds a store beside a running
// training step is not held up. Blocks of more than 32 MB are mapped by
// themselves (alloc + release of 0.8 GB: 0.11 + 0.33 ms); memory of the default
// stream-ordered pool is returned to the device at the next synchronization and
// takes 0.66 + 1.17 ms, and at 32 MB and less its fixed cost is the smaller one.
// ---------------------------------------------------------------------------
namespace {

struct MapApi {
    decltype(&cuMemAddressReserve) reserve = nullptr;
    decltype(&cuMemAddressFree) unreserve = nullptr;
    decltype(&cuMemCreate) create = nullptr;
    decltype(&cuMemRelease) release = nullptr;
    decltype(&cuMemMap) map = nullptr;
    decltype(&cuMemUnmap) unmap = nullptr;
    decltype(&cuMemSetAccess) set_access = nullptr;
    decltype(&cuMemGetAllocationGranularity) granularity = nullptr;
    bool ok = true;

    template <typename F>
    void find(const char *name, F &f) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !p) {
            cudaGetLastError();
            ok = false;
        }
        f = reinterpret_cast<F>(p);
    }
    MapApi() {
        find("cuMemAddressReserve", reserve);
        find("cuMemAddressFree", unreserve);
        find("cuMemCreate", create);
        find("cuMemRelease", release);
        find("cuMemMap", map);
        find("cuMemUnmap", unmap);
        find("cuMemSetAccess", set_access);
        find("cuMemGetAllocationGranularity", granularity);
    }
};

const MapApi &map_api() {
    static const MapApi api;
    return api;
}

class Scratch {
  public:
    // `bytes` of device memory, usable on `s` until release().
    template <typename T>
    cudaError_t get(T **out, size_t bytes, cudaStream_t s) {
        if (bytes > ((size_t)32 << 20) && map_api().ok) {
            CUdeviceptr va = 0;
            size_t len = 0;
            if (map_block(bytes, &va, &len)) {
                *out = reinterpret_cast<T *>(va);
                mapped_.push_back({va, len});
                return cudaSuccess;
            }
        }  // no room: the pool may hold memory that it can reuse
        void *p = nullptr;
        const cudaError_t e = cudaMallocAsync(&p, bytes, s);
        if (e != cudaSuccess) return e;
        *out = static_cast<T *>(p);
        pooled_.push_back(p);
        return cudaSuccess;
    }
    // Gives everything back; returns when the work on `s` is complete.
    cudaError_t release(cudaStream_t s) {
        for (void *p : pooled_) cudaFreeAsync(p, s);
        const cudaError_t e = cudaStreamSynchronize(s);
        for (const Block &b : mapped_) {
            map_api().unmap(b.va, b.len);
            map_api().unreserve(b.va, b.len);
        }
        pooled_.clear();
        mapped_.clear();
        return e;
    }

  private:
    struct Block {
        CUdeviceptr va;
        size_t len;
    };
    static bool map_block(size_t bytes, CUdeviceptr *va, size_t *len) {
        const MapApi &api = map_api();
        CUmemAllocationProp prop = {};
        prop.type = CU_MEM_ALLOCATION_TYPE_PINNED;
        prop.location.type = CU_MEM_LOCATION_TYPE_DEVICE;
        if (cudaGetDevice(&prop.location.id) != cudaSuccess) return false;
        size_t unit = 0;
        if (api.granularity(&unit, &prop, CU_MEM_ALLOC_GRANULARITY_RECOMMENDED) != CUDA_SUCCESS || unit == 0) return false;
        *len = (bytes + unit - 1) / unit * unit;
        CUmemGenericAllocationHandle mem = 0;
        if (api.create(&mem, *len, &prop, 0) != CUDA_SUCCESS) return false;
        bool done = false;
        if (api.reserve(va, *len, 0, 0, 0) == CUDA_SUCCESS) {
            if (api.map(*va, *len, 0, mem, 0) == CUDA_SUCCESS) {
                CUmemAccessDesc access = {};
                access.location = prop.location;
                access.flags = CU_MEM_ACCESS_FLAGS_PROT_READWRITE;
                done = api.set_access(*va, *len, &access, 1) == CUDA_SUCCESS;
                if (!done) api.unmap(*va, *len);
            }
            if (!done) api.unreserve(*va, *len);
        }
        api.release(mem);  // the mapping keeps it
        return done;
    }
    std::vector<Block> mapped_;
    std::vector<void *> pooled_;
};

}  // namespace

// ---------------------------------------------------------------------------
cudaError_t build_store(const Layout &L, const uint32_t *coords, const float *vals, int64_t nnz, int64_t cap,
                        BuildOut &out, cudaStream_t s, std::string &why) {
    cudaError_t e = cudaSuccess;
    const int64_t npad = ((nnz + 31) / 32) * 32 + 32;
    const int64_t nbits = std::min(std::max(L.B, 1), 64);  // sorted low bits (a length-1 shape has none: one pass)
    uint64_t *lo = nullptr, *hi = nullptr, *hi2 = nullptr, *bkey = nullptr;
    uint64_t *d_rkeys = nullptr;
    uint32_t *idx = nullptr, *idx2 = nullptr, *counts = nullptr, *flags = nullptr;
    unsigned long long *d_bad = nullptr;
    const bool wide = L.B > 64;
    const bool has_blocks = L.B > L.line;
    Scratch scratch;
#define TRY(x)                      \
    do {                            \
        e = (x);                    \
        if (e != cudaSuccess) goto done; \
    } while (0)
    // The store's own arrays serve as one half of the sort's buffers (keys and
    // positions; the values' array, filled last, holds the other positions);
    // only the second key buffer is scratch.
    TRY(cudaMalloc(&out.keys, sizeof(uint64_t) * npad));
    TRY(cudaMalloc(&out.vals, sizeof(float) * npad));
    TRY(cudaMalloc(&out.perm, sizeof(uint32_t) * (nnz > 0 ? nnz : 1)));
    TRY(cudaMemsetAsync(out.keys + nnz, 0, sizeof(uint64_t) * (npad - nnz), s));
    TRY(cudaMemsetAsync(out.vals + nnz, 0, sizeof(float) * (npad - nnz), s));
    if (nnz > 0) {
        const int64_t ntiles = (nnz + kRsTile - 1) / kRsTile;
        TRY(scratch.get(&lo, sizeof(uint64_t) * nnz, s));
        TRY(scratch.get(&counts, sizeof(uint32_t) * 256 * ntiles, s));
        TRY(scratch.get(&d_bad, sizeof(unsigned long long), s));
        TRY(cudaMemsetAsync(d_bad, 0xFF, sizeof(unsigned long long), s));
        idx = out.perm;
        idx2 = reinterpret_cast<uint32_t *>(out.vals);
        if (wide) {
            TRY(scratch.get(&hi, sizeof(uint64_t) * nnz, s));
            TRY(scratch.get(&hi2, sizeof(uint64_t) * nnz, s));
        }
        {
            LinArgs a;
            memset(&a, 0, sizeof(a));
            a.N = L.N;
            for (int n = 0; n < L.N; ++n) {
                a.dims_m1[n] = (uint32_t)(L.dims[n] - 1);
                a.bits[n] = L.bits[n];
                a.table[n] = a.ntables;
                a.ntables += (L.bits[n] + 7) / 8;
                memcpy(a.keypos[n], L.keypos[n], 32);
            }
            uint64_t *src = key_source(out.keys, lo, (int)nbits);
            const size_t shm = (size_t)a.ntables * 256 * sizeof(uint64_t) * (wide ? 2 : 1);
            if (wide) {
                TRY(allow_smem((const void *)k_linearize<true>, shm));
                k_linearize<true><<<table_grid(nnz), 256, shm, s>>>(coords, nnz, a, src, hi, d_bad);
            } else {
                k_linearize<false><<<table_grid(nnz), 256, shm, s>>>(coords, nnz, a, src, nullptr, d_bad);
            }
            TRY(cudaGetLastError());
        }
        {
            unsigned long long bad = 0;
            TRY(cudaMemcpyAsync(&bad, d_bad, sizeof(bad), cudaMemcpyDeviceToHost, s));
            TRY(cudaStreamSynchronize(s));
            if (bad != ~0ull) {
                out.first_bad = (int64_t)bad;
                why = "coordinate row " + std::to_string((long long)bad) + " is out of range";
                goto done;
            }
        }
        // sort by the low word, then (stably) by the high word
        TRY(radix_sort_pairs<uint64_t>(out.keys, idx, lo, idx2, nullptr, nnz, (int)nbits, counts, s));
        if (wide) {
            k_gather_u64<<<grid_for(nnz, 256), 256, 0, s>>>(hi, idx, nnz, hi2);
            TRY(cudaGetLastError());
            // an odd number of passes reads from its second key buffer and
            // ends in its first: hi2 is the source either way; the positions
            // start in idx, so they may not be the first pass's output
            const bool odd = (rs_passes(L.B - 64) & 1) != 0;
            if (odd) {
                TRY(cudaMemcpyAsync(idx2, idx, sizeof(uint32_t) * nnz, cudaMemcpyDeviceToDevice, s));
                TRY(radix_sort_pairs<uint64_t>(hi, idx, hi2, idx2, idx2, nnz, L.B - 64, counts, s));
            } else {
                TRY(radix_sort_pairs<uint64_t>(hi2, idx, hi, idx2, idx, nnz, L.B - 64, counts, s));
            }
        }
        if (has_blocks) TRY(scratch.get(&bkey, sizeof(uint64_t) * nnz, s));
        if (wide) {
            EncArgs a;
            memset(&a, 0, sizeof(a));
            a.N = L.N;
            a.has_blocks = has_blocks ? 1 : 0;
            for (int n = 0; n < L.N; ++n) {
                a.lowmask[n] = L.width[n] >= 32 ? 0xFFFFFFFFu : ((1u << L.width[n]) - 1u);
                a.shift[n] = L.shift[n];
                a.width[n] = L.width[n];
                a.boff[n] = L.boff[n];
            }
            k_reencode<<<grid_for(nnz, 256), 256, 0, s>>>(coords, vals, idx, nnz, a, out.keys, out.vals, bkey);
        } else {
            SpreadArgs a;
            memset(&a, 0, sizeof(a));
            a.nbytes = (L.B + 7) / 8;
            a.has_blocks = has_blocks ? 1 : 0;
            memset(a.to, 0xFF, sizeof(a.to));  // no such bit
            for (int n = 0; n < L.N; ++n)
                for (int l = 0; l < L.bits[n]; ++l)
                    a.to[L.keypos[n][l]] =
                        (uint8_t)(l < L.width[n] ? L.shift[n] + l : 64 + L.boff[n] + (l - L.width[n]));
            const size_t shm = (size_t)a.nbytes * 256 * sizeof(uint64_t) * (has_blocks ? 2 : 1);
            if (has_blocks)
                k_respread<true><<<table_grid(nnz), 256, shm, s>>>(out.keys, vals, idx, nnz, a, out.keys, out.vals, bkey);
            else
                k_respread<false><<<table_grid(nnz), 256, shm, s>>>(out.keys, vals, idx, nnz, a, out.keys, out.vals, bkey);
        }
        TRY(cudaGetLastError());
    }
    // block runs
    {
        std::vector<int64_t> run_start;
        std::vector<uint64_t> run_key;
        if (nnz > 0 && has_blocks) {
            TRY(scratch.get(&flags, sizeof(uint32_t) * nnz, s));
            k_run_flags<<<grid_for(nnz, 256), 256, 0, s>>>(bkey, nnz, flags);
            TRY(cudaGetLastError());
            uint32_t last_flag = 0;
            TRY(cudaMemcpyAsync(&last_flag, flags + nnz - 1, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
            TRY(scan_exclusive(flags, nnz, s));
            uint32_t last_scan = 0;
            TRY(cudaMemcpyAsync(&last_scan, flags + nnz - 1, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
            TRY(cudaStreamSynchronize(s));
            const int64_t nruns = (int64_t)last_scan + last_flag;
            int64_t *d_starts = reinterpret_cast<int64_t *>(lo);  // reuse: nruns <= nnz
            TRY(scratch.get(&d_rkeys, sizeof(uint64_t) * nruns, s));
            k_run_compact<<<grid_for(nnz, 256), 256, 0, s>>>(bkey, flags, nnz, d_starts, d_rkeys);
            TRY(cudaGetLastError());
            run_start.resize(nruns);
            run_key.resize(nruns);
            TRY(cudaMemcpyAsync(run_start.data(), d_starts, sizeof(int64_t) * nruns, cudaMemcpyDeviceToHost, s));
            TRY(cudaMemcpyAsync(run_key.data(), d_rkeys, sizeof(uint64_t) * nruns, cudaMemcpyDeviceToHost, s));
            TRY(cudaStreamSynchronize(s));
        } else if (nnz > 0) {
            run_start.push_back(0);
            run_key.push_back(0);
        }
        // split runs at the cap: pieces of ceil(c / ceil(c / cap)) entries
        out.bstart.clear();
        out.bhigh.clear();
        for (size_t r = 0; r < run_start.size(); ++r) {
            const int64_t a = run_start[r];
            const int64_t b = (r + 1 < run_start.size()) ? run_start[r + 1] : nnz;
            const int64_t cnt = b - a;
            const int64_t pieces = (cnt + cap - 1) / cap;
            const int64_t piece = (cnt + pieces - 1) / pieces;
            for (int64_t p = a; p < b; p += piece) {
                out.bstart.push_back(p);
                for (int n = 0; n < L.N; ++n) {
                    const uint64_t m = L.kbits[n] >= 64 ? ~0ull : ((1ull << L.kbits[n]) - 1ull);
                    out.bhigh.push_back((uint32_t)((run_key[r] >> L.boff[n]) & m));
                }
            }
        }
        out.bstart.push_back(nnz);
    }
done:
#undef TRY
    {
        const cudaError_t es = scratch.release(s);
        if (e == cudaSuccess) e = es;
    }
    return e;
}

cudaError_t gather_f64(const double *src, const uint32_t *perm, int64_t nnz, double *dst, cudaStream_t s) {
    if (nnz <= 0) return cudaSuccess;
    k_gather_f64<<<grid_for(nnz, 256), 256, 0, s>>>(src, perm, nnz, dst);
    return cudaGetLastError();
}

cudaError_t build_tile_block(const int64_t *d_bstart, int64_t nblocks, int64_t nnz, uint32_t *tile_block,
                             cudaStream_t s) {
    const int64_t ntiles = (nnz + 31) / 32;
    if (ntiles == 0) return cudaSuccess;
    k_tile_block<<<grid_for(ntiles, 256), 256, 0, s>>>(d_bstart, nblocks, ntiles, tile_block);
    return cudaGetLastError();
}

cudaError_t mode_histogram(const StoreView &sv, int mode, uint32_t *counts, cudaStream_t s) {
    if (sv.end <= sv.begin) return cudaSuccess;
    const int64_t ntiles = (sv.end - sv.begin + 31) / 32;
    const int64_t stride = std::max<int64_t>(1, ntiles >> 20);  // at most ~2^20 sampled tiles
    const int64_t nsamp = (ntiles + stride - 1) / stride;
    if (sv.dims[mode] <= kHistRows)
        k_histogram<true><<<grid_for(nsamp * 32, 256), 256, sizeof(uint32_t) * sv.dims[mode], s>>>(sv, mode, stride, counts);
    else
        k_histogram<false><<<grid_for(nsamp * 32, 256), 256, 0, s>>>(sv, mode, stride, counts);
    return cudaGetLastError();
}

cudaError_t top_rows(const uint32_t *counts, int64_t I, int k, int64_t most, uint32_t *rows_out, cudaStream_t s) {
    int nbits = 1;  // of the largest count: above them every complemented count is all ones
    while (nbits < 32 && (most >> nbits) > 0) ++nbits;
    uint32_t *key = nullptr, *row = nullptr, *key2 = nullptr, *row2 = nullptr, *tiles = nullptr;
    const int64_t ntiles = (I + kRsTile - 1) / kRsTile;
    cudaError_t e = cudaMallocAsync(&key, sizeof(uint32_t) * I, s);
    if (e == cudaSuccess) e = cudaMallocAsync(&row, sizeof(uint32_t) * I, s);
    if (e == cudaSuccess) e = cudaMallocAsync(&key2, sizeof(uint32_t) * I, s);
    if (e == cudaSuccess) e = cudaMallocAsync(&row2, sizeof(uint32_t) * I, s);
    if (e == cudaSuccess) e = cudaMallocAsync(&tiles, sizeof(uint32_t) * 256 * ntiles, s);
    if (e == cudaSuccess) {
        k_complement<<<grid_for(I, 256), 256, 0, s>>>(counts, I, key_source(key, key2, nbits));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = radix_sort_pairs<uint32_t>(key, row, key2, row2, nullptr, I, nbits, tiles, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(rows_out, row, sizeof(uint32_t) * std::min<int64_t>(k, I), cudaMemcpyDeviceToDevice, s);
    for (uint32_t *b : {key, row, key2, row2, tiles})
        if (b) cudaFreeAsync(b, s);
    return e;
}

}  // namespace blco
