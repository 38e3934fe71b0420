// Sparse MTTKRP (Eq. 1) of a whole resident store that has its tile order
// (tile_order.cu): one CTA per tile of kTile consecutive store positions.
//
//   1. The CTA reads the tile's keys, values and ranks (coalesced), decodes
//      every nonzero's rows and scatters a record to its rank in shared
//      memory: no sort, no search for the row's on-chip copy per nonzero. One
//      thread prefetches the arrays of the CTA's next tile into L2, so that
//      the loads that open a tile do not wait for DRAM.
//   2. Subgroups of G lanes walk R consecutive ranks each, gather the other
//      modes' rows (4 elements per lane and load) and keep the run's sum.
//   3. Where a run (equal target rows) ends inside the subgroup's ranks, its
//      sum goes to the CTA's shared-memory copy of the row if the row is one
//      of the mode's hottest, else to global memory with
//      red.global.add.v4.f32. A row has one run per tile, so the subgroup
//      that holds its end is the only one to update the copy: a plain
//      read-modify-write. The part of a run that goes on in the next
//      subgroup's ranks is added after the CTA's barrier, where only such
//      parts meet, with atomics.
//   The CTA adds its copies to the output once, at its end.
//
// Bound by the L1 data pipe, where a gathered row costs a wavefront per 128
// bytes whether it hits or not: 3.8 wavefronts per nonzero at 3 modes and
// R = 32 (2 of them gathers), 73 % of the pipe's rate. Against the kernel that
// sorts 32 nonzeros at a time (mttkrp_kernels.cuh): 328 warp instructions per
// 32 nonzeros instead of 410, 3.8 wavefronts instead of 4.8 (40M nonzeros, mode
// 0); float32, sum of the per-mode launches: 3 modes, 150M nonzeros, R = 32:
// 9.09 -> 7.47 ms; 4 modes, 100M, R = 32: 9.37 -> 8.75;
// 3 modes, 50M, R = 64: 4.75 -> 4.22; 5 modes, 50M, R = 16: 7.66 -> 5.47.
// Without the prefetch 11 % slower at 3 modes. Measured and not kept: 512
// threads per CTA (25 % slower: longer waits at the barrier), 5 or 6 CTAs per
// SM and 4 ranks per load batch (no faster), the 32 hottest gathered rows in
// shared memory (35 % slower: two predicated loads per row), and gathering the
// partner's row once per fiber (10 % slower: a fiber's end is predicated work
// in all four subgroups of a warp; it pays for float64, below).
#pragma once
#include <cooperative_groups.h>

#include <algorithm>

#include "mttkrp_kernels.cuh"
#include "tile_stage.cuh"

namespace blco {
namespace {

constexpr int kTiledThreads = 256;
// Shared-memory copies of the hottest rows, one set per CTA.
constexpr int kTiledHotBytes = 8 * 1024;
// The CTAs of a cluster sum their copies before one of them adds a row's sum to
// the output: the additions there, one per cluster, made most of a hot row's
// rounding error. Pairs halve them at no cost (7.46 and 7.48 ms for the 3-mode
// sum above); clusters of 4 or 8 leave SM slots of a GPC unused (7.72, 8.42).
constexpr int kTiledCluster = 2;
// A staged target row: the row, or the slot of its on-chip copy with this bit.
constexpr uint32_t kSlotBit = 0x80000000u;

struct TParams {
    const uint64_t *keys;
    const float *vals;
    const double *vals64;
    int vals_aligned;  // the values start on a 16-byte boundary
    int64_t nnz;
    const uint32_t *tile_block;
    const int64_t *bstart;
    const uint32_t *bbase;
    int single_block;
    const uint16_t *rank;
    const uint32_t *ends;
    const uint32_t *fends;
    int n_inner;             // gathered modes besides the partner
    Gather gat[kMaxGather];  // the inner modes
    Gather par;              // the partner
    uint64_t t_mask;
    int t_shift;
    int t_mode;
    void *out;
    int ncopies;
    int64_t copy_stride;
    const uint32_t *hot_rows;
    int kw;  // rows with an on-chip copy
};

__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

template <int NG>
__host__ __device__ constexpr int inner_slots() {
    return NG > 0 ? NG - 1 : kMaxGather - 2;  // at most MAXN - 2 inner modes
}

// Shared memory of a CTA: a record per rank, `words` further words per rank,
// the copies of the hottest target rows.
struct TiledSmem {
    size_t extra, hot, total;
};
__host__ __device__ __forceinline__ TiledSmem tiled_smem(size_t rec_bytes, int entries, int words, int kw,
                                                         size_t row_bytes) {
    TiledSmem L;
    L.extra = rec_bytes * entries;
    L.hot = align16(L.extra + (size_t)words * entries * sizeof(uint32_t));
    L.total = L.hot + (size_t)kw * row_bytes;
    return L;
}

// Decodes the tile's nonzeros and scatters them to their ranks: put(rank,
// valid, index in the tile, first inner row, partner's row, target row or
// slot) stores the record, further inner rows go to `extra`.
template <int NI, int P, typename Put>
__device__ __forceinline__ void stage_tile(const TParams &p, int64_t base, int nvalid, int ni, Put &&put,
                                           uint32_t *extra) {
    constexpr int PER = kTile / kTiledThreads;
    uint64_t key[PER];
    uint32_t rk[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int q = threadIdx.x + i * kTiledThreads;
        key[i] = q < nvalid ? ld_stream_u64(p.keys + base + q) : 0ull;
        rk[i] = __ldcs(p.rank + base + q);  // written for the whole tile
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int q = threadIdx.x + i * kTiledThreads;
        const bool valid = q < nvalid;
        uint32_t t = (uint32_t)((key[i] >> p.t_shift) & p.t_mask);
        uint32_t k = (uint32_t)((key[i] >> p.par.shift) & p.par.mask);
        uint32_t o[NI > 0 ? NI : 1];
#pragma unroll
        for (int j = 0; j < NI; ++j)
            o[j] = j < ni ? (uint32_t)((key[i] >> p.gat[j].shift) & p.gat[j].mask) : 0u;
        if (!p.single_block && valid) {
            const int64_t pos = base + q;
            uint32_t b = __ldg(p.tile_block + (pos >> 5));
            while (pos >= __ldg(p.bstart + b + 1)) ++b;
            const uint32_t *bb = p.bbase + (size_t)b * MAXN;
            t += __ldg(bb + p.t_mode);
            k += __ldg(bb + p.par.mode);
#pragma unroll
            for (int j = 0; j < NI; ++j)
                if (j < ni) o[j] += __ldg(bb + p.gat[j].mode);
        }
        // positions past the end: row 0 of every factor (every mode has one)
        // and value 0, at ranks whose sums are never stored
        const uint32_t r = staged_at<P>(rk[i] & (kTile - 1)), slot = rk[i] / kTile;
        put(r, valid, q, o[0], k, slot < (uint32_t)p.kw ? kSlotBit | slot : t);
#pragma unroll
        for (int j = 1; j < NI; ++j)
            if (j < ni) extra[(j - 1) * staged<P>() + r] = o[j];
    }
}

// Asks for the arrays of a later, full tile in L2 (one thread of the CTA).
__device__ __forceinline__ void prefetch_tile(const TParams &p, int64_t tile, int64_t ntiles, const void *vals,
                                              int val_bytes) {
    if (threadIdx.x != 0 || tile >= ntiles - 1) return;
    const auto ask = [](const void *a, int bytes) {
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"(bytes));
    };
    ask(p.keys + tile * kTile, kTile * (int)sizeof(uint64_t));
    if (p.vals_aligned) ask(static_cast<const char *>(vals) + tile * kTile * val_bytes, kTile * val_bytes);
    ask(p.rank + tile * kTile, kTile * (int)sizeof(uint16_t));
    ask(p.ends + tile * (kTile / 32), kTile / 8);
}

// Resident CTAs per SM the register budget is sized for.
template <int R, int NG>
__host__ __device__ constexpr int tiled_min_ctas() {
    return NG == 0 || R > 64 ? 3 : 4;
}

template <typename T, int R, int NG>
__global__ void __launch_bounds__(kTiledThreads, tiled_min_ctas<R, NG>()) k_mttkrp_tiled(const TParams p) {
    constexpr int VEC = lane_vec<T, R>();
    constexpr int H = VEC / 2;
    constexpr int G = R / VEC;
    constexpr int SUBS = kTiledThreads / G;
    constexpr int P = kTile / SUBS;  // ranks per subgroup
    constexpr int PB = P < 32 ? P : 32;
    constexpr int CH = 2;  // ranks whose row loads are issued back to back
    constexpr int NI = inner_slots<NG>();
    static_assert(VEC == 4 && P % PB == 0 && PB % CH == 0, "four elements per lane");

    extern __shared__ __align__(16) unsigned char smem[];
    const int ni = NG > 0 ? NG - 1 : p.n_inner;
    const TiledSmem L = tiled_smem(sizeof(uint4), staged<P>(), ni > 1 ? ni - 1 : 0, p.kw, R * sizeof(float));
    uint4 *rec = reinterpret_cast<uint4 *>(smem);  // first inner row, value, partner's row, target row or slot
    uint32_t *extra = reinterpret_cast<uint32_t *>(smem + L.extra);
    float *hot = reinterpret_cast<float *>(smem + L.hot);

    for (int i = threadIdx.x; i < p.kw * R; i += kTiledThreads) hot[i] = 0.f;

    const int sub = threadIdx.x / G;
    const int c = threadIdx.x % G;
    const int s0 = sub * P;
    float *const out0 =
        static_cast<float *>(p.out) + (p.ncopies > 1 ? (size_t)(blockIdx.x % p.ncopies) * p.copy_stride : 0);
    float *const outp = out0 + c * VEC;
    float *const hotc = hot + c * VEC;
    const char *const inp = static_cast<const char *>(p.gat[0].ptr) + (size_t)c * VEC * sizeof(T);
    const char *const parp = static_cast<const char *>(p.par.ptr) + (size_t)c * VEC * sizeof(T);

    const int64_t ntiles = (p.nnz + kTile - 1) / kTile;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t base = tile * kTile;
        const int nvalid = p.nnz - base < kTile ? (int)(p.nnz - base) : kTile;
        const uint32_t *endw = p.ends + tile * (kTile / 32) + (s0 >> 5);
        uint32_t ew = __ldg(endw);
        prefetch_tile(p, tile + gridDim.x, ntiles, p.vals, (int)sizeof(float));
        stage_tile<NI, P>(
            p, base, nvalid, ni,
            [&](uint32_t r, bool valid, int q, uint32_t o, uint32_t k, uint32_t row) {
                const float v = valid ? ld_stream_f32(p.vals + base + q) : 0.f;
                rec[r] = make_uint4(o, __float_as_uint(v), k, row);
            },
            extra);
        __syncthreads();

        f2 acc[H];
#pragma unroll
        for (int h = 0; h < H; ++h) acc[h] = 0ull;
        bool open = false;
        uint32_t open_row = 0;
        if (s0 < nvalid) {
            const uint4 *rp = rec + s0 + sub;  // one unused entry after every P ranks
            const uint32_t *xp = extra + s0 + sub;
#pragma unroll 1
            for (int b = 0; b < P; b += PB) {
                uint32_t e = ew >> (s0 & 31);
                if (b + PB < P) {
                    ew = __ldg(endw + (b >> 5) + 1);
                } else {
                    // a run that does not end at the last rank leaves a part open
                    open = !((e >> (PB - 1)) & 1u) && s0 + P <= nvalid;
                }
#pragma unroll 1
                for (int u = 0; u < PB; u += CH, e >>= CH, rp += CH, xp += CH) {
                    uint4 rc[CH];
                    f2 x[CH][H], k[CH][H];
#pragma unroll
                    for (int j = 0; j < CH; ++j) rc[j] = rp[j];
#pragma unroll
                    for (int j = 0; j < CH; ++j) {
                        if (NG != 0 || ni > 0) Chunk<T>::load(inp + (size_t)rc[j].x * (R * sizeof(T)), x[j]);
                        Chunk<T>::load(parp + (size_t)rc[j].z * (R * sizeof(T)), k[j]);
                    }
#pragma unroll
                    for (int q = 1; q < NI; ++q) {
                        if (q < ni) {
                            f2 g[CH][H];
                            const char *gp = static_cast<const char *>(p.gat[q].ptr) + (size_t)c * VEC * sizeof(T);
#pragma unroll
                            for (int j = 0; j < CH; ++j)
                                Chunk<T>::load(gp + (size_t)xp[(q - 1) * staged<P>() + j] * (R * sizeof(T)), g[j]);
#pragma unroll
                            for (int j = 0; j < CH; ++j)
#pragma unroll
                                for (int h = 0; h < H; ++h) x[j][h] = mul2(x[j][h], g[j][h]);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < CH; ++j) {
                        const float v = __uint_as_float(rc[j].y);
                        const f2 vv = pack2(v, v);
#pragma unroll
                        for (int h = 0; h < H; ++h) {
                            x[j][h] = (NG != 0 || ni > 0) ? mul2(vv, x[j][h]) : vv;
                            acc[h] = fma2(x[j][h], k[j][h], acc[h]);
                        }
                        if (e & (1u << j)) {
                            const uint32_t row = rc[j].w;
                            if (row & kSlotBit) {
                                ulonglong2 *a = reinterpret_cast<ulonglong2 *>(hotc + (row & ~kSlotBit) * R);
                                ulonglong2 cur = *a;
                                cur.x = add2(cur.x, acc[0]);
                                cur.y = add2(cur.y, acc[1]);
                                *a = cur;
                            } else {
                                float sv[VEC];
#pragma unroll
                                for (int h = 0; h < H; ++h) unpack2(acc[h], sv[2 * h], sv[2 * h + 1]);
                                red_add_v4(outp + (size_t)row * R, sv[0], sv[1], sv[2], sv[3]);
                            }
#pragma unroll
                            for (int h = 0; h < H; ++h) acc[h] = 0ull;
                        }
                    }
                }
            }
            if (open) open_row = rec[s0 + sub + P - 1].w;
        }
        __syncthreads();
        if (open) {
            float sv[VEC];
#pragma unroll
            for (int h = 0; h < H; ++h) unpack2(acc[h], sv[2 * h], sv[2 * h + 1]);
            if (open_row & kSlotBit) {
                float *a = hotc + (open_row & ~kSlotBit) * R;
#pragma unroll
                for (int i = 0; i < VEC; ++i) atomicAdd(a + i, sv[i]);
            } else {
                red_add_v4(outp + (size_t)open_row * R, sv[0], sv[1], sv[2], sv[3]);
            }
        }
    }

    // --- add the cluster's copies to the output once, each CTA a part of them
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    cl.sync();
    constexpr int Q = R / 4;
    for (int i = cl.block_rank() * kTiledThreads + threadIdx.x; i < p.kw * Q; i += kTiledCluster * kTiledThreads) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int b = 0; b < kTiledCluster; ++b) {
            const float4 x = reinterpret_cast<const float4 *>(cl.map_shared_rank(hot, b))[i];
            v.x += x.x;
            v.y += x.y;
            v.z += x.z;
            v.w += x.w;
        }
        if (v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f)
            red_add_v4(out0 + (size_t)__ldg(p.hot_rows + i / Q) * R + i % Q * 4, v.x, v.y, v.z, v.w);
    }
    cl.sync();  // the copies stay until every CTA has read them
}

// -------------------------------------------------------------------------
// float64 values, factors and sums
// -------------------------------------------------------------------------
// Bound by the float64 pipe (2 lanes per SM and cycle), so the operations per
// nonzero are what counts: along a fiber one multiply-add per element and
// inner mode, at its end one more with the partner's row, where a product per
// gathered row and a sum are N operations per nonzero. A subgroup is a whole
// warp from R = 32 on, so a fiber's end costs only the warp that has one. 20M
// nonzeros of the 3-mode Zipf shape (2^20, 2^19, 2^11), R = 32, all modes:
// 10.9 ms with the kernel of mttkrp_f64.cu, 6.8 here. For 3 and 4 modes
// (order_pays_f64): without an inner mode a fiber's sum takes as many
// operations as the terms, and from 5 modes on fibers are one or two nonzeros
// long (2 modes 10M nonzeros, R = 32: 2.7 ms there, 8.7 here; 5 modes 2M, R =
// 64: 6.3 and 10.6; 7 modes 10M, R = 32: 0.90 of its speed).
__device__ __forceinline__ void red_add_double(double *addr, double v) {
    asm volatile("red.global.add.f64 [%0], %1;" ::"l"(addr), "d"(v));
}

template <int VEC>
__device__ __forceinline__ void load_doubles(const double *p, double (&f)[VEC]) {
    if constexpr (VEC == 2) {
        const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
        f[0] = v.x;
        f[1] = v.y;
    } else {
        f[0] = __ldg(p);
    }
}

struct __align__(16) Rec64 {
    double val;
    uint32_t in, par;
};

__device__ __forceinline__ bool is_finite(double x) {
    return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}

// acc plus a fiber's terms one by one, `n` ranks from `rp` on, times the
// partner's element `k`: where the fiber's sum or `k` is not finite, their
// product is not the sum of the terms (0 times infinity among them).
template <int NI>
__device__ __noinline__ double add_terms(double acc, const Rec64 *rp, const uint32_t *xp, int stride, int n,
                                         const TParams &p, int R, int e, double k) {
    for (int r = 0; r < n; ++r) {
        double x = rp[r].val * __ldg(static_cast<const double *>(p.gat[0].ptr) + (size_t)rp[r].in * R + e);
        for (int q = 1; q < NI; ++q)
            x *= __ldg(static_cast<const double *>(p.gat[q].ptr) + (size_t)xp[(q - 1) * stride + r] * R + e);
        acc = fma(x, k, acc);
    }
    return acc;
}

template <int R, int NG>
__global__ void __launch_bounds__(kTiledThreads, R > 32 ? 2 : 3) k_mttkrp64_tiled(const TParams p) {
    constexpr int G = R < 32 ? R : 32;
    constexpr int VEC = R / G;
    constexpr int SUBS = kTiledThreads / G;
    constexpr int P = kTile / SUBS;
    constexpr int CH = 4;
    constexpr int NI = inner_slots<NG>();
    static_assert(P % 32 == 0 && VEC <= 2, "whole words of the bit masks");
    static_assert(NG == 2 || NG == 3, "one or two inner modes");

    extern __shared__ __align__(16) unsigned char smem[];
    // one word per rank more than the float32 kernel: the target row or slot
    const TiledSmem L = tiled_smem(sizeof(Rec64), staged<P>(), NI, p.kw, R * sizeof(double));
    Rec64 *rec = reinterpret_cast<Rec64 *>(smem);
    uint32_t *srow = reinterpret_cast<uint32_t *>(smem + L.extra);
    uint32_t *extra = srow + staged<P>();
    double *hot = reinterpret_cast<double *>(smem + L.hot);

    for (int i = threadIdx.x; i < p.kw * R; i += kTiledThreads) hot[i] = 0.0;

    const int sub = threadIdx.x / G;
    const int c = threadIdx.x % G;
    const int s0 = sub * P;
    double *const outp = static_cast<double *>(p.out) + c * VEC;
    double *const hotc = hot + c * VEC;
    const double *const inp = static_cast<const double *>(p.gat[0].ptr) + c * VEC;
    const double *const parp = static_cast<const double *>(p.par.ptr) + c * VEC;

    const int64_t ntiles = (p.nnz + kTile - 1) / kTile;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t base = tile * kTile;
        const int nvalid = p.nnz - base < kTile ? (int)(p.nnz - base) : kTile;
        const uint32_t *endw = p.ends + tile * (kTile / 32) + (s0 >> 5);
        const uint32_t *fendw = p.fends + tile * (kTile / 32) + (s0 >> 5);
        uint32_t ew = __ldg(endw), fw = __ldg(fendw);
        prefetch_tile(p, tile + gridDim.x, ntiles, p.vals64, (int)sizeof(double));
        stage_tile<NI, P>(
            p, base, nvalid, NI,
            [&](uint32_t r, bool valid, int q, uint32_t o, uint32_t k, uint32_t row) {
                Rec64 rc;
                rc.val = valid ? __ldcs(p.vals64 + base + q) : 0.0;
                rc.in = o;
                rc.par = k;
                rec[r] = rc;
                srow[r] = row;
            },
            extra);
        __syncthreads();

        double acc[VEC], fs[VEC];
#pragma unroll
        for (int i = 0; i < VEC; ++i) acc[i] = fs[i] = 0.0;
        bool open = false;
        uint32_t open_row = 0;
        if (s0 < nvalid) {
            const Rec64 *rp = rec + s0 + sub;
            const uint32_t *xp = extra + s0 + sub, *rowp = srow + s0 + sub;
            int first = s0 + sub;  // the open fiber's first rank
#pragma unroll 1
            for (int b = 0; b < P; b += 32) {
                uint32_t e = ew, fe = fw;
                if (b + 32 < P) {
                    ew = __ldg(endw + (b >> 5) + 1);
                    fw = __ldg(fendw + (b >> 5) + 1);
                } else {
                    open = !(e >> 31) && s0 + P <= nvalid;
                    fe |= 0x80000000u;  // the last rank ends its part of the fiber
                }
#pragma unroll 1
                for (int u = 0; u < 32; u += CH, e >>= CH, fe >>= CH, rp += CH, xp += CH, rowp += CH) {
                    Rec64 rc[CH];
                    double x[CH][VEC], k[CH][VEC];
#pragma unroll
                    for (int j = 0; j < CH; ++j) rc[j] = rp[j];
#pragma unroll
                    for (int j = 0; j < CH; ++j)
                        load_doubles<VEC>(inp + (size_t)rc[j].in * R, x[j]);
#pragma unroll
                    for (int j = 0; j < CH; ++j)
                        if (fe & (1u << j)) load_doubles<VEC>(parp + (size_t)rc[j].par * R, k[j]);
#pragma unroll
                    for (int q = 1; q < NI; ++q) {
                        const double *gp = static_cast<const double *>(p.gat[q].ptr) + c * VEC;
                        double g[CH][VEC];
#pragma unroll
                        for (int j = 0; j < CH; ++j)
                            load_doubles<VEC>(gp + (size_t)xp[(q - 1) * staged<P>() + j] * R, g[j]);
#pragma unroll
                        for (int j = 0; j < CH; ++j)
#pragma unroll
                            for (int i = 0; i < VEC; ++i) x[j][i] *= g[j][i];
                    }
#pragma unroll
                    for (int j = 0; j < CH; ++j) {
#pragma unroll
                        for (int i = 0; i < VEC; ++i)
                            fs[i] = fma(rc[j].val, x[j][i], fs[i]);
                        if (fe & (1u << j)) {
#pragma unroll
                            for (int i = 0; i < VEC; ++i) {
                                if (is_finite(fs[i]) && is_finite(k[j][i]))
                                    acc[i] = fma(fs[i], k[j][i], acc[i]);
                                else
                                    acc[i] = add_terms<NI>(acc[i], rec + first, extra + first, staged<P>(),
                                                           (int)(rp + j - rec) - first + 1, p, R, c * VEC + i,
                                                           k[j][i]);
                                fs[i] = 0.0;
                            }
                            first = (int)(rp + j - rec) + 1;
                            if (e & (1u << j)) {  // a run's end is a fiber's end
                                const uint32_t row = rowp[j];
#pragma unroll
                                for (int i = 0; i < VEC; ++i) {
                                    if (row & kSlotBit)
                                        hotc[(row & ~kSlotBit) * R + i] += acc[i];
                                    else
                                        red_add_double(outp + (size_t)row * R + i, acc[i]);
                                    acc[i] = 0.0;
                                }
                            }
                        }
                    }
                }
            }
            if (open) open_row = srow[s0 + sub + P - 1];
        }
        __syncthreads();
        if (open) {
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                if (open_row & kSlotBit)
                    atomicAdd(hotc + (open_row & ~kSlotBit) * R + i, acc[i]);
                else
                    red_add_double(outp + (size_t)open_row * R + i, acc[i]);
            }
        }
    }

    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    cl.sync();
    for (int i = cl.block_rank() * kTiledThreads + threadIdx.x; i < p.kw * R; i += kTiledCluster * kTiledThreads) {
        double v = 0.0;
#pragma unroll
        for (int b = 0; b < kTiledCluster; ++b) v += cl.map_shared_rank(hot, b)[i];
        if (v != 0.0) red_add_double(static_cast<double *>(p.out) + (size_t)__ldg(p.hot_rows + i / R) * R + i % R, v);
    }
    cl.sync();
}

// -------------------------------------------------------------------------
// launch helpers
// -------------------------------------------------------------------------
TParams tiled_params(const StoreView &sv, const TileOrder &to, const void *const *fac, int mode, const HotRows &hot,
                     size_t row_bytes) {
    TParams p;
    memset(&p, 0, sizeof(p));
    p.keys = sv.keys;
    p.vals = sv.vals;
    p.vals64 = sv.vals64;
    p.vals_aligned = (reinterpret_cast<uintptr_t>(sv.vals) & 15) == 0;  // a caller's gradient may not be
    p.nnz = sv.end;
    p.tile_block = sv.tile_block;
    p.bstart = sv.bstart;
    p.bbase = sv.bbase;
    p.single_block = sv.single_block;
    p.rank = to.rank[mode];
    p.ends = to.ends[mode];
    p.fends = to.fends[mode];
    p.t_shift = sv.shift[mode];
    p.t_mask = sv.mask[mode];
    p.t_mode = mode;
    const int par = order_partner(sv.dims, sv.N, mode);
    for (int k = 0; k < sv.N; ++k) {
        if (k == mode) continue;
        Gather &g = k == par ? p.par : p.gat[p.n_inner++];
        g.ptr = fac[k];
        g.shift = sv.shift[k];
        g.mask = sv.mask[k];
        g.mode = k;
    }
    p.hot_rows = hot.rows;
    p.kw = std::min(std::min(hot.count, kOrderCold), (int)(kTiledHotBytes / row_bytes));
    return p;
}

// Clusters of a kernel that are resident at once with `shm` bytes of shared
// memory, at least 1 (a cluster stays inside a GPC, so that is not the SMs' CTAs
// over the cluster's size).
template <typename K>
int resident_clusters(K kern, const cudaLaunchConfig_t &cfg, std::atomic<uint64_t> &last) {
    const int n = remembered(last, cfg.dynamicSmemBytes,
                             [&](int *clusters) { return cudaOccupancyMaxActiveClusters(clusters, kern, &cfg); });
    return n > 0 ? n : 1;
}

template <typename K>
cudaError_t launch_tiled(K kern, const TParams &p, size_t shm, std::atomic<uint64_t> &last, cudaStream_t s) {
    const cudaError_t e = allow_smem((const void *)kern, shm);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (p.nnz + kTile - 1) / kTile;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kTiledCluster);
    cfg.blockDim = dim3(kTiledThreads);
    cfg.dynamicSmemBytes = shm;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kTiledCluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const int64_t need = (tiles + kTiledCluster - 1) / kTiledCluster;
    cfg.gridDim = dim3((unsigned)(std::min<int64_t>(resident_clusters(kern, cfg, last), need) * kTiledCluster));
    return cudaLaunchKernelEx(&cfg, kern, p);
}

template <typename T, int R, int NG>
cudaError_t run_tiled(const TParams &p, cudaStream_t s) {
    constexpr int P = kTile / (kTiledThreads / (R / lane_vec<T, R>()));
    static std::atomic<uint64_t> last{0};
    return launch_tiled(
        k_mttkrp_tiled<T, R, NG>, p,
        tiled_smem(sizeof(uint4), staged<P>(), p.n_inner > 1 ? p.n_inner - 1 : 0, p.kw, R * sizeof(float)).total, last,
        s);
}

template <typename T, int R>
cudaError_t tiled_by_ng(const TParams &p, cudaStream_t s) {
    switch (p.n_inner) {
        case 1: return run_tiled<T, R, 2>(p, s);
        case 2: return run_tiled<T, R, 3>(p, s);
        case 3: return run_tiled<T, R, 4>(p, s);
        default: return run_tiled<T, R, 0>(p, s);
    }
}

template <typename T>
cudaError_t tiled_as(const StoreView &sv, const TileOrder &to, const FactorSet &fs, int R, int mode, const HotRows &hot,
                     float *out, const OutCopies &oc, cudaStream_t s) {
    if (sv.end <= 0) return cudaSuccess;
    TParams p = tiled_params(sv, to, fs.ptr, mode, hot, R * sizeof(float));
    p.out = out;
    p.ncopies = oc.n > 1 ? oc.n : 1;
    p.copy_stride = oc.stride;
    switch (R) {
        case 8: return run_tiled<T, 8, 0>(p, s);
        case 16: return tiled_by_ng<T, 16>(p, s);
        case 32: return tiled_by_ng<T, 32>(p, s);
        case 64: return tiled_by_ng<T, 64>(p, s);
        case 128: return run_tiled<T, 128, 0>(p, s);
    }
    return cudaErrorInvalidValue;
}

template <int R, int NG>
cudaError_t run_tiled64(const TParams &p, cudaStream_t s) {
    constexpr int P = kTile / (kTiledThreads / (R < 32 ? R : 32));
    static std::atomic<uint64_t> last{0};
    return launch_tiled(
        k_mttkrp64_tiled<R, NG>, p,
        tiled_smem(sizeof(Rec64), staged<P>(), inner_slots<NG>(), p.kw, R * sizeof(double)).total, last, s);
}

template <int R>
cudaError_t tiled64_by_ng(const TParams &p, cudaStream_t s) {
    switch (p.n_inner) {
        case 1: return run_tiled64<R, 2>(p, s);
        case 2: return run_tiled64<R, 3>(p, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace
}  // namespace blco
