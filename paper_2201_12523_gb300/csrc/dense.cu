// Dense helpers around the sparse kernels: output zeroing, float32 ->
// 16-bit factor conversion, and the FP64 pieces of CP-ALS (Algorithm 1):
// Grams, the Hadamard product of Grams, its inverse (or eigen
// pseudo-inverse) solve, column normalization and the fit.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>

#include "internal.h"

namespace blco {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

unsigned grid_cap(int64_t n, int threads) {
    int64_t g = (n + threads - 1) / threads;
    const int64_t cap = (int64_t)sm_count() * 8;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (unsigned)g;
}

__global__ void k_zero4(float4 *p, int64_t n4) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}
__global__ void k_zero1(float *p, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = 0.f;
}

__global__ void k_to_bf16(const float *__restrict__ s, __nv_bfloat16 *__restrict__ d, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        d[i] = __float2bfloat16_rn(s[i]);
}
__global__ void k_to_f16(const float *__restrict__ s, __half *__restrict__ d, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        d[i] = __float2half_rn(s[i]);
}

template <typename T>
__device__ __forceinline__ float to_f(T v);
template <>
__device__ __forceinline__ float to_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <>
__device__ __forceinline__ float to_f<__half>(__half v) { return __half2float(v); }

// G = A^T A. Each thread owns a 4 x 4 block of G in the upper triangle
// (diagonal blocks included) and accumulates its 16 dot products over its
// CTA's rows with Ogita, Rump and Oishi's Dot2 (SIAM J. Sci. Comput. 26(6),
// 2005): TwoProduct by FMA gives each float32 product exactly as p + e, and
// TwoSum carries the rounding error of every addition, so each partial is a
// float32 pair as accurate as a sum in twice the float32 precision. The pair
// is added in float64 (hi + lo), the CTA's thread groups are summed in
// shared memory in float64, and CTAs meet in float64 atomics (both halves of
// an off-diagonal block). This keeps the FP64 pipe, which is a small fraction
// of the FP32 rate on this GPU, off the O(I R^2) part of the work.
//
// Bound by the ten float32 operations per product. CTAs are as wide as whole
// thread groups need (at most kGramThreads): with 256 threads, R = 64 left one
// group of 136 threads and the other 120 idle, and 2^20 rows took 1.30 ms; two
// groups in 288 threads take 1.02 with two CTAs per SM (1.13 with three, whose
// 72 registers spill; at R = 16 and 50 three are 7-10 % faster, so two only
// from kGramWideRank on). Packed f32x2 arithmetic: 1.18, that pipe's rate.
constexpr int kGramRows = 32;  // rows staged in shared memory per step
constexpr int kGramThreads = 288;
constexpr int kGramWideRank = 60;

struct GramShape {
    int R4;      // R rounded up to 4 (padding columns are zero)
    int B;       // 4 x 4 blocks per side
    int nblk;    // blocks in the upper triangle
    int ny;      // parts of the blocks, one per blockIdx.y
    int per_y;   // blocks of a part
    int groups;  // thread groups per CTA that split the rows
};

__host__ __device__ inline GramShape gram_shape(int R) {
    GramShape g;
    g.R4 = (R + 3) & ~3;
    g.B = g.R4 / 4;
    g.nblk = g.B * (g.B + 1) / 2;
    g.ny = (g.nblk + kGramThreads - 1) / kGramThreads;
    g.per_y = (g.nblk + g.ny - 1) / g.ny;
    g.groups = kGramThreads / g.per_y;
    return g;
}

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float z = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}

// One more term x * y of a Dot2 sum (hi, lo).
__device__ __forceinline__ void dot2_add(float x, float y, float &hi, float &lo) {
    const float p = __fmul_rn(x, y);
    const float e = __fmaf_rn(x, y, -p);  // x*y == p + e exactly
    float sum, err;
    two_sum(hi, p, sum, err);
    hi = sum;
    lo = __fadd_rn(lo, __fadd_rn(err, e));
}

// A sum of products in three floats, four terms at a time. The products and
// the sum of the four are split free of error (TwoProduct, TwoSum), the small
// parts of the four added in float32, and both added to the sum with their
// errors kept (as Dot3 of Ogita, Rump and Oishi, 2005): 13 float32 operations a
// term, where float64 takes a conversion and an FMA of a pipe with 2 lanes per
// SM. For columns of 1 to 2^20 normal numbers the result (added over threads
// and CTAs in float64) is off by at most 8e-16, the float64 sum it stands for
// by 4e-15; Dot2, whose error grows with the terms of a thread, by 5e-13 at 500.
// All that while the products are in float32's range: one is off by up to
// 2^-149 where it or its error underflows, and not finite where it overflows. A
// CTA (a warp in k_norm2) adds its sum to the total and takes it again in float64
// where it is not finite, or where the total so far is not yet large against
// such errors of all n terms, n 2^-95, with entries other than 0 among its own:
// when everything is small, not where only a few CTAs' rows are (sweeps of small
// tensors with long modes, whose rows are mostly empty, lost 5 % to that).
struct WideSum {
    float hi = 0.f, mid = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(const float (&x)[4], const float (&y)[4]) {
        float p[4], e[4], s0, s1, t, r0, r1, r2, a, b, c;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            p[i] = __fmul_rn(x[i], y[i]);
            e[i] = __fmaf_rn(x[i], y[i], -p[i]);
        }
        two_sum(p[0], p[1], s0, r0);
        two_sum(p[2], p[3], s1, r1);
        two_sum(s0, s1, t, r2);
        const float u = __fadd_rn(__fadd_rn(__fadd_rn(e[0], e[1]), __fadd_rn(e[2], e[3])),
                                  __fadd_rn(__fadd_rn(r0, r1), r2));
        two_sum(hi, t, hi, a);
        two_sum(mid, u, mid, b);
        two_sum(mid, a, mid, c);
        lo = __fadd_rn(lo, __fadd_rn(b, c));
    }
    __device__ __forceinline__ double value() const { return (double)hi + ((double)mid + (double)lo); }
};

// Adds a sum to *total. False where it has to be taken again (see above).
__device__ __forceinline__ bool add_sum(double *total, double sum, bool seen, double enough) {
    if (!(fabs(sum) < INFINITY)) return false;
    if (!seen) return true;  // 0
    return fabs(atomicAdd(total, sum) + sum) >= enough;
}
// Puts the float64 sum in its place.
__device__ __forceinline__ void replace_sum(double *total, double sum, double by) {
    atomicAdd(total, fabs(sum) < INFINITY ? by - sum : by);
}

__device__ __forceinline__ uint32_t bits_of(const float (&x)[4]) {
    return (__float_as_uint(x[0]) | __float_as_uint(x[1]) | __float_as_uint(x[2]) | __float_as_uint(x[3])) & 0x7FFFFFFFu;
}

// Column scales from the columns' sums of squares: lambda = sqrt, 1 / lambda
// (1 for a zero column).
__device__ __forceinline__ float inv_norm(double colsq, double *lambda) {
    const double l = sqrt(colsq);
    *lambda = l;
    return l > 0.0 ? (float)(1.0 / l) : 1.f;
}

// With SCALE (float factors, one part of blocks), A's columns are first divided
// by their norms, in place, and the Gram is that of the scaled A; CTA 0 writes
// lambda. Scaling here instead of in a pass of its own saves that pass's read
// and write (0.15 ms at 2^20 x 64).
template <typename T, bool SCALE, int CTAS>
__global__ void __launch_bounds__(kGramThreads, CTAS) k_gram(const T *A, T *A_out, int64_t I, int R, int64_t rows_per_cta,
                                                       const double *__restrict__ colsq, double *__restrict__ lambda,
                                                       double *__restrict__ G) {
    extern __shared__ __align__(16) unsigned char smem[];
    const GramShape sh = gram_shape(R);
    float *tile = reinterpret_cast<float *>(smem);                       // kGramRows x R4
    double *red = reinterpret_cast<double *>(tile + kGramRows * sh.R4);  // groups x per_y x 16
    __shared__ float inv[SCALE ? 64 : 1];
    const int tid = threadIdx.x;
    if (SCALE) {
        if (tid < R) {
            double l;
            inv[tid] = inv_norm(colsq[tid], &l);
            if (blockIdx.x == 0) lambda[tid] = l;
        }
    }
    const int grp = tid / sh.per_y;
    const int lbl = tid % sh.per_y;  // block inside the part
    const int blk = blockIdx.y * sh.per_y + lbl;
    const bool active = grp < sh.groups && blk < sh.nblk && (!SCALE || G);
    int br = 0, rem = active ? blk : 0;  // upper-triangle block -> (br, bc)
    while (rem >= sh.B - br) {
        rem -= sh.B - br;
        ++br;
    }
    const int bc = br + rem;
    float hi[16], lo[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) hi[k] = lo[k] = 0.f;
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_cta;
    const int64_t r1 = r0 + rows_per_cta < I ? r0 + rows_per_cta : I;
    // rows of whole 16-byte words (8 bytes of 16-bit factors) move four at a time
    const bool vec = sizeof(T) == 4 && R == sh.R4 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
    for (int64_t b0 = r0; b0 < r1; b0 += kGramRows) {
        const int nr = (int)((r1 - b0) < kGramRows ? (r1 - b0) : kGramRows);
        __syncthreads();
        if (vec) {
            const float4 *src = reinterpret_cast<const float4 *>(A + b0 * R);
            for (int i = tid; i < kGramRows * sh.B; i += blockDim.x) {
                float4 v = i < nr * sh.B ? src[i] : make_float4(0.f, 0.f, 0.f, 0.f);
                if (SCALE && i < nr * sh.B) {
                    const int c = i % sh.B * 4;
                    v.x *= inv[c];
                    v.y *= inv[c + 1];
                    v.z *= inv[c + 2];
                    v.w *= inv[c + 3];
                    reinterpret_cast<float4 *>(A_out + b0 * R)[i] = v;
                }
                reinterpret_cast<float4 *>(tile)[i] = v;
            }
        } else {
            for (int i = tid; i < kGramRows * sh.R4; i += blockDim.x) {
                const int row = i / sh.R4, col = i % sh.R4;
                float v = 0.f;
                if (row < nr && col < R) {
                    v = to_f<T>(A[(b0 + row) * R + col]);
                    if constexpr (SCALE) {
                        v *= inv[col];
                        A_out[(b0 + row) * R + col] = v;
                    }
                }
                tile[i] = v;
            }
        }
        __syncthreads();
        if (!active) continue;
        for (int i = grp; i < nr; i += sh.groups) {
            const float4 x = *reinterpret_cast<const float4 *>(tile + i * sh.R4 + br * 4);
            const float4 y = *reinterpret_cast<const float4 *>(tile + i * sh.R4 + bc * 4);
            const float xa[4] = {x.x, x.y, x.z, x.w}, ya[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) dot2_add(xa[u], ya[v], hi[u * 4 + v], lo[u * 4 + v]);
        }
    }
    if (SCALE && !G) return;
    // sum the thread groups of this CTA in float64, then one atomic per entry
    if (active)
#pragma unroll
        for (int k = 0; k < 16; ++k) red[(grp * sh.per_y + lbl) * 16 + k] = (double)hi[k] + (double)lo[k];
    __syncthreads();
    const int nact = min(sh.per_y, sh.nblk - (int)blockIdx.y * sh.per_y);
    for (int i = tid; i < nact * 16; i += blockDim.x) {
        const int lb = i / 16, k = i % 16;
        double v = 0.0;
        for (int g2 = 0; g2 < sh.groups; ++g2) v += red[(g2 * sh.per_y + lb) * 16 + k];
        int rr = 0, rm = (int)blockIdx.y * sh.per_y + lb;
        while (rm >= sh.B - rr) {
            rm -= sh.B - rr;
            ++rr;
        }
        const int r = rr * 4 + k / 4, c = (rr + rm) * 4 + k % 4;
        if (r >= R || c >= R) continue;
        atomicAdd(&G[(size_t)r * R + c], v);
        if (rr != rr + rm) atomicAdd(&G[(size_t)c * R + r], v);
    }
}

__global__ void k_zero_d(double *p, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = 0.0;
}

struct GramPtrs {
    const double *g[MAXN];
};

// -------------------------------------------------------------------------
// one CTA: V = Hadamard of Grams (k != mode); W = V^{-1}, or the eigen
// pseudo-inverse (cyclic Jacobi) when V is not positive definite. Output W as
// float32 (the apply step) and info; zeroes the column sums of squares that
// the apply step adds to.
//
// The inverse is Gauss-Jordan elimination on the symmetric matrix (the sweep
// operator, J. H. Goodnight, The American Statistician 33(3), 1979): its pivots
// are the squares of Cholesky's, so positive definiteness is decided as a
// Cholesky factorization decides it. The lower triangle stays in registers
// (R (R + 1) / 2 entries over 256 threads) and a step passes only its pivot
// column through shared memory. Bound by the one SM's FP64 pipe at R = 64
// (R^2 / 2 multiply-adds per step) and by the step's chain (reciprocal, two
// barriers) at R = 32: Cholesky with one thread per column of the inverse took
// 376 us at R = 64 and 129 us at R = 32, this 122 and 41 (with a float64 division
// and a third barrier per step 154 and 62).
// -------------------------------------------------------------------------
// 1 / x to float64 rounding: Newton's iteration from the float reciprocal, whose
// error (about 2^-23) squares twice; a float64 division is a longer chain.
// Outside the floats' range, and where x is not positive, it is the division.
__device__ __forceinline__ double reciprocal(double x) {
    if (!(x > 1e-30 && x < 1e30)) return 1.0 / x;
    double r = (double)(1.f / (float)x);
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

constexpr int kSolveThreads = 256;
constexpr int kSolveMaxRank = 64;
constexpr int kSolveSlots = (kSolveMaxRank * (kSolveMaxRank + 1) / 2 + kSolveThreads - 1) / kSolveThreads;

__global__ void __launch_bounds__(kSolveThreads) k_solve_small(const GramPtrs gp, int N, int mode, int R,
                                                               float *__restrict__ Wf, double *__restrict__ colsq,
                                                               int32_t *__restrict__ info) {
    extern __shared__ __align__(16) unsigned char smem[];
    double *V = reinterpret_cast<double *>(smem);  // R x R: V, then the Jacobi vectors
    double *L = V + R * R;                           // R x R work
    const int tid = threadIdx.x;
    if (tid < R) colsq[tid] = 0.0;
    for (int p = tid; p < R * R; p += kSolveThreads) {
        double v = 1.0;
        for (int k = 0; k < N; ++k)
            if (k != mode) v *= gp.g[k][p];
        V[p] = v;
    }
    __shared__ double pd_tol, rcp[2];
    __shared__ double col[2][kSolveMaxRank], colr[kSolveMaxRank];
    __shared__ int ok;
    __syncthreads();
    if (tid < 32) {
        // smallest pivot accepted as positive: R * eps * max_i V_ii; at or
        // below it V is treated as not positive definite (numerically
        // singular or indefinite) and the pseudo-inverse is used
        double m = 0.0;
        for (int i = tid; i < R; i += 32) m = fmax(m, V[i * R + i]);
        for (int o = 16; o >= 1; o >>= 1) m = fmax(m, __shfl_xor_sync(kFull, m, o));
        if (tid == 0) {
            ok = 1;
            pd_tol = (double)R * 2.220446049250313e-16 * m;
        }
    }
    // entry (row, column) of the lower triangle in slot q of this thread
    const int ntri = R * (R + 1) / 2;
    const int slots = (ntri + kSolveThreads - 1) / kSolveThreads;
    double x[kSolveSlots];
    int ri[kSolveSlots], ci[kSolveSlots];
#pragma unroll
    for (int q = 0; q < kSolveSlots; ++q) {
        const int t = tid + q * kSolveThreads;
        int i = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);  // row, up to rounding
        if (i * (i + 1) / 2 > t) --i;
        if ((i + 1) * (i + 2) / 2 <= t) ++i;
        ri[q] = t < ntri ? i : -1;
        ci[q] = t < ntri ? t - i * (i + 1) / 2 : -1;
        x[q] = t < ntri ? V[ri[q] * R + ci[q]] : 0.0;
    }
    // passes on the part of row and column j that slot q holds
    const auto publish = [&](int q, int j) {
        if (ci[q] == j) {
            col[j & 1][ri[q]] = x[q];
            if (ri[q] == j) rcp[j & 1] = reciprocal(x[q]);
        } else if (ri[q] == j) {
            col[j & 1][ci[q]] = x[q];
        }
    };
#pragma unroll
    for (int q = 0; q < kSolveSlots; ++q)
        if (q < slots) publish(q, 0);
    __syncthreads();
    for (int j = 0; j < R; ++j) {
        const double *c = col[j & 1];
        const double d = rcp[j & 1];
        if (tid < R) {
            colr[tid] = c[tid] * d;
            if (tid == j && !(c[j] > pd_tol)) ok = 0;
        }
        __syncthreads();
        if (!ok) break;
#pragma unroll
        for (int q = 0; q < kSolveSlots; ++q) {
            if (q >= slots || ri[q] < 0) continue;
            if (ri[q] == j)
                x[q] = ci[q] == j ? -d : colr[ci[q]];
            else if (ci[q] == j)
                x[q] = colr[ri[q]];
            else
                x[q] = fma(-colr[ri[q]], c[ci[q]], x[q]);
            publish(q, j + 1);
        }
        __syncthreads();
    }
    if (ok) {
#pragma unroll
        for (int q = 0; q < kSolveSlots; ++q) {
            if (ri[q] < 0) continue;
            Wf[ri[q] * R + ci[q]] = Wf[ci[q] * R + ri[q]] = (float)-x[q];
        }
        if (tid == 0) *info = 0;
        return;
    }
    __syncthreads();
    // ---- eigen pseudo-inverse: cyclic Jacobi rotations on L := V, Q := I
    double *Q = V;
    for (int p = tid; p < R * R; p += blockDim.x) {
        L[p] = V[p];
        Q[p] = (p / R == p % R) ? 1.0 : 0.0;
    }
    __syncthreads();
    __shared__ double cs[128][2];
    __shared__ int pairs_p[64], pairs_q[64];
    __shared__ double off;
    const int Rp = (R + 1) & ~1;  // even count for round-robin pairing (a dummy index when R is odd)
    for (int sweep = 0; sweep < 30; ++sweep) {
        if (tid == 0) off = 0.0;
        __syncthreads();
        for (int p = tid; p < R * R; p += blockDim.x)
            if (p / R != p % R) atomicAdd(&off, L[p] * L[p]);
        __syncthreads();
        double diag = 0.0;
        for (int i = 0; i < R; ++i) diag += L[i * R + i] * L[i * R + i];
        if (off <= 1e-30 * diag || off == 0.0) break;
        for (int round = 0; round < Rp - 1; ++round) {
            // round-robin schedule: position 0 fixed, the rest rotate
            if (tid < Rp / 2) {
                const int a = tid == 0 ? 0 : 1 + (tid - 1 + round) % (Rp - 1);
                const int b = 1 + (Rp - 2 - tid + round) % (Rp - 1);
                pairs_p[tid] = a < b ? a : b;
                pairs_q[tid] = a < b ? b : a;
            }
            __syncthreads();
            if (tid < Rp / 2) {
                const int p = pairs_p[tid], q = pairs_q[tid];
                double c = 1.0, s = 0.0;
                if (q < R && p != q) {
                    const double apq = L[p * R + q];
                    if (apq != 0.0) {
                        const double theta = (L[q * R + q] - L[p * R + p]) / (2.0 * apq);
                        const double t = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                        c = 1.0 / sqrt(t * t + 1.0);
                        s = t * c;
                    }
                }
                cs[tid][0] = c;
                cs[tid][1] = s;
            }
            __syncthreads();
            // rows: L <- J^T L
            for (int w = tid; w < (Rp / 2) * R; w += blockDim.x) {
                const int pr = w / R, col = w % R;
                const int p = pairs_p[pr], q = pairs_q[pr];
                if (q < R && p != q) {
                    const double c = cs[pr][0], s = cs[pr][1];
                    const double lp = L[p * R + col], lq = L[q * R + col];
                    L[p * R + col] = c * lp - s * lq;
                    L[q * R + col] = s * lp + c * lq;
                }
            }
            __syncthreads();
            // columns: L <- L J, Q <- Q J
            for (int w = tid; w < (Rp / 2) * R; w += blockDim.x) {
                const int pr = w / R, row = w % R;
                const int p = pairs_p[pr], q = pairs_q[pr];
                if (q < R && p != q) {
                    const double c = cs[pr][0], s = cs[pr][1];
                    const double lp = L[row * R + p], lq = L[row * R + q];
                    L[row * R + p] = c * lp - s * lq;
                    L[row * R + q] = s * lp + c * lq;
                    const double qp = Q[row * R + p], qq = Q[row * R + q];
                    Q[row * R + p] = c * qp - s * qq;
                    Q[row * R + q] = s * qp + c * qq;
                }
            }
            __syncthreads();
        }
    }
    // W = Q diag(1/w with cutoff) Q^T
    __shared__ double wmax;
    if (tid == 0) {
        double m = 0.0;
        for (int i = 0; i < R; ++i) m = fmax(m, fabs(L[i * R + i]));
        wmax = m;
    }
    __syncthreads();
    const double cut = wmax * R * 2.220446049250313e-16;
    for (int p = tid; p < R * R; p += blockDim.x) {
        const int i = p / R, j = p % R;
        double s = 0.0;
        for (int k = 0; k < R; ++k) {
            const double w = L[k * R + k];
            if (fabs(w) > cut) s += Q[i * R + k] * Q[j * R + k] / w;
        }
        Wf[p] = (float)s;
    }
    if (tid == 0) *info = 1;
}

// A = M W (float32) and the columns' sums of squares (WideSum, float64 between
// threads and CTAs). A thread computes 4 rows x 4 columns of a tile staged in
// shared memory, summing over k in increasing order with one FMA per term; A
// may be M. G, if not NULL, is zeroed for the Gram that follows.
//
// Bound by the float32 FMAs at R = 64 (2 I R^2), by HBM at small R. One warp
// per row with two shared loads per FMA took 0.95 ms at 2^20 x 64 and a
// float64 pass for the sums of squares 0.25; together 0.30 here, 0.03 of it the
// sums (four CTAs per SM: at 74 registers, three, it took 0.04 more).
constexpr int kApplyThreads = 256;

struct ApplyShape {
    int R4;      // R rounded up to 4
    int cg, rg;  // column groups of 4, row groups
    int rows;    // rows of a tile
    int stride;  // floats per staged row: R4 + 4, so that neighbouring row groups hit different banks
};
__host__ __device__ inline ApplyShape apply_shape(int R) {
    ApplyShape s;
    s.R4 = (R + 3) & ~3;
    s.cg = s.R4 / 4;
    s.rg = kApplyThreads / s.cg;
    s.rows = 4 * s.rg;
    s.stride = s.R4 + 4;
    return s;
}
inline size_t apply_smem(int R) {
    const ApplyShape s = apply_shape(R);
    const size_t stage = sizeof(float) * ((size_t)s.R4 * s.R4 + (size_t)s.rows * s.stride);
    return std::max(stage, sizeof(double) * 4 * kApplyThreads);
}

// Sum of squares in float64 of the entries of column `c` that a thread of row
// group `rg` has stored. Apart, so that it costs k_apply no registers.
__device__ __noinline__ double stored_squares(const float *A, int64_t I, int R, int c, int rg) {
    const ApplyShape sh = apply_shape(R);
    double v = 0.0;
    for (int64_t i0 = (int64_t)blockIdx.x * sh.rows; i0 < I; i0 += (int64_t)gridDim.x * sh.rows)
        for (int64_t i = i0 + rg; i < I && i < i0 + sh.rows; i += sh.rg) {
            const double x = A[i * R + c];
            v += x * x;
        }
    return v;
}

__global__ void __launch_bounds__(kApplyThreads, 4) k_apply(const float *M, int64_t I, int R,
                                                         const float *__restrict__ Wg, float *A,
                                                         double *__restrict__ colsq, double *__restrict__ G) {
    extern __shared__ __align__(16) unsigned char smem[];
    const ApplyShape sh = apply_shape(R);
    float *W = reinterpret_cast<float *>(smem);  // R4 x R4, zero beyond R
    float *Ms = W + sh.R4 * sh.R4;               // rows x stride, zero beyond R
    const int tid = threadIdx.x;
    const int c = tid % sh.cg * 4, rg = tid / sh.cg;
    if (G && blockIdx.x == 0)
        for (int p = tid; p < R * R; p += kApplyThreads) G[p] = 0.0;
    for (int p = tid; p < sh.R4 * sh.R4; p += kApplyThreads) {
        const int k = p / sh.R4, n = p % sh.R4;
        W[p] = k < R && n < R ? Wg[k * R + n] : 0.f;
    }
    const bool vec = R == sh.R4 && ((reinterpret_cast<uintptr_t>(M) | reinterpret_cast<uintptr_t>(A)) & 15) == 0;
    WideSum sq[4];
    uint32_t seen = 0;  // of all four columns
    const int64_t ntiles = (I + sh.rows - 1) / sh.rows;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t i0 = t * sh.rows;
        const int nr = I - i0 < sh.rows ? (int)(I - i0) : sh.rows;
        __syncthreads();
        if (vec) {
            const float4 *src = reinterpret_cast<const float4 *>(M + i0 * R);
            for (int p = tid; p < nr * sh.cg; p += kApplyThreads)
                *reinterpret_cast<float4 *>(Ms + p / sh.cg * sh.stride + p % sh.cg * 4) = src[p];
        } else {
            for (int p = tid; p < nr * sh.R4; p += kApplyThreads) {
                const int r = p / sh.R4, k = p % sh.R4;
                Ms[r * sh.stride + k] = k < R ? M[(i0 + r) * R + k] : 0.f;
            }
        }
        __syncthreads();
        if (rg >= sh.rg) continue;
        float acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int n = 0; n < 4; ++n) acc[a][n] = 0.f;
        const float *mrow = Ms + rg * sh.stride;  // rows rg + a * sh.rg
        for (int k = 0; k < sh.R4; k += 4) {
            float m[4][4], w[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
                *reinterpret_cast<float4 *>(m[a]) =
                    *reinterpret_cast<const float4 *>(mrow + a * sh.rg * sh.stride + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
                *reinterpret_cast<float4 *>(w[kk]) = *reinterpret_cast<const float4 *>(W + (k + kk) * sh.R4 + c);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int n = 0; n < 4; ++n) acc[a][n] = fmaf(m[a][kk], w[kk][n], acc[a][n]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int r = rg + a * sh.rg;
            if (r >= nr) {
#pragma unroll
                for (int n = 0; n < 4; ++n) acc[a][n] = 0.f;
                continue;
            }
            float *dst = A + (i0 + r) * R + c;
            if (vec) {
                *reinterpret_cast<float4 *>(dst) = make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
            } else {
#pragma unroll
                for (int n = 0; n < 4; ++n)
                    if (c + n < R) dst[n] = acc[a][n];
            }
        }
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const float x[4] = {acc[0][n], acc[1][n], acc[2][n], acc[3][n]};
            sq[n].add(x, x);
            seen |= bits_of(x);
        }
    }
    __syncthreads();
    double *red = reinterpret_cast<double *>(smem);  // [rg][R4]
    if (rg < sh.rg)
#pragma unroll
        for (int n = 0; n < 4; ++n) red[rg * sh.R4 + c + n] = sq[n].value();
    const bool any = __syncthreads_or(seen != 0);
    const auto column_sum = [&]() {
        double v = 0.0;
        for (int g = 0; g < sh.rg; ++g) v += red[g * sh.R4 + tid];
        return v;
    };
    __shared__ bool again[kSolveMaxRank];
    double v = 0.0;
    if (tid < R) {
        v = column_sum();
        again[tid] = !add_sum(&colsq[tid], v, any, (double)I * 0x1p-95);
    }
    if (__syncthreads_or(tid < R && again[tid])) {
        if (rg < sh.rg)
            for (int n = 0; n < 4 && c + n < R; ++n)
                if (again[c + n]) red[rg * sh.R4 + c + n] = stored_squares(A, I, R, c + n, rg);
        __syncthreads();
        if (tid < R && again[tid]) replace_sum(&colsq[tid], v, column_sum());
    }
}

// <M, A> per column (WideSum, float64 between threads and CTAs) -> acc[R]. One
// round of kColdotCtas CTAs per SM, as many as its registers allow.
constexpr int kColdotCtas = 6;
__global__ void __launch_bounds__(256, kColdotCtas) k_coldot(const float *__restrict__ M, const float *__restrict__ A,
                                                   int64_t I, int R, double *__restrict__ acc) {
    __shared__ double red[256];
    const int nsub = 256 / R;
    const int c = threadIdx.x % R, sub = threadIdx.x / R;
    const int64_t first = (int64_t)blockIdx.x * nsub + sub, step = (int64_t)gridDim.x * nsub;
    WideSum d;
    uint32_t seen = 0;
    if (sub < nsub) {
        int64_t i = first;
        for (; i + 3 * step < I; i += 4 * step) {
            float x[4], y[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                x[k] = M[(i + k * step) * R + c];
                y[k] = A[(i + k * step) * R + c];
            }
            d.add(x, y);
            seen |= bits_of(x);
        }
        for (; i < I; i += step) {
            const float x[4] = {M[i * R + c], 0.f, 0.f, 0.f}, y[4] = {A[i * R + c], 0.f, 0.f, 0.f};
            d.add(x, y);
            seen |= bits_of(x);
        }
    }
    red[threadIdx.x] = d.value();
    const bool any = __syncthreads_or(seen != 0);
    const auto column_sum = [&]() {
        double v = 0.0;
        for (int g = 0; g < nsub; ++g) v += red[g * R + threadIdx.x];
        return v;
    };
    __shared__ bool again[128];
    double v = 0.0;
    if (threadIdx.x < R) {
        v = column_sum();
        again[threadIdx.x] = !add_sum(&acc[threadIdx.x], v, any, (double)I * 0x1p-95);
    }
    if (__syncthreads_or(threadIdx.x < R && again[threadIdx.x])) {
        if (sub < nsub && again[c]) {
            double part = 0.0;
            for (int64_t i = first; i < I; i += step) part += (double)M[i * R + c] * (double)A[i * R + c];
            red[threadIdx.x] = part;
        }
        __syncthreads();
        if (threadIdx.x < R && again[threadIdx.x]) replace_sum(&acc[threadIdx.x], v, column_sum());
    }
}

__global__ void __launch_bounds__(256) k_fit_final(double normX2, const GramPtrs gp, int N, int R,
                                                   const double *__restrict__ lambda,
                                                   const double *__restrict__ dots, double *__restrict__ fit) {
    __shared__ double part[8], inner[8];
    double s = 0.0;
    for (int p = threadIdx.x; p < R * R; p += 256) {
        double v = 1.0;
        for (int k = 0; k < N; ++k) v *= gp.g[k][p];
        s += lambda[p / R] * v * lambda[p % R];
    }
    double d = threadIdx.x < R ? lambda[threadIdx.x] * dots[threadIdx.x] : 0.0;
    for (int o = 16; o >= 1; o >>= 1) {
        s += __shfl_xor_sync(kFull, s, o);
        d += __shfl_xor_sync(kFull, d, o);
    }
    if ((threadIdx.x & 31) == 0) {
        part[threadIdx.x >> 5] = s;
        inner[threadIdx.x >> 5] = d;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double xh2 = 0.0, in = 0.0;
        for (int i = 0; i < 8; ++i) {
            xh2 += part[i];
            in += inner[i];
        }
        double r2 = normX2 + xh2 - 2.0 * in;
        if (r2 < 0.0) r2 = 0.0;
        *fit = 1.0 - sqrt(r2) / sqrt(normX2);
    }
}

// WideSum per thread, float64 between threads: bound by the read of v (in float64
// throughout, 8M values took 36 us; now 22).
__global__ void __launch_bounds__(256) k_norm2(const float *__restrict__ v, int64_t n, double *__restrict__ out) {
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    WideSum d;
    uint32_t seen = 0;
    int64_t i = first;
    for (; i + 3 * step < n; i += 4 * step) {
        const float x[4] = {v[i], v[i + step], v[i + 2 * step], v[i + 3 * step]};
        d.add(x, x);
        seen |= bits_of(x);
    }
    for (; i < n; i += step) {
        const float x[4] = {v[i], 0.f, 0.f, 0.f};
        d.add(x, x);
        seen |= bits_of(x);
    }
    const auto warp_sum = [](double s) {
        for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        return s;
    };
    const bool lead = (threadIdx.x & 31) == 0;
    const double s = warp_sum(d.value());
    const bool any = __any_sync(kFull, seen != 0);
    bool again = false;
    if (lead) again = !add_sum(out, s, any, 0x1p-63);  // up to 2^32 values, in batches
    if (__any_sync(kFull, again)) {
        double t = 0.0;
        for (i = first; i < n; i += step) t += (double)v[i] * (double)v[i];
        t = warp_sum(t);
        if (lead) replace_sum(out, s, t);
    }
}

// out = sum of the private output copies (n floats each, n % 4 == 0,
// 16-byte aligned), one float4 per thread and step; copies summed in order.
__global__ void k_sum_copies(const float4 *__restrict__ copies, int ncopies, int64_t n4, float4 *__restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
        float4 a = copies[i];
        for (int c = 1; c < ncopies; ++c) {
            const float4 b = copies[(int64_t)c * n4 + i];
            a.x += b.x;
            a.y += b.y;
            a.z += b.z;
            a.w += b.w;
        }
        out[i] = a;
    }
}

}  // namespace

cudaError_t launch_sum_copies(const float *copies, int ncopies, int64_t n, float *out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int64_t n4 = n / 4;
    k_sum_copies<<<grid_cap(n4, 256), 256, 0, s>>>(reinterpret_cast<const float4 *>(copies), ncopies, n4,
                                                    reinterpret_cast<float4 *>(out));
    return cudaGetLastError();
}

cudaError_t launch_zero(float *p, int64_t n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if ((reinterpret_cast<uintptr_t>(p) & 15) == 0 && (n & 3) == 0) {
        k_zero4<<<grid_cap(n / 4, 256), 256, 0, s>>>(reinterpret_cast<float4 *>(p), n / 4);
    } else {
        k_zero1<<<grid_cap(n, 256), 256, 0, s>>>(p, n);
    }
    return cudaGetLastError();
}

namespace {
struct ZeroList {
    float4 *p[MAXN];
    int64_t end[MAXN];  // of array k among all of them, one after another
    int count;
};
__global__ void k_zero_list(const ZeroList z) {
    const int64_t total = z.end[z.count - 1];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int k = 0;
        while (i >= z.end[k]) ++k;
        z.p[k][k > 0 ? i - z.end[k - 1] : i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}
}  // namespace

// Zeroes several 16-byte aligned arrays, of multiples of 4 floats, in one launch.
cudaError_t launch_zero_list(float *const *p, const int64_t *n, int count, cudaStream_t s) {
    ZeroList z = {};
    int64_t total = 0;
    for (int i = 0; i < count; ++i) {
        if (!p[i] || n[i] <= 0) continue;
        total += n[i] / 4;
        z.p[z.count] = reinterpret_cast<float4 *>(p[i]);
        z.end[z.count++] = total;
    }
    if (z.count == 0) return cudaSuccess;
    k_zero_list<<<grid_cap(total, 256), 256, 0, s>>>(z);
    return cudaGetLastError();
}

cudaError_t launch_convert(const float *src, void *dst, blco_dtype dt, int64_t n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (dt == BLCO_BF16)
        k_to_bf16<<<grid_cap(n, 256), 256, 0, s>>>(src, static_cast<__nv_bfloat16 *>(dst), n);
    else if (dt == BLCO_F16)
        k_to_f16<<<grid_cap(n, 256), 256, 0, s>>>(src, static_cast<__half *>(dst), n);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

namespace {

struct GramLaunch {
    dim3 grid;
    int threads;
    size_t shm;
    int64_t rows;
};

int gram_ctas(int R) { return R >= kGramWideRank ? 2 : 3; }

// as many CTAs as are resident in total, each over a contiguous range of rows
GramLaunch gram_launch(int64_t I, int R) {
    const GramShape sh = gram_shape(R);
    const int64_t ctas_max = std::max<int64_t>(1, (int64_t)sm_count() * gram_ctas(R) / sh.ny);
    GramLaunch g;
    g.rows = (I + ctas_max - 1) / ctas_max;
    g.rows = std::max<int64_t>(kGramRows, (g.rows + kGramRows - 1) / kGramRows * kGramRows);
    g.threads = (sh.groups * sh.per_y + 31) / 32 * 32;
    g.shm = sizeof(float) * kGramRows * sh.R4 + sizeof(double) * sh.groups * sh.per_y * 16;
    g.grid = dim3((unsigned)((I + g.rows - 1) / g.rows), (unsigned)sh.ny);
    return g;
}

template <typename T, bool SCALE, int CTAS>
cudaError_t run_gram_as(const T *A, T *A_out, int64_t I, int R, const double *colsq, double *lambda, double *G,
                        cudaStream_t s) {
    const GramLaunch g = gram_launch(I, R);
    auto kern = k_gram<T, SCALE, CTAS>;
    cudaError_t e = allow_smem((const void *)kern, g.shm);
    if (e != cudaSuccess) return e;
    kern<<<g.grid, g.threads, g.shm, s>>>(A, A_out, I, R, g.rows, colsq, lambda, G);
    return cudaGetLastError();
}

template <typename T, bool SCALE>
cudaError_t run_gram(const void *A, T *A_out, int64_t I, int R, const double *colsq, double *lambda, double *G,
                     cudaStream_t s) {
    const T *a = static_cast<const T *>(A);
    return gram_ctas(R) == 2 ? run_gram_as<T, SCALE, 2>(a, A_out, I, R, colsq, lambda, G, s)
                             : run_gram_as<T, SCALE, 3>(a, A_out, I, R, colsq, lambda, G, s);
}

__global__ void k_zero_lambda(double *lambda, double *G, int R) {
    for (int i = threadIdx.x; i < R; i += blockDim.x) lambda[i] = 0.0;
    if (G)
        for (int i = threadIdx.x; i < R * R; i += blockDim.x) G[i] = 0.0;
}

// The CP-ALS update of one factor with its scratch given: R x R floats, R doubles.
cudaError_t run_update(const double *const *grams, int N, int mode, int R, const float *M, int64_t I, float *A,
                       double *lambda, double *G_out, int32_t *info, float *Wf, double *colsq, cudaStream_t s) {
    GramPtrs gp;
    for (int k = 0; k < MAXN; ++k) gp.g[k] = k < N ? grams[k] : nullptr;
    const size_t shm_solve = sizeof(double) * 2 * R * R;
    cudaError_t e = allow_smem((const void *)k_solve_small, shm_solve);
    if (e != cudaSuccess) return e;
    k_solve_small<<<1, kSolveThreads, shm_solve, s>>>(gp, N, mode, R, Wf, colsq, info);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (I <= 0) {
        k_zero_lambda<<<1, 256, 0, s>>>(lambda, G_out, R);
        return cudaGetLastError();
    }
    const size_t shm = apply_smem(R);
    e = allow_smem((const void *)k_apply, shm);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (I + apply_shape(R).rows - 1) / apply_shape(R).rows;
    const int64_t ctas = std::min<int64_t>(tiles, (int64_t)sm_count() * 4);
    k_apply<<<(unsigned)ctas, kApplyThreads, shm, s>>>(M, I, R, Wf, A, colsq, G_out);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return run_gram<float, true>(A, A, I, R, colsq, lambda, G_out, s);
}

}  // namespace

cudaError_t launch_gram(const void *A, blco_dtype fdt, int64_t I, int R, double *G, cudaStream_t s) {
    k_zero_d<<<1, 256, 0, s>>>(G, R * R);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || I <= 0) return e;
    switch (fdt) {
        case BLCO_F32: return run_gram<float, false>(A, nullptr, I, R, nullptr, nullptr, G, s);
        case BLCO_BF16: return run_gram<__nv_bfloat16, false>(A, nullptr, I, R, nullptr, nullptr, G, s);
        case BLCO_F16: return run_gram<__half, false>(A, nullptr, I, R, nullptr, nullptr, G, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_cpals_update(const double *const *grams, int N, int mode, int R, const float *M, int64_t I,
                                float *A, double *lambda, double *G_out, int32_t *info, cudaStream_t s) {
    unsigned char *buf = nullptr;
    const size_t wf = (sizeof(float) * R * R + 255) / 256 * 256;
    cudaError_t e = cudaMallocAsync(&buf, wf + sizeof(double) * R, s);
    if (e != cudaSuccess) return e;
    e = run_update(grams, N, mode, R, M, I, A, lambda, G_out, info, reinterpret_cast<float *>(buf),
                   reinterpret_cast<double *>(buf + wf), s);
    cudaFreeAsync(buf, s);
    return e;
}

cudaError_t launch_cpals_fit(double normX2, const double *const *grams, int N, int R, const double *lambda,
                             const float *M, const float *A, int64_t I, double *fit, cudaStream_t s) {
    GramPtrs gp;
    for (int k = 0; k < MAXN; ++k) gp.g[k] = k < N ? grams[k] : nullptr;
    double *dots = nullptr;
    cudaError_t e = cudaMallocAsync(&dots, sizeof(double) * R, s);
    if (e != cudaSuccess) return e;
    k_zero_d<<<1, 128, 0, s>>>(dots, R);
    if (I > 0) {
        const int64_t ctas = std::min<int64_t>(grid_cap(I, 256 / R), (int64_t)sm_count() * kColdotCtas);
        k_coldot<<<(unsigned)ctas, 256, 0, s>>>(M, A, I, R, dots);
    }
    k_fit_final<<<1, 256, 0, s>>>(normX2, gp, N, R, lambda, dots, fit);
    e = cudaGetLastError();
    cudaFreeAsync(dots, s);
    return e;
}

cudaError_t launch_norm2(const float *v, int64_t n, double *out, cudaStream_t s) {
    k_zero_d<<<1, 32, 0, s>>>(out, 1);
    if (n > 0) k_norm2<<<grid_cap(n, 256), 256, 0, s>>>(v, n, out);
    return cudaGetLastError();
}

cudaError_t launch_norm2_acc(const float *v, int64_t n, double *out, cudaStream_t s) {
    if (n > 0) k_norm2<<<grid_cap(n, 256), 256, 0, s>>>(v, n, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// CP-ALS update without allocation.
//
// Some callers cannot let a library allocate device memory during a call:
// a process that reserved the GPU's memory up front for its own pool (a
// cudaMalloc would fail or escape its accounting), or a latency-critical loop
// where the device-wide synchronization of cudaFree is not acceptable. For
// them the update's scratch (the float32 inverse of V and the column sums of
// squares) lives in one file-scope device array that
// every GPU which loads the library holds until the process exits.
// ---------------------------------------------------------------------------
namespace {

constexpr int kNoAllocMaxRank = 64;
constexpr size_t kNoAllocWfBytes = sizeof(float) * kNoAllocMaxRank * kNoAllocMaxRank;
constexpr size_t kNoAllocColsqOff = (kNoAllocWfBytes + 255) & ~size_t(255);
constexpr size_t kNoAllocScratchBytes = kNoAllocColsqOff + sizeof(double) * kNoAllocMaxRank;

// Shared by every call on a device; holds the previous call's contents.
static __device__ __align__(256) unsigned char g_update_scratch[kNoAllocScratchBytes];

// The array's device address is looked up once per device and context
// (cudaGetSymbolAddress: the host-side name of the array is not a device
// address) and cached with the id of the context it belongs to. A context
// that is destroyed and recreated (cudaDeviceReset) reloads the module,
// possibly at another address; its new id makes the next call look the
// address up again instead of using a stale one.
typedef int (*CtxGetCurrentFn)(void **);
typedef int (*CtxGetIdFn)(void *, unsigned long long *);

struct ScratchCache {
    unsigned long long ctx_id = 0;  // 0: nothing cached
    void *addr = nullptr;
};

std::mutex g_scratch_mutex;
ScratchCache g_scratch[64];
CtxGetCurrentFn g_ctx_current = nullptr;
CtxGetIdFn g_ctx_id = nullptr;
bool g_driver_looked_up = false;

// Id of the calling thread's current context, 0 if unknown.
unsigned long long current_ctx_id() {
    if (!g_driver_looked_up) {
        g_driver_looked_up = true;
        void *f = nullptr, *g = nullptr;
        cudaDriverEntryPointQueryResult q1, q2;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q1) == cudaSuccess &&
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &g, 12000, cudaEnableDefault, &q2) == cudaSuccess &&
            q1 == cudaDriverEntryPointSuccess && q2 == cudaDriverEntryPointSuccess) {
            g_ctx_current = reinterpret_cast<CtxGetCurrentFn>(f);
            g_ctx_id = reinterpret_cast<CtxGetIdFn>(g);
        }
        cudaGetLastError();
    }
    if (!g_ctx_current || !g_ctx_id) return 0;
    void *ctx = nullptr;
    unsigned long long id = 0;
    if (g_ctx_current(&ctx) != 0 || !ctx || g_ctx_id(ctx, &id) != 0) return 0;
    return id;
}

// Device address of g_update_scratch in the current device's context.
cudaError_t update_scratch(unsigned char **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    const unsigned long long id = current_ctx_id();
    ScratchCache &c = g_scratch[dev];
    if (id == 0 || c.ctx_id != id) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_update_scratch);  // also makes the primary context current
        if (e != cudaSuccess) return e;
        c.addr = p;
        c.ctx_id = current_ctx_id();  // 0 (no driver entry points): look up again on every call
    }
    *out = static_cast<unsigned char *>(c.addr);
    return cudaSuccess;
}

}  // namespace

int cpals_update_noalloc_max_rank() { return kNoAllocMaxRank; }

cudaError_t launch_cpals_update_noalloc(const double *const *grams, int N, int mode, int R, const float *M,
                                        int64_t I, float *A, double *lambda, double *G_out, int32_t *info,
                                        cudaStream_t s) {
    if (R < 1 || R > kNoAllocMaxRank) return cudaErrorInvalidValue;
    unsigned char *base = nullptr;
    cudaError_t e = update_scratch(&base);
    if (e != cudaSuccess) return e;
    return run_update(grams, N, mode, R, M, I, A, lambda, G_out, info, reinterpret_cast<float *>(base),
                      reinterpret_cast<double *>(base + kNoAllocColsqOff), s);
}

}  // namespace blco
