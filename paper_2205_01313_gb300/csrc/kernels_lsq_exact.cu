// kernels_lsq_exact.cu -- the exact least-squares fitness on the CUDA cores:
// f_i = ||A x_i - b||^2 in FP32 or FP64 with every rounding in the oracle's
// order.
//
// Per particle i: for each residual row m, r = -b_m, then r = fma(A_md, x_id, r)
// for d ascending; the squares are summed for m ascending (FP32: f = fma(r, r, f);
// FP64: f = f + r * r, the square rounded first, f rounded to binary32 at the
// end; a product of two binary32 values is exact in binary64).
//
// Only the sum over m ties the rows of a particle together, so the work is
// split there: lsq_resid_kernel computes residuals as a register-tiled matrix
// product over all (row, particle) tiles at once -- each residual one chain
// over d in one thread, as the order demands -- and lsq_sumsq_kernel then adds
// a particle's squares in row order. The residuals pass through a workspace
// R[m][i] of at most kExactWsBytes (half the L2; less where memory is short), a chunk of rows (and of
// particles, for very large swarms) at a time; the running sums carry over from
// chunk to chunk.
//
// Measured on one GB300 (one evaluation; before: a block kept 64 particles x
// all M, 32 blocks for 2048 particles on 152 SMs): FP32 2048 x 500 x 2000
// 1.9 ms -> 101 us (the product 46 TFLOP/s), 8192 x 1024 x 4096 7.88 -> 1.23 ms
// (60 TFLOP/s of about 80 at 128 lanes per SM and clock; the shared-memory reads and
// the doubling of A's values beside the multiplications are the rest); FP64 8192 x 1024 x
// 4096 127 -> 64 ms (1.08 TFLOP/s, the FP64 pipe: A and x are converted once
// per stage, not in every thread's inner loop).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "cupso_device.cuh"
#include "cupso_internal.h"
#include "lsq_internal.h"

namespace cupso {

namespace {

constexpr size_t kExactWsBytes = 64u << 20;   // residual workspace at most
constexpr size_t kExactWsLeast = 1u << 20;    // and where memory is short
constexpr int kResidThreads = 128;            // 16 x 8 threads of TM x TN residuals
constexpr int kBk = 16;                       // dimensions per shared-memory stage
constexpr int kTrimD = 64;                    // FP32: the trimmed inner loop up to here
constexpr int kRowTile = 128;                 // chunk sizes are multiples of this
constexpr int kSumCopiers = 128;              // the threads after the summing warp
constexpr int kSumThreads = 32 + kSumCopiers;
constexpr int kSumStageBytes = 8192;
constexpr int kSumStages = 6;

// TM x TN residuals of one thread: r[a][c] += av[a] * xv[c], one rounding each.
template <typename T, int TM, int TN>
struct Acc;

// FP32 residuals in pairs (fma.rn.f32x2: two independent IEEE fmas per
// instruction: 2048 x 500 x 2000 in 100 us against 157 with scalar fmas).
template <int TM, int TN>
struct Acc<float, TM, TN> {
    unsigned long long r[TM][TN / 2];
    __device__ __forceinline__ void set(int a, float v) {
        unsigned long long p;
        asm("mov.b64 %0, {%1, %1};" : "=l"(p) : "f"(v));
#pragma unroll
        for (int c = 0; c < TN / 2; ++c) r[a][c] = p;
    }
    // av: rows, x2: particles in pairs
    __device__ __forceinline__ void step(const float (&av)[TM], const unsigned long long (&x2)[TN / 2]) {
#pragma unroll
        for (int a = 0; a < TM; ++a) {
            unsigned long long a2;
            asm("mov.b64 %0, {%1, %1};" : "=l"(a2) : "f"(av[a]));
#pragma unroll
            for (int c = 0; c < TN / 2; ++c) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(r[a][c]) : "l"(a2), "l"(x2[c]));
        }
    }
    __device__ __forceinline__ float get(int a, int c) const {
        float lo, hi;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r[a][c / 2]));
        return (c & 1) ? hi : lo;
    }
};

template <int TM, int TN>
struct Acc<double, TM, TN> {
    double r[TM][TN];
    __device__ __forceinline__ void set(int a, double v) {
#pragma unroll
        for (int c = 0; c < TN; ++c) r[a][c] = v;
    }
    __device__ __forceinline__ void step(const double (&av)[TM], const double (&xv)[TN]) {
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
            for (int c = 0; c < TN; ++c) r[a][c] = __fma_rn(av[a], xv[c], r[a][c]);
    }
    __device__ __forceinline__ double get(int a, int c) const { return r[a][c]; }
};

// 4 consecutive T from shared memory (16-byte aligned), floats in pairs.
__device__ __forceinline__ void ld4s(const float* p, unsigned long long* v) {
    const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(p);
    v[0] = q.x; v[1] = q.y;
}
__device__ __forceinline__ void ld4s(const float* p, float* v) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void ld4s(const double* p, double* v) {
    const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4g(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4g(double* p, const double* v) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
}

}  // namespace

// Residuals of rows [m0, m1) (m0 a tile multiple): R[(m - m0) * ldr + i] for the
// particles of this block's tile (FP64: their squares, rounded, so that the sum
// over rows is left with one operation per row on the narrow FP64 pipe). X(i, d) = x[d * ldx + i]; x 16-byte aligned, ldx
// a multiple of 64 (columns past the last particle are computed and never
// summed). vecA: A's rows may be read as float4 (D % 4 == 0, A 16-byte aligned).
//
// Block tile 16 TM rows x 8 TN particles, K in slices of kBk through two shared
// stages: the next slice's A is loaded to registers, its x copied to the other
// stage (FP64: to registers, converted), while the current one is multiplied, so one
// barrier per slice. A's slice is transposed on its way ([k][row], padded), both
// operands are then read as 16-byte vectors that a warp shares (4 row groups x 8
// particle groups). Zeros past D leave a residual's square unchanged.
// TRIM: no multiplications past D and, a warp at a time, past the last row. Zeros take as long: FP64
// 30000 x 2 x 14 75 us an iteration with them, 22 without, 30000 x 2 x 300 343 and 116 (before
// the split into tiles 26 and 183). In FP32 with more dimensions the second form of the
// inner loop costs more than it saves (2048 x 500 x 2000 338 and 347 us for two iterations).
// FUSED: the block goes through all rows, tile by tile, adds its particles' squares itself and
// writes f; no workspace, no second launch (M = 40, one tile: 12.0 -> 10.1 us per iteration of
// a 256 x 16 swarm).
template <typename T, int TM, int TN, bool FUSED, bool TRIM>
__global__ void __launch_bounds__(kResidThreads, TM * TN == 128 ? 2 : TM * TN == 64 ? 3 : 1) lsq_resid_kernel(const float* __restrict__ x, int ldx, int D,
                                                                  const float* __restrict__ A,
                                                                  const float* __restrict__ b, int m0, int m1,
                                                                  T* __restrict__ R, int ldr, int vecA, int N,
                                                                  float* __restrict__ f) {
    constexpr int BM = 16 * TM, BN = 8 * TN;
    constexpr int AK = kBk * BM / kResidThreads;   // A elements per thread and slice: consecutive k of one row
    constexpr int XV = kBk * BN / 4 / kResidThreads;   // float4 of x per thread and slice
    constexpr bool kF32 = sizeof(T) == 4;
    __shared__ __align__(16) T As[2][kBk][BM + 4];
    __shared__ __align__(16) T Xs[2][kBk][BN];
    const int tid = threadIdx.x;
    // a warp's 4 row groups x 8 particle groups, neighbouring lanes in different rows: a
    // quarter of the warp then reads 2 rows' and 4 particles' vectors (8192 x 1024 x 4096:
    // 1572 us an iteration with 1 and 8, 1469 so)
    const int tx = (tid >> 1) & 7, ty = ((tid >> 4) << 1) | (tid & 1);
    const int i0 = blockIdx.x * BN;
    const int arow = tid % BM, ak = (tid / BM) * AK;
    const float* aptr = A;
    float ar[AK];
    float4 xr[XV];
    auto fetch = [&](int k0, int st) {
        const int ka = k0 + ak;
        if (vecA) {
#pragma unroll
            for (int j = 0; j < AK; j += 4) {
                const float4 q = ka + j < D ? *reinterpret_cast<const float4*>(aptr + ka + j) : make_float4(0.f, 0.f, 0.f, 0.f);
                ar[j] = q.x; ar[j + 1] = q.y; ar[j + 2] = q.z; ar[j + 3] = q.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < AK; ++j) ar[j] = ka + j < D ? aptr[ka + j] : 0.0f;
        }
#pragma unroll
        for (int q = 0; q < XV; ++q) {
            const int e = tid + q * kResidThreads, k = k0 + e / (BN / 4);
            const float* from = x + (size_t)k * ldx + i0 + 4 * (e % (BN / 4));
            if constexpr (kF32) {   // straight to the stage
                const unsigned to = (unsigned)__cvta_generic_to_shared(&Xs[st][e / (BN / 4)][4 * (e % (BN / 4))]);
                const unsigned n = k < D ? 16u : 0u;   // zeros past D
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(k < D ? from : x), "r"(n)
                             : "memory");
            } else {
                xr[q] = k < D ? *reinterpret_cast<const float4*>(from) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    };
    auto stage = [&](int st) {
#pragma unroll
        for (int j = 0; j < AK; ++j) As[st][ak + j][arow] = (T)ar[j];
        if constexpr (kF32) asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
        for (int q = 0; q < (kF32 ? 0 : XV); ++q) {
            const int e = tid + q * kResidThreads;
            const T v[4] = {(T)xr[q].x, (T)xr[q].y, (T)xr[q].z, (T)xr[q].w};
            st4g(&Xs[st][e / (BN / 4)][4 * (e % (BN / 4))], v);
        }
    };
    // the thread's rows ty * 4 + j (+ 64) and particles tx * 4 + j (+ 32, 64, 96)
    auto row_of = [&](int a) { return (a / 4) * (BM * 4 / TM) + ty * 4 + a % 4; };
    Acc<T, TM, TN> acc;
    const int slices = (D + kBk - 1) / kBk;
    // acc = the residuals of the tile at row mt
    auto residuals = [&](int mt) {
        aptr = A + (size_t)min(mt + arow, m1 - 1) * (size_t)D;   // rows past m1 are computed, not stored
        // the rows of a warp lie together, so that one past the last row need not multiply
        const bool busy = mt + (tid >> 5) * 16 < m1;
#pragma unroll
        for (int a = 0; a < TM; ++a) {
            const int m = mt + row_of(a);
            acc.set(a, m < m1 ? -(T)b[m] : (T)0);
        }
        fetch(0, 0);
        stage(0);
        __syncthreads();
        for (int s = 0; s < slices; ++s) {
            const int st = s & 1;
            if (s + 1 < slices) fetch((s + 1) * kBk, st ^ 1);
            auto multiply = [&](int k) {
                T av[TM];
                std::conditional_t<kF32, unsigned long long, T> xv[kF32 ? TN / 2 : TN];
#pragma unroll
                for (int a = 0; a < TM; a += 4) ld4s(&As[st][k][(a / 4) * (BM * 4 / TM) + ty * 4], av + a);
#pragma unroll
                for (int c = 0; c < TN; c += 4) ld4s(&Xs[st][k][(c / 4) * (BN * 4 / TN) + tx * 4], xv + (kF32 ? c / 2 : c));
                acc.step(av, xv);
            };
            const int kn = TRIM ? (busy ? min(kBk, D - s * kBk) : 0) : kBk;
            if (kn == kBk) {
#pragma unroll
                for (int k = 0; k < kBk; ++k) multiply(k);
            } else {
#pragma unroll 2
                for (int k = 0; k < kn; ++k) multiply(k);
            }
            if (s + 1 < slices) stage(st ^ 1);   // the other stage: read last before the previous barrier
            __syncthreads();
        }
    };
    if constexpr (FUSED) {
        __shared__ __align__(16) T Rs[BM][BN + 4];
        T sum = (T)0;
        for (int mt = m0; mt < m1; mt += BM) {
            residuals(mt);   // with barriers between the last tile's sums and the next one's Rs
#pragma unroll
            for (int a = 0; a < TM; ++a)
#pragma unroll
                for (int c = 0; c < TN; ++c) Rs[row_of(a)][(c / 4) * (BN * 4 / TN) + tx * 4 + c % 4] = acc.get(a, c);
            __syncthreads();
            if (tid < BN) {
                const int rows = min(BM, m1 - mt);
#pragma unroll 8
                for (int m = 0; m < rows; ++m) {
                    const T r = Rs[m][tid];
                    if constexpr (sizeof(T) == 8) sum = __dadd_rn(sum, __dmul_rn(r, r));
                    else sum = __fmaf_rn(r, r, sum);
                }
            }
        }
        if (tid < BN && i0 + tid < N) {
            if constexpr (sizeof(T) == 8) f[i0 + tid] = __double2float_rn(sum);
            else f[i0 + tid] = sum;
        }
    } else {
        const int mt = m0 + blockIdx.y * BM;
        residuals(mt);
#pragma unroll
        for (int a = 0; a < TM; ++a) {
            const int m = mt + row_of(a);
            if (m >= m1) continue;
            T* row = R + (size_t)(m - m0) * (size_t)ldr + i0;
#pragma unroll
            for (int c = 0; c < TN; c += 4) {
                T v[4] = {acc.get(a, c), acc.get(a, c + 1), acc.get(a, c + 2), acc.get(a, c + 3)};
                if constexpr (sizeof(T) == 8) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) v[e] = __dmul_rn(v[e], v[e]);
                }
                st4g(row + (c / 4) * (BN * 4 / TN) + tx * 4, v);
            }
        }
    }
}

// carry[i] (+)= the squares of R[0 .. rows - 1][i] (FP64: R itself) in row order; the last chunk
// rounds the sum into f[i]. A block takes 32 particles: four warps copy the
// rows into a ring of kSumStages shared stages ahead of warp 0, which adds one
// particle per lane -- a dependent chain of `rows` operations that no split can
// shorten, so only the loads are taken off it.
template <typename T>
__global__ void __launch_bounds__(kSumThreads) lsq_sumsq_kernel(const T* __restrict__ R, int ldr, int rows, int N,
                                                                T* __restrict__ carry, int first, int last,
                                                                float* __restrict__ f) {
    constexpr int kRows = kSumStageBytes / (32 * (int)sizeof(T));   // rows per stage
    constexpr int kVec = 16 / (int)sizeof(T);
    constexpr int kCopies = kSumStageBytes / 16 / kSumCopiers;
    constexpr int kAhead = 16;
    static_assert(kRows % kAhead == 0 && kSumStageBytes % (16 * kSumCopiers) == 0, "whole groups");
    __shared__ __align__(16) T ring[kSumStages][kRows][32];
    const int tid = threadIdx.x, i0 = blockIdx.x * 32, i = i0 + tid;
    const int stages = (rows + kRows - 1) / kRows;
    auto issue = [&](int st) {
        if (st < stages && tid >= 32) {
#pragma unroll
            for (int q = 0; q < kCopies; ++q) {
                const int e = tid - 32 + q * kSumCopiers, rr = e / (32 / kVec), col = (e % (32 / kVec)) * kVec;
                const int row = st * kRows + rr;
                if (row < rows) {
                    const unsigned sa = (unsigned)__cvta_generic_to_shared(&ring[st % kSumStages][rr][col]);
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa),
                                 "l"(R + (size_t)row * (size_t)ldr + i0 + col)
                                 : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    T acc = (T)0;
    if (tid < 32 && !first && i < N) acc = carry[i];
#pragma unroll
    for (int st = 0; st < kSumStages - 1; ++st) issue(st);
    for (int st = 0; st < stages; ++st) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kSumStages - 2) : "memory");
        __syncthreads();   // every thread's copies of stage st have landed; stage st - 1 is read
        issue(st + kSumStages - 1);
        if (tid < 32) {
            const int n = min(kRows, rows - st * kRows);
            const T(*row)[32] = ring[st % kSumStages];
            auto add = [&](T v) {
                if constexpr (sizeof(T) == 8) acc = __dadd_rn(acc, v);
                else acc = __fmaf_rn(v, v, acc);
            };
            if (n == kRows) {   // the next kAhead rows' values are read while these are added
                T v[kAhead], w[kAhead];
#pragma unroll
                for (int e = 0; e < kAhead; ++e) v[e] = row[e][tid];
#pragma unroll
                for (int rr = kAhead; rr <= kRows; rr += kAhead) {
                    if (rr < kRows) {
#pragma unroll
                        for (int e = 0; e < kAhead; ++e) w[e] = row[rr + e][tid];
                    }
#pragma unroll
                    for (int e = 0; e < kAhead; ++e) add(v[e]);
#pragma unroll
                    for (int e = 0; e < kAhead; ++e) v[e] = w[e];
                }
            } else {
                for (int rr = 0; rr < n; ++rr) add(row[rr][tid]);
            }
        }
    }
    if (tid < 32 && i < N) {
        if (!last) carry[i] = acc;
        else if constexpr (sizeof(T) == 8) f[i] = __double2float_rn(acc);
        else f[i] = acc;
    }
}

namespace {

size_t align256(size_t n) { return (n + 255) / 256 * 256; }

// The workspace's particles (a multiple of 128) and rows (of kRowTile) for N
// particles and M rows: everything when it fits, else fewer rows, and fewer
// particles only when one row tile of all of them does not fit.
struct ExactChunk {
    int particles, rows;
};
ExactChunk exact_chunk(int N, int M, size_t esz, size_t ws_most) {
    const long long Np = ((long long)N + 127) / 128 * 128;
    const long long most = (long long)(ws_most / (esz * kRowTile)) / 128 * 128;   // 131072 or 65536 particles of 64 MB
    const long long pc = std::min(Np, most);
    const long long all = ((long long)M + kRowTile - 1) / kRowTile * kRowTile;
    const long long fit = (long long)(ws_most / ((size_t)pc * esz)) / kRowTile * kRowTile;
    return ExactChunk{(int)pc, (int)std::min(all, fit)};
}

// The rows that one tile takes, so that the block adds its particles' squares itself: 64 of a small
// tile, in FP32 128 of a large one. 300 x 24 x 100 11.0 us an iteration against 13.3, 8192 x 60 x
// 128 17.0 and 19.2; with more dimensions 128 x 64 tiles and the second launch are faster, 8192 x
// 256 x 128 38.9 and 36.3.
bool one_tile(int M, int D, bool fp64) { return M <= 64 || (!fp64 && M <= 128 && D <= 128); }

template <typename T, int TM, int TN, bool FUSED = false>
void launch_resid(const float* x, int ldx, int Np, int D, const float* A, const float* b, int m0, int m1, T* R,
                  cudaStream_t st, int N = 0, float* f = nullptr) {
    const int vecA = D % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15u) == 0;
    const dim3 grid((unsigned)(Np / (8 * TN)), FUSED ? 1u : (unsigned)((m1 - m0 + 16 * TM - 1) / (16 * TM)));
    if (sizeof(T) == 8 || D <= kTrimD)
        lsq_resid_kernel<T, TM, TN, FUSED, true><<<grid, kResidThreads, 0, st>>>(x, ldx, D, A, b, m0, m1, R, Np, vecA, N, f);
    else
        lsq_resid_kernel<T, TM, TN, FUSED, false><<<grid, kResidThreads, 0, st>>>(x, ldx, D, A, b, m0, m1, R, Np, vecA, N, f);
}

template <typename T>
cudaError_t exact_launch(const float* x, int ldx, int N, int D, const float* A, const float* b, int M, float* f,
                         void* ws, size_t ws_most, int num_sms, cudaStream_t st) {
    if (ldx % 128 != 0 || ldx < N || (reinterpret_cast<uintptr_t>(x) & 15u) != 0) return cudaErrorInvalidValue;
    const bool one = one_tile(M, D, sizeof(T) == 8);
    if (one || !ws) {
        if (M <= 64 || !one || sizeof(T) == 8) launch_resid<T, 4, 4, true>(x, ldx, (N + 127) / 128 * 128, D, A, b, 0, M, nullptr, st, N, f);
        else if constexpr (sizeof(T) == 4)
            launch_resid<T, 8, 4, true>(x, ldx, (N + 127) / 128 * 128, D, A, b, 0, M, nullptr, st, N, f);
        return cudaGetLastError();
    }
    const ExactChunk ch = exact_chunk(N, M, sizeof(T), ws_most);
    T* carry = static_cast<T*>(ws);
    T* R = reinterpret_cast<T*>(static_cast<char*>(ws) + align256(sizeof(T) * (size_t)ch.particles));
    for (int p0 = 0; p0 < N; p0 += ch.particles) {
        const int n = std::min(ch.particles, N - p0), np = (n + 127) / 128 * 128;
        for (int m0 = 0; m0 < M; m0 += ch.rows) {
            const int m1 = m0 + std::min(ch.rows, M - m0);
            if constexpr (sizeof(T) == 8) {
                launch_resid<T, 4, 4>(x + p0, ldx, np, D, A, b, m0, m1, R, st);
            } else {
                // 128 x 64 tiles once they cover half the SMs (1024 x 1024 x 1024, 128 of them:
                // 70 us against 97 with 64 x 32 tiles), the small ones below (1024 x 64 x 512,
                // 64 large tiles: 6.3 us against 8.3). 128 x 128 tiles take a fifth less time for
                // the same residuals (half the shared-memory reads per product), so they run
                // where the tiles of the fullest SM come to less at that rate: an iteration of
                // 8192 x 1024 x 4096 1279 us against 1471, 2048 x 500 x 2000 136 against 142;
                // 4000 x 300 x 1200, 3 tiles against 5, 112 against 105
                // and the SMs mostly get two (8000 x 16 x 130, 126 tiles: 16.9 against 15.7)
                const long long rows = (m1 - m0 + 127) / 128, big = (long long)(np / 64) * rows;
                const long long wide = (long long)(np / 128) * rows;
                const long long of128 = (wide + num_sms - 1) / num_sms, of64 = (big + num_sms - 1) / num_sms;
                if (5 * of128 < 3 * of64 && 2 * wide >= 3 * num_sms)
                    launch_resid<T, 8, 16>(x + p0, ldx, np, D, A, b, m0, m1, R, st);
                else if (2 * big >= num_sms) launch_resid<T, 8, 8>(x + p0, ldx, np, D, A, b, m0, m1, R, st);
                else launch_resid<T, 4, 4>(x + p0, ldx, np, D, A, b, m0, m1, R, st);
            }
            lsq_sumsq_kernel<T><<<(n + 31) / 32, kSumThreads, 0, st>>>(R, np, m1 - m0, n, carry, m0 == 0, m1 == M, f + p0);
            const cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            if (m1 == M) break;
        }
    }
    return cudaSuccess;
}

// Whether the kernel that goes through all rows in the block (FUSED) is used for its own sake
// where the rows need more than a tile.
//  * `once` (an evaluation): it needs no workspace, and an allocation of more than a megabyte
//    costs about 110 us, most of it once `front` is that large anyway, where small ones come out
//    of memory the process has mapped (3000 x 8 x 500 37 us in the old kernel, 163 with a
//    workspace, 32 so). It loses the SMs that blocks of 32 particles leave idle, and in FP32 the
//    rate of larger tiles: estimated, in us, from 0.4 (FP32; 9.3 FP64) a slice and tile and 0.9 (6)
//    for a tile's sums; sweep over N 64 .. 100000, D 2 .. 1000, M 65 .. 4000.
//  * in a swarm's iterations: with few dimensions and many particles the residuals' way through
//    memory is longer than their product (an iteration of 100000 x 30 x 300 117 us with a
//    workspace, 110 in the old kernel, 92 so; 100000 x 2 x 4000 about 700 and 410).
bool fused_anyway(int N, int D, int M, bool fp64, bool once, size_t front, size_t ws, int num_sms) {
    const double share = (N + 31) / 32 / (double)num_sms;   // blocks per SM
    if (!once) return !fp64 && (D <= 16 ? share >= 2.0 : D <= 32 && share >= 12.0);
    const double tiles = (M + 63) / 64, slices = D / 16.0;
    const double idle = std::ceil(share) - share, short_of = std::max(0.0, 1.0 - share);
    const double loss = fp64 ? tiles * (9.3 * slices + 6.0) * idle
                             : tiles * ((0.4 * slices + 0.9) * short_of + 0.15 * slices * share);
    constexpr size_t kSmall = 1u << 20;
    return loss <= (front > kSmall ? 40.0 : front + ws > kSmall ? 110.0 : 3.0);
}

}  // namespace

cudaError_t lsq_exact_alloc(void** p, size_t front, int N, int D, int M, bool fp64, bool once, int num_sms, void** ws,
                            size_t* ws_most) {
    const size_t esz = fp64 ? 8 : 4;
    *ws = nullptr;
    *ws_most = 0;
    for (size_t most = one_tile(M, D, fp64) ? 0 : kExactWsBytes; most >= kExactWsLeast; most /= 4) {
        const ExactChunk ch = exact_chunk(N, M, esz, most);
        const size_t bytes = align256(esz * (size_t)ch.particles) + esz * (size_t)ch.particles * (size_t)ch.rows;
        if (fused_anyway(N, D, M, fp64, once, front, bytes, num_sms)) break;
        const cudaError_t e = cudaMalloc(p, front + bytes);
        if (e == cudaSuccess) {
            *ws = static_cast<char*>(*p) + front;
            *ws_most = most;
        }
        if (e != cudaErrorMemoryAllocation) return e;
        cudaGetLastError();
    }
    return cudaMalloc(p, front);
}

cudaError_t lsq_exact_launch(const float* x, int ldx, int N, int D, const float* A, const float* b, int M, bool fp64,
                             float* f, void* ws, size_t ws_most, int num_sms, cudaStream_t st) {
    return fp64 ? exact_launch<double>(x, ldx, N, D, A, b, M, f, ws, ws_most, num_sms, st)
                : exact_launch<float>(x, ldx, N, D, A, b, M, f, ws, ws_most, num_sms, st);
}

}  // namespace cupso
