// fp64_common.cuh -- device building blocks of the double-precision swarm: gbest
// candidates, uniforms, clamps, Eq. 1 and 2, fitness functions.
#pragma once

#include <cuda_runtime.h>

#include "cupso_device.cuh"
#include "paper_kernels.h"

namespace cupso {

// ---------------------------------------------------------------------------
// Candidate keys
// ---------------------------------------------------------------------------
__device__ __forceinline__ PKey key_none() { return PKey{~0ull, kNoIdx, 0u}; }

__device__ __forceinline__ bool key_less(const PKey& a, const PKey& b) {
    return a.k < b.k || (a.k == b.k && a.i < b.i);
}

__device__ __forceinline__ PKey warp_min_key(PKey a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        PKey b;
        b.k = __shfl_xor_sync(0xFFFFFFFFu, a.k, o);
        b.i = __shfl_xor_sync(0xFFFFFFFFu, a.i, o);
        b.pad = 0u;
        if (key_less(b, a)) a = b;
    }
    return a;
}

// Minimum over the block (every thread returns it). red: >= 32 entries.
__device__ __forceinline__ PKey block_min_key(PKey k, PKey* red) {
    k = warp_min_key(k);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = k;
    __syncthreads();
    if (threadIdx.x < 32) {
        PKey m = threadIdx.x < (blockDim.x + 31) / 32 ? red[threadIdx.x] : key_none();
        m = warp_min_key(m);
        if (threadIdx.x == 0) red[0] = m;
    }
    __syncthreads();
    const PKey r = red[0];
    __syncthreads();
    return r;
}

// ---------------------------------------------------------------------------
// Double precision building blocks
// ---------------------------------------------------------------------------

// Two words -> (m + 1) 2^-53 with m = hi 2^21 + (lo >> 11), in (0, 1], times
// 2^k. The double is assembled from integer parts: exponent from the leading
// bit of v = m + 1 (plus k), the bits below it as the fraction (v <= 2^53, so
// it is exact; callers keep |k| <= 512, so the result stays normal).
__device__ __forceinline__ double u53_pow2(uint32_t hi, uint32_t lo, int k) {
    const unsigned long long v = (((unsigned long long)hi << 21) | (unsigned long long)(lo >> 11)) + 1ull;
    const int lz = __clzll((long long)v);
    const unsigned long long frac = ((v << lz) << 1) >> 12;
    const unsigned long long e = (unsigned long long)(1033 - lz + k);
    return __longlong_as_double((long long)((e << 52) | frac));
}

__device__ __forceinline__ double u53(uint32_t hi, uint32_t lo) { return u53_pow2(hi, lo, 0); }

// c * u53(hi, lo), rounded once: an exponent shift when c = 2^k (exact).
__device__ __forceinline__ double c_times_u53(double c, int cexp, uint32_t hi, uint32_t lo) {
    if (cexp != kNoExp) return u53_pow2(hi, lo, cexp);
    return __dmul_rn(c, u53(hi, lo));
}

// Closed clamp to [lo, hi] with a NaN going to lo, as comparisons of the
// values' order keys (klo, khi: keys of lo, hi). Equal to the floating-point
// comparison form for every a (-0 and +0 compare equal in both), but it runs
// on the integer pipes instead of the FP64 one -- as long as neither step is
// written in a way that the compiler turns back into an FP64 instruction: clearing
// the sign bit becomes one (hence the exclusive or: k = -magnitude for a negative
// a), and so does a test for NaN against constants (hence kinf, the key of infinity,
// as a parameter; a NaN lies above it or, with the sign bit, below every other).
__device__ __forceinline__ double clamp64(double a, double lo, double hi, long long klo, long long khi,
                                          long long kinf) {
    const long long b = __double_as_longlong(a), sign = b >> 63;
    const long long k = (b ^ (sign & 0x7FFFFFFFFFFFFFFFll)) - sign;
    return k < klo ? lo : (k > khi ? (k > kinf ? lo : hi) : a);
}

__device__ __forceinline__ unsigned long long fit_key64(double f) {
    if (f != f) return ~0ull;
    unsigned long long b = (unsigned long long)__double_as_longlong(f);
    if ((b << 1) == 0ull) b = 0ull;  // -0 -> +0
    return (b >> 63) ? ~b : (b | (1ull << 63));
}

template <int FIT>
struct FitAcc64 {
    double acc = 0.0;
    double prev = 0.0;
    __device__ __forceinline__ void add(int d, double x) {
        if constexpr (FIT == kSphere) {
            acc = __fma_rn(x, x, acc);
        } else if constexpr (FIT == kRosenbrock) {
            if (d > 0) {
                const double p = __fma_rn(-prev, prev, x);
                const double q = __dsub_rn(1.0, prev);
                acc = __dadd_rn(acc, __fma_rn(__dmul_rn(100.0, p), p, __dmul_rn(q, q)));
            }
            prev = x;
        } else if constexpr (FIT == kCubicMax) {
            const double h = __fma_rn(__fma_rn(__dsub_rn(x, 0.8), x, -1000.0), x, 8000.0);
            acc = __dadd_rn(acc, h);
        }
    }
    __device__ __forceinline__ double finish() const { return FIT == kCubicMax ? -acc : acc; }
};

// Eq. 1 and Eq. 2 in binary64 with the clamps of Alg. 1 (same order as FP32),
// from the dimension's Philox words. Products that are exact by construction
// (w v with w = 1, c r with c a power of two) are formed without the FP64 pipe.
template <bool W1>
__device__ __forceinline__ void move_one64_t(double& x, double& v, double pb, double g, uint4 r, const SwarmDev64& s) {
    const double cognitive = __dsub_rn(pb, x);
    const double social = __dsub_rn(g, x);
    double vel = W1 ? v : __dmul_rn(s.w, v);
    vel = __fma_rn(c_times_u53(s.c1, s.c1_exp, r.x, r.y), cognitive, vel);
    vel = __fma_rn(c_times_u53(s.c2, s.c2_exp, r.z, r.w), social, vel);
    v = clamp64(vel, s.vlo, s.vmax, s.k_vlo, s.k_vhi, s.k_inf);
    x = clamp64(__dadd_rn(x, v), s.lo, s.hi, s.k_lo, s.k_hi, s.k_inf);
}

// The two forms apart: as one, the product w v is formed (on the narrow FP64 pipe)
// and then not used.
__device__ __forceinline__ void move_one64(double& x, double& v, double pb, double g, uint4 r, const SwarmDev64& s) {
    if (s.w_one) move_one64_t<true>(x, v, pb, g, r, s);
    else move_one64_t<false>(x, v, pb, g, r, s);
}

// ---------------------------------------------------------------------------
// Fitness from per-dimension terms, for the kernels that spread a particle's
// dimensions over threads: the terms are formed in parallel, then one thread
// per particle adds them in order d = 0 .. D-1 (the same operations, in the
// same order, as FitAcc64).
// ---------------------------------------------------------------------------
template <int FIT>
struct FitTerms64 {
    static constexpr bool kNeedsNext = (FIT == kRosenbrock);
    // term of dimension d (x = x_d, xn = x_{d+1}); Rosenbrock: d < D - 1 only
    __device__ static __forceinline__ double term(double x, double xn) {
        if constexpr (FIT == kCubicMax) {
            return __fma_rn(__fma_rn(__dsub_rn(x, 0.8), x, -1000.0), x, 8000.0);
        } else if constexpr (FIT == kRosenbrock) {
            const double p = __fma_rn(-x, x, xn);
            const double q = __dsub_rn(1.0, x);
            return __fma_rn(__dmul_rn(100.0, p), p, __dmul_rn(q, q));
        } else {
            return 0.0;   // sphere: the sum fuses x * x, no separate term
        }
    }
    // sequential sum over d of particle column p (stride P) of X / H
    __device__ static __forceinline__ double sum(const double* X, const double* H, int P, int p, int D) {
        double acc = 0.0;
        if constexpr (FIT == kSphere) {
            for (int d = 0; d < D; ++d) {
                const double x = X[(size_t)d * P + p];
                acc = __fma_rn(x, x, acc);
            }
        } else {
            const int n = FIT == kRosenbrock ? D - 1 : D;
            for (int d = 0; d < n; ++d) acc = __dadd_rn(acc, H[(size_t)d * P + p]);
        }
        return FIT == kCubicMax ? -acc : acc;
    }
};

}  // namespace cupso
