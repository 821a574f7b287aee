// fit_terms.cuh -- a particle's fitness split over threads: the per-dimension
// terms are formed in parallel, one thread per particle adds them in order.
#pragma once

#include <cuda_runtime.h>

#include "cupso_device.cuh"

namespace cupso {

// Fitness from per-dimension terms; sum() equals FitAcc<FIT> over d in order.
template <int FIT>
struct FitTerms {
    // Rosenbrock's term d pairs x_d with x_{d+1}
    static constexpr bool kNeedsNext = (FIT == kRosenbrock);
    // no term array: the sum fuses x * x itself
    static constexpr bool kNoTerm = (FIT == kSphere);
    // SMALL: |x| <= kSmallX
    template <bool SMALL = false>
    __device__ static __forceinline__ float term(float x, float xn) {
        if constexpr (FIT == kRastrigin) {
            return __fmaf_rn(x, x, __fmaf_rn(-10.0f, cosine2pi<SMALL>(x), 10.0f));
        } else if constexpr (FIT == kAckley) {
            return cosine2pi<SMALL>(x);
        } else if constexpr (FIT == kRosenbrock) {
            const float p = __fmaf_rn(-x, x, xn);
            const float q = __fsub_rn(1.0f, x);
            return __fmaf_rn(__fmul_rn(100.0f, p), p, __fmul_rn(q, q));
        } else if constexpr (FIT == kCubicMax) {
            return __fmaf_rn(__fmaf_rn(__fsub_rn(x, 0.8f), x, -1000.0f), x, 8000.0f);
        } else {
            return 0.0f;
        }
    }
    // two dimensions' terms, |x| <= kSmallX (not Rosenbrock's)
    __device__ static __forceinline__ float2 two(float x0, float x1) {
        if constexpr (FIT == kRastrigin || FIT == kAckley) {
            float c0, c1;
            cos2pi_small2(x0, x1, c0, c1);
            if constexpr (FIT == kAckley) return make_float2(c0, c1);
            const f32x2 x = pack2(x0, x1);
            unpack2(fma2(x, x, fma2(both(-10.0f), pack2(c0, c1), both(10.0f))), c0, c1);
            return make_float2(c0, c1);
        } else {
            return make_float2(term<true>(x0, 0.0f), term<true>(x1, 0.0f));
        }
    }
    // particle column p (stride P) of X and H
    __device__ static __forceinline__ float sum(const float* X, const float* H, int P, int p, int D) {
        FitAcc<FIT> a;
        if constexpr (FIT == kSphere) {
#pragma unroll 8
            for (int d = 0; d < D; ++d) {
                const float x = X[d * P + p];
                a.acc = __fmaf_rn(x, x, a.acc);
            }
        } else if constexpr (FIT == kAckley) {
#pragma unroll 8
            for (int d = 0; d < D; ++d) {
                const float x = X[d * P + p];
                a.acc = __fmaf_rn(x, x, a.acc);
                a.acc2 = __fadd_rn(a.acc2, H[d * P + p]);
            }
        } else {
            const int n = FIT == kRosenbrock ? D - 1 : D;
#pragma unroll 8
            for (int d = 0; d < n; ++d) a.acc = __fadd_rn(a.acc, H[d * P + p]);
        }
        return a.finish(D);
    }
};

}  // namespace cupso
