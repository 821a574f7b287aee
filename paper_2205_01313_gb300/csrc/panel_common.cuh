// panel_common.cuh -- building blocks of the kernels on the panel layout
// (kernels_panel.cu, kernels_batch_panel.cu): copies into the ring, and the fitness
// sum that passes from lane to lane of a particle.
#pragma once

#include <cuda_runtime.h>

#include "cupso_device.cuh"

namespace cupso {

__device__ __forceinline__ void cp16(float4* smem, const float* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// The running fitness sums of lane `src`.
template <int FIT>
__device__ __forceinline__ void pull(FitAcc<FIT>& a, int src) {
    a.acc = __shfl_sync(0xFFFFFFFFu, a.acc, src);
    if constexpr (FIT == kAckley) a.acc2 = __shfl_sync(0xFFFFFFFFu, a.acc2, src);
}

// cos(2 pi x) of four values.
template <bool SMALL>
__device__ __forceinline__ void cosines(const float (&x)[4], float (&c)[4]) {
    if constexpr (SMALL) {
        cos2pi_small2(x[0], x[1], c[0], c[1]);
        cos2pi_small2(x[2], x[3], c[2], c[3]);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) c[k] = cos2pi(x[k]);
    }
}

// Adds the fitness terms of this lane's four dimensions (d0 .. d0 + 3) in the
// oracle's order. The terms themselves do not depend on the running sum
// (Rastrigin's x^2 - 10 cos 2 pi x + 10, Rosenbrock's 100 (x_{d+1} - x_d^2)^2 +
// (1 - x_d)^2, the cubic's Horner value), so every lane computes its own at
// once; only their folding into the sum, which keeps the order over d, passes
// from lane to lane of the particle: in phase k the particle's lane k continues
// the sum of lane k - 1 (lane 0 that of lane L - 1, which ended the previous
// panel). Sphere and Ackley fold x with an fma, as the oracle does. After the
// last phase, lane L - 1 of the particle holds the sum through its panel.
// `carry` is x_{d0 - 1} for the particle's lane 0 (the last value of the
// previous panel), updated here to this panel's last value.
// LAST: the panel may reach past D; those dimensions are not added. SMALL: every
// |x| <= kSmallX.
template <int FIT, int L, bool LAST, bool SMALL = false>
__device__ __forceinline__ void panel_sum(FitAcc<FIT>& a, const float4& X, int d0, int D, int j, int lane_id,
                                          float& carry) {
    const float x[4] = {X.x, X.y, X.z, X.w};
    float t[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    const int base = lane_id - j;
    if constexpr (FIT == kRastrigin) {
        cosines<SMALL>(x, t);
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
            const f32x2 xx = pack2(x[k], x[k + 1]);
            unpack2(fma2(xx, xx, fma2(both(-10.0f), pack2(t[k], t[k + 1]), both(10.0f))), t[k], t[k + 1]);
        }
    } else if constexpr (FIT == kAckley) {
        cosines<SMALL>(x, t);
    } else if constexpr (FIT == kCubicMax) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            t[k] = __fmaf_rn(__fmaf_rn(__fsub_rn(x[k], 0.8f), x[k], -1000.0f), x[k], 8000.0f);
    } else if constexpr (FIT == kRosenbrock) {
        // term of dimension d (d >= 1) from x_{d-1} and x_d
        const float from_left = __shfl_sync(0xFFFFFFFFu, X.w, lane_id - 1 < base ? lane_id : lane_id - 1);
        float prev = j == 0 ? carry : from_left;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float pp = __fmaf_rn(-prev, prev, x[k]);
            const float qq = __fsub_rn(1.0f, prev);
            t[k] = __fmaf_rn(__fmul_rn(100.0f, pp), pp, __fmul_rn(qq, qq));
            prev = x[k];
        }
        carry = __shfl_sync(0xFFFFFFFFu, X.w, base + L - 1);
    }
#pragma unroll
    for (int ph = 0; ph < L; ++ph) {
        pull(a, base + (ph + L - 1) % L);
        if (j == ph) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (LAST && d0 + k >= D) break;
                if constexpr (FIT == kSphere) {
                    a.acc = __fmaf_rn(x[k], x[k], a.acc);
                } else if constexpr (FIT == kAckley) {
                    a.acc = __fmaf_rn(x[k], x[k], a.acc);
                    a.acc2 = __fadd_rn(a.acc2, t[k]);
                } else if constexpr (FIT == kRosenbrock) {
                    if (d0 + k > 0) a.acc = __fadd_rn(a.acc, t[k]);
                } else {
                    a.acc = __fadd_rn(a.acc, t[k]);
                }
            }
        }
    }
}

}  // namespace cupso
