// cupso_lsq.cu -- host side of the least-squares fitness.
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>

#include "../../include/cupso.h"
#include "cupso_device.cuh"
#include "cupso_internal.h"
#include "lsq_internal.h"

using namespace cupso;

namespace {

size_t up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Largest magnitude in x[0 .. n - 1] as the bits of a float (0 before the first
// launch; non-negative floats order as their bits, NaN is skipped).
__global__ void __launch_bounds__(256) absmax_kernel(const float* __restrict__ x, size_t n, int vec,
                                                     unsigned int* __restrict__ out) {
    float v = 0.0f;
    const size_t stride = (size_t)gridDim.x * blockDim.x, t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t done = 0;
    if (vec) {
        const float4* x4 = reinterpret_cast<const float4*>(x);
        const size_t n4 = n / 4;
#pragma unroll 4
        for (size_t e = t; e < n4; e += stride) {
            const float4 q = x4[e];
            v = fmaxf(v, fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)), fmaxf(fabsf(q.z), fabsf(q.w))));
        }
        done = 4 * n4;
    }
    for (size_t e = done + t; e < n; e += stride) v = fmaxf(v, fabsf(x[e]));
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(v));
}

// The FP8 scale that brings a largest magnitude to the e4m3 limit.
__device__ __forceinline__ float fp8_scale(float amax) { return amax > 0.0f ? 448.0f / amax : 1.0f; }

// Both operands of the product from row-major sources, one warp per row:
//  * rows 0 .. Mp - 1 of A: as BF16, or scaled by the row's own factor and
//    rounded to FP8 e4m3 (448 / its largest magnitude; the row is read twice, the
//    second time from L1), with inv[m] = 1 / (sx * that factor), 0 past M; and
//    negb[m] = roff[m] = -b[m], 0 past M (negation is exact, so y + negb[m]
//    rounds exactly as y - b[m]; roff starts at reference point 0);
//  * with X: rows 0 .. Np - 1 of X, as BF16 or X * sx in FP8.
// Zero past the last row and past D. sx: from *xmax (absmax_kernel) when given.
// One pass over either source in one launch; before, A took three (largest
// magnitudes, a scaled FP32 copy, the conversion) and X one of its own: 4000 x
// 1000 and 8192 x 1000 in FP8 46 us for the four, 48 us with the offsets.
struct OperandArgs {
    const float *A, *b, *X;
    int M, Mp, N, Np, D, Kp, vecA, vecX;
    float sx;
    const unsigned int* xmax;
    float *inv, *negb, *roff;
    void *Aq, *Xq;
};

template <bool FP8>
__device__ __forceinline__ void convert_row(const float* __restrict__ src, int D, int Kp, bool vec, float scale, int lane,
                                            char* __restrict__ dst) {
#pragma unroll 4
    for (int k = 4 * lane; k < Kp; k += 128) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (src) {
            if (vec) {
                if (k < D) v = *reinterpret_cast<const float4*>(src + k);
            } else {
                if (k + 0 < D) v.x = src[k + 0];
                if (k + 1 < D) v.y = src[k + 1];
                if (k + 2 < D) v.z = src[k + 2];
                if (k + 3 < D) v.w = src[k + 3];
            }
        }
        if constexpr (FP8) {
            const __nv_fp8x4_e4m3 q(make_float4(v.x * scale, v.y * scale, v.z * scale, v.w * scale));
            *reinterpret_cast<uint32_t*>(dst + k) = q.__x;
        } else {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
            *reinterpret_cast<uint2*>(dst + 2 * (size_t)k) =
                make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
        }
    }
}

template <bool FP8>
__global__ void __launch_bounds__(256) operands_kernel(const OperandArgs p) {
    constexpr size_t esz = FP8 ? 1 : 2;
    const int lane = threadIdx.x & 31;
    const long long rows = (long long)p.Mp + (p.X ? p.Np : 0);
    const float sx = !FP8 ? 1.0f : (p.xmax ? fp8_scale(__uint_as_float(*p.xmax)) : p.sx);
    for (long long r = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += (long long)gridDim.x * 8) {
        if (r < p.Mp) {
            const int m = (int)r;
            const float* src = m < p.M ? p.A + (size_t)m * p.D : nullptr;
            float sa = 1.0f;
            if constexpr (FP8) {
                float v = 0.0f;
                if (src) {
                    if (p.vecA) {
#pragma unroll 4
                        for (int k = 4 * lane; k < p.D; k += 128) {
                            const float4 q = *reinterpret_cast<const float4*>(src + k);
                            v = fmaxf(v, fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)), fmaxf(fabsf(q.z), fabsf(q.w))));
                        }
                    } else {
                        for (int k = lane; k < p.D; k += 32) v = fmaxf(v, fabsf(src[k]));
                    }
                }
                for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
                sa = fp8_scale(v);
            }
            if (lane == 0) {
                const float nb = src ? -p.b[m] : 0.0f;
                p.negb[m] = nb;
                p.roff[m] = nb;
                if constexpr (FP8) p.inv[m] = src ? 1.0f / (sx * sa) : 0.0f;
            }
            convert_row<FP8>(src, p.D, p.Kp, p.vecA, sa, lane, static_cast<char*>(p.Aq) + (size_t)m * p.Kp * esz);
        } else {
            const int i = (int)(r - p.Mp);
            convert_row<FP8>(i < p.N ? p.X + (size_t)i * p.D : nullptr, p.D, p.Kp, p.vecX, sx, lane,
                             static_cast<char*>(p.Xq) + (size_t)i * p.Kp * esz);
        }
    }
}

// out[d * ld + i] = in[i][d] for an N x D row-major matrix.
__global__ void transpose_kernel(const float* __restrict__ in, int N, int D, size_t ld, float* __restrict__ out) {
    __shared__ float t[32][33];
    const int d0 = blockIdx.x * 32, i0 = blockIdx.y * 32;
    for (int k = threadIdx.y; k < 32; k += 8) {
        const int i = i0 + k, d = d0 + threadIdx.x;
        if (i < N && d < D) t[k][threadIdx.x] = in[(size_t)i * D + d];
    }
    __syncthreads();
    for (int k = threadIdx.y; k < 32; k += 8) {
        const int d = d0 + k, i = i0 + threadIdx.x;
        if (i < N && d < D) out[(size_t)d * ld + i] = t[threadIdx.x][k];
    }
}

// f[i] = part[0][i] + part[1][i] + ... in that order, 16 loads in flight.
__global__ void sum_parts_kernel(const float* __restrict__ part, int nparts, int Np, int N, float* __restrict__ f) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        float s = 0.0f;
        for (int k0 = 0; k0 < nparts; k0 += 16) {
            float v[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = k0 + e < nparts ? part[(size_t)(k0 + e) * Np + i] : 0.0f;
#pragma unroll
            for (int e = 0; e < 16; ++e)
                if (k0 + e < nparts) s = __fadd_rn(s, v[e]);
        }
        f[i] = s;
    }
}

}  // namespace

// Everything the tensor-core fitness needs for fixed A, b: operand copies,
// scales, padded b, and the TMA descriptors (built for a given X buffer). With
// X (row-major [N][D]) its operand as well, for an evaluation of given
// positions; the FP8 scale of X is then that of its largest magnitude.
int cupso::lsq_setup_tc(LsqTcState* st, const float* A, const float* b, int M, int D, int Np, bool fp8, float sx,
                        const float* X, int N, cudaStream_t stream) {
    st->fp8 = fp8;
    st->M = M;
    st->D = D;
    st->Np = Np;
    st->Mp = (int)up((size_t)M, 256);
    st->Kp = (int)up((size_t)D, fp8 ? 128 : 64);
    st->sx = fp8 ? sx : 1.0f;
    const size_t esz = fp8 ? 1 : 2;
    const size_t bytes_A = (size_t)st->Mp * st->Kp * esz, bytes_X = (size_t)Np * st->Kp * esz;
    const size_t nparts = (size_t)st->Mp / 128;   // one partial sum per 128 residual rows
    const size_t bytes = up(bytes_A, 256) + up(bytes_X, 256) + up(sizeof(float) * st->Mp, 256) * 3 +
                         up(sizeof(float) * nparts * Np, 256) + 512;
    cudaError_t e = cudaMalloc(&st->arena, bytes);
    if (e != cudaSuccess) return set_cuda_error(e, "cudaMalloc (lsq)"), e == cudaErrorMemoryAllocation ? CUPSO_ERR_OOM : CUPSO_ERR_CUDA;
    char* p = static_cast<char*>(st->arena);
    st->Aq = p; p += up(bytes_A, 256);
    st->Xq = p; p += up(bytes_X, 256);
    st->negb = reinterpret_cast<float*>(p); p += up(sizeof(float) * st->Mp, 256);
    st->roff = reinterpret_cast<float*>(p); p += up(sizeof(float) * st->Mp, 256);
    st->inv = reinterpret_cast<float*>(p); p += up(sizeof(float) * st->Mp, 256);
    st->part = reinterpret_cast<float*>(p); p += up(sizeof(float) * nparts * Np, 256);
    st->status = reinterpret_cast<unsigned int*>(p); p += 256;
    st->roff_stale = reinterpret_cast<int*>(p);
    unsigned int* xmax = st->status + 1;
    e = cudaMemsetAsync(st->status, 0, 512, stream);
    if (e == cudaSuccess) e = lsq_prepare();
    if (e != cudaSuccess) return set_cuda_error(e, "lsq setup"), CUPSO_ERR_CUDA;
    if (!lsq_tc_plan(&st->plan, st->Xq, st->Aq, fp8, Np, st->Mp, st->Kp)) {
        set_last_error("cuTensorMapEncodeTiled unavailable or rejected the operand layout");
        return CUPSO_ERR_UNSUPPORTED;
    }
    auto vec = [&](const float* q) { return D % 4 == 0 && (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
    if (fp8 && X) {
        const size_t n = (size_t)N * D;
        const int grid = (int)std::max<size_t>(1, std::min<size_t>((n + 4095) / 4096, 1216));
        absmax_kernel<<<grid, 256, 0, stream>>>(X, n, (reinterpret_cast<uintptr_t>(X) & 15u) == 0, xmax);
    }
    const OperandArgs args{A, b, X, M, st->Mp, N, Np, D, st->Kp, vec(A), vec(X), st->sx, fp8 && X ? xmax : nullptr,
                           st->inv, st->negb, st->roff, st->Aq, st->Xq};
    const long long rows = (long long)st->Mp + (X ? Np : 0);
    const int grid = (int)std::min<long long>((rows + 7) / 8, 1 << 16);
    if (fp8) operands_kernel<true><<<grid, 256, 0, stream>>>(args);
    else operands_kernel<false><<<grid, 256, 0, stream>>>(args);
    e = cudaGetLastError();
    if (e != cudaSuccess) return set_cuda_error(e, "lsq operands"), CUPSO_ERR_CUDA;
    return CUPSO_OK;
}

void cupso::lsq_free_tc(LsqTcState* st) {
    if (st->arena) cudaFree(st->arena);
    st->arena = nullptr;
}

// f[i] for the positions X(i, k) = src[i * si + k * sk], i < N.
int cupso::lsq_eval_tc(LsqTcState* st, const float* src, size_t si, size_t sk, int N, float* f, cudaStream_t stream) {
    cudaError_t e = lsq_convert(src, si, sk, N, st->D, st->Np, st->Kp, st->fp8, st->sx, st->Xq, stream);
    if (e != cudaSuccess) return set_cuda_error(e, "lsq operand conversion"), CUPSO_ERR_CUDA;
    return lsq_eval_tc_operand(st, N, f, stream);
}

int cupso::lsq_eval_tc_partials(LsqTcState* st, cudaStream_t stream) {
    cudaError_t e = lsq_tc_launch(st->plan, st->roff, st->fp8 ? st->inv : nullptr, st->part, st->status,
                                  2000000000ll, stream);
    if (e != cudaSuccess) return set_cuda_error(e, "lsq tensor-core launch"), CUPSO_ERR_CUDA;
    return CUPSO_OK;
}

int cupso::lsq_eval_tc_operand(LsqTcState* st, int N, float* f, cudaStream_t stream) {
    cudaError_t e = lsq_tc_launch(st->plan, st->negb, st->fp8 ? st->inv : nullptr, st->part, st->status,
                                  2000000000ll, stream);
    const int used = lsq_tc_partials(st->plan);
    if (e == cudaSuccess) {
        sum_parts_kernel<<<std::max(1, std::min(1024, (N + 255) / 256)), 256, 0, stream>>>(st->part, used, st->Np, N, f);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return set_cuda_error(e, "lsq tensor-core launch"), CUPSO_ERR_CUDA;
    return CUPSO_OK;
}

extern "C" int cupso_lsq_eval(const float* A_dev, const float* b_dev, int M, int D, const float* X_dev, int N,
                              int precision, float* f_out_dev, void* cuda_stream) {
    if (!A_dev || !b_dev || !X_dev || !f_out_dev || M < 1 || D < 1 || N < 1 ||
        precision < CUPSO_LSQ_FP32 || precision > CUPSO_LSQ_FP64) {
        set_last_error("cupso_lsq_eval: invalid argument");
        return CUPSO_ERR_INVALID_ARG;
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (precision == CUPSO_LSQ_FP32 || precision == CUPSO_LSQ_FP64) {
        // the exact kernels read X(i, d) = x[d * ld + i]: transposed into a temporary, with their workspace behind it
        const bool f64 = precision == CUPSO_LSQ_FP64;
        const int ld = (N + 127) / 128 * 128;
        const size_t xbytes = up(sizeof(float) * (size_t)ld * D, 256);
        int dev = 0, sms = 1;
        float* xd = nullptr;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        void* ws = nullptr;
        size_t ws_most = 0;
        if (e == cudaSuccess)
            e = lsq_exact_alloc(reinterpret_cast<void**>(&xd), xbytes, N, D, M, f64, true, sms, &ws, &ws_most);
        if (e != cudaSuccess) return set_cuda_error(e, "cudaMalloc"), CUPSO_ERR_OOM;
        transpose_kernel<<<dim3((D + 31) / 32, (N + 31) / 32), dim3(32, 8), 0, st>>>(X_dev, N, D, (size_t)ld, xd);
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = lsq_exact_launch(xd, ld, N, D, A_dev, b_dev, M, f64, f_out_dev, ws, ws_most, sms, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        cudaFree(xd);
        if (e != cudaSuccess) return set_cuda_error(e, "lsq fp32/fp64"), CUPSO_ERR_CUDA;
        return CUPSO_OK;
    }
    if (!lsq_tc_available()) {
        set_last_error("tensor-core least squares needs cuTensorMapEncodeTiled from the driver");
        return CUPSO_ERR_UNSUPPORTED;
    }
    LsqTcState s{};
    const int Np = (N + 127) / 128 * 128;
    int rc = lsq_setup_tc(&s, A_dev, b_dev, M, D, Np, precision == CUPSO_LSQ_FP8, 1.0f, X_dev, N, st);
    if (rc == CUPSO_OK) rc = lsq_eval_tc_operand(&s, N, f_out_dev, st);
    unsigned int status = 0;
    cudaError_t e = cudaSuccess;
    if (rc == CUPSO_OK) e = cudaMemcpyAsync(&status, s.status, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
    const cudaError_t es = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = es;
    lsq_free_tc(&s);
    if (rc != CUPSO_OK) return rc;
    if (e != cudaSuccess) return set_cuda_error(e, "lsq eval"), CUPSO_ERR_CUDA;
    if (status & kStatusTimeout) return CUPSO_ERR_DEVICE_TIMEOUT;
    return CUPSO_OK;
}
