// kernels_state.cu -- the swarm state between the caller's particle-major rows
// and the device layouts, for cupso_get_state / cupso_set_state.
//
// The caller's arrays are [N][D]; the device holds them dimension-major [D][Np]
// or in panels (kernels_panel.cu). Rows travel through a staging buffer on the
// device, a chunk of particles at a time, and are rearranged there: one pass at
// memory speed, beside a host link of 130-170 GB/s. On the host the same
// rearrangement walks one side with a stride of a whole row: 20000 x 48, three
// arrays each way, 9.1 ms of a 9.2 ms load-step-store pass.
//
// Bound by memory: the dimension-major form goes through a 32 x 32 shared tile so
// that both sides are read and written in whole 128-byte lines; in the panel
// form a particle's W values are contiguous on both sides (32 or 64 bytes), so
// each thread moves them directly.
#include <cuda_runtime.h>

#include <algorithm>

#include "cupso_device.cuh"
#include "cupso_internal.h"
#include "stream_common.cuh"

namespace cupso {

namespace {

constexpr int kTileT = 32;

// dst[d * Np + i0 + p] = rows[p * D + d] for p < n, 0 for n <= p < np.
template <typename T>
__global__ void __launch_bounds__(256) pack_rows_kernel(const T* __restrict__ rows, T* __restrict__ dst, int D, size_t Np,
                                                        size_t i0, int n, int np) {
    __shared__ T t[kTileT][kTileT + 1];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int p0 = blockIdx.x * kTileT;
    for (int d0 = blockIdx.y * kTileT; d0 < D; d0 += gridDim.y * kTileT) {
#pragma unroll
        for (int k = ty; k < kTileT; k += 8) {
            const int p = p0 + k, d = d0 + tx;
            t[k][tx] = (p < n && d < D) ? rows[(size_t)p * D + d] : (T)0;
        }
        __syncthreads();
#pragma unroll
        for (int k = ty; k < kTileT; k += 8) {
            const int d = d0 + k, p = p0 + tx;
            if (d < D && p < np) dst[(size_t)d * Np + i0 + p] = t[tx][k];
        }
        __syncthreads();
    }
}

// rows[p * D + d] = src[d * Np + i0 + p], p < n.
template <typename T>
__global__ void __launch_bounds__(256) unpack_rows_kernel(const T* __restrict__ src, T* __restrict__ rows, int D, size_t Np,
                                                          size_t i0, int n) {
    __shared__ T t[kTileT][kTileT + 1];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int p0 = blockIdx.x * kTileT;
    for (int d0 = blockIdx.y * kTileT; d0 < D; d0 += gridDim.y * kTileT) {
#pragma unroll
        for (int k = ty; k < kTileT; k += 8) {
            const int d = d0 + k, p = p0 + tx;
            if (d < D && p < n) t[k][tx] = src[(size_t)d * Np + i0 + p];
        }
        __syncthreads();
#pragma unroll
        for (int k = ty; k < kTileT; k += 8) {
            const int p = p0 + k, d = d0 + tx;
            if (p < n && d < D) rows[(size_t)p * D + d] = t[tx][k];
        }
        __syncthreads();
    }
}

// The same against panels of W: element (d, i) at ((d / W) * Np + i) * W + d % W. D % W == 0.
template <int W, bool PACK>
__global__ void __launch_bounds__(256) panel_rows_kernel(float* __restrict__ rows, float* __restrict__ state, int D,
                                                         size_t Np, size_t i0, int n, int np) {
    const size_t items = (size_t)(D / W) * (size_t)np;
    for (size_t it = (size_t)blockIdx.x * blockDim.x + threadIdx.x; it < items; it += (size_t)gridDim.x * blockDim.x) {
        const size_t q = it / (size_t)np;
        const int p = (int)(it - q * (size_t)np);
        float* a = rows + (size_t)p * D + q * W;
        float* s = state + (q * Np + i0 + (size_t)p) * W;
#pragma unroll
        for (int k = 0; k < W; k += 4) {
            if constexpr (PACK) st4(s + k, p < n ? ld4(a + k) : make_float4(0.f, 0.f, 0.f, 0.f));
            else if (p < n) st4(a + k, ld4(s + k));
        }
    }
}

dim3 tile_grid(int particles, int D) {
    return dim3((unsigned)((particles + kTileT - 1) / kTileT), (unsigned)std::min((D + kTileT - 1) / kTileT, 1024));
}

int panel_grid(int D, int W, int np) {
    return (int)std::max<long long>(1, std::min<long long>(((long long)(D / W) * np + 255) / 256, 1 << 14));
}

template <bool PACK>
void launch_panel(float* rows, float* state, int D, int Np, int W, int i0, int n, int np, cudaStream_t st) {
    const int g = panel_grid(D, W, np);
    if (W == 16) panel_rows_kernel<16, PACK><<<g, 256, 0, st>>>(rows, state, D, (size_t)Np, (size_t)i0, n, np);
    else panel_rows_kernel<8, PACK><<<g, 256, 0, st>>>(rows, state, D, (size_t)Np, (size_t)i0, n, np);
}

// gbest = lexicographic argmin over (pbest_fit, index): every block folds its
// minimum into the key by an atomicMin (all ones before the launch); the last
// one gathers gbest_pos and sets the iteration. One block alone took 0.7 us per
// 1000 particles. panel: the layout of pb (0: dimension-major).
__global__ void __launch_bounds__(kBlock) recompute_kernel(const __grid_constant__ SwarmDev s, uint32_t t, int panel,
                                                           int fill_pad) {
    __shared__ unsigned long long red[kBlock / 32];
    __shared__ int s_last;
    unsigned long long k = kKeyNone;
    bool nan = false;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < (uint32_t)s.Np; i += gridDim.x * blockDim.x) {
        if (i >= (uint32_t)s.N) {
            if (fill_pad) s.pf[i] = __int_as_float(0x7f800000);
            continue;
        }
        const float f = s.pf[i];
        const unsigned long long kk = pack_key(f, i);
        k = kk < k ? kk : k;
        nan |= (f != f);
    }
    k = block_min(k, red);
    if (__syncthreads_or(nan) && threadIdx.x == 0) atomicOr(s.status, kStatusNaN);
    if (threadIdx.x == 0) {
        atomicMin(s.gkey, k);
        __threadfence();
        s_last = atomicAdd(s.ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    k = __ldcg(s.gkey);
    const size_t g = (size_t)(k & 0xFFFFFFFFull), Np = (size_t)s.Np;
    float* G = s.G + (size_t)(t & 1u) * s.D;
    for (int d = threadIdx.x; d < s.D; d += blockDim.x)
        G[d] = panel ? s.pb[((size_t)(d / panel) * Np + g) * panel + d % panel] : s.pb[(size_t)d * Np + g];
    if (threadIdx.x == 0) {
        s.gkey[1] = k;
        *s.t_dev = t;
        *s.ticket = 0u;
    }
}

}  // namespace

template <typename T>
cudaError_t launch_pack_rows(const T* rows, T* dst, int D, int Np, int panel, int i0, int n, int np, cudaStream_t st) {
    if constexpr (sizeof(T) == 4) {
        if (panel) {
            launch_panel<true>(const_cast<T*>(rows), dst, D, Np, panel, i0, n, np, st);
            return cudaGetLastError();
        }
    }
    pack_rows_kernel<T><<<tile_grid(np, D), 256, 0, st>>>(rows, dst, D, (size_t)Np, (size_t)i0, n, np);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_unpack_rows(const T* src, T* rows, int D, int Np, int panel, int i0, int n, cudaStream_t st) {
    if constexpr (sizeof(T) == 4) {
        if (panel) {
            launch_panel<false>(rows, const_cast<T*>(src), D, Np, panel, i0, n, n, st);
            return cudaGetLastError();
        }
    }
    unpack_rows_kernel<T><<<tile_grid(n, D), 256, 0, st>>>(src, rows, D, (size_t)Np, (size_t)i0, n);
    return cudaGetLastError();
}

template cudaError_t launch_pack_rows<float>(const float*, float*, int, int, int, int, int, int, cudaStream_t);
template cudaError_t launch_pack_rows<double>(const double*, double*, int, int, int, int, int, int, cudaStream_t);
template cudaError_t launch_unpack_rows<float>(const float*, float*, int, int, int, int, int, cudaStream_t);
template cudaError_t launch_unpack_rows<double>(const double*, double*, int, int, int, int, int, cudaStream_t);

cudaError_t launch_recompute(const SwarmDev& s, uint32_t t, int panel, bool fill_pad, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(s.gkey, 0xFF, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    const int grid = std::max(1, std::min(304, s.Np / (4 * kBlock)));
    recompute_kernel<<<grid, kBlock, 0, st>>>(s, t, panel, fill_pad ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace cupso
