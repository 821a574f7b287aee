// kernels_batch_panel.cu -- many independent swarms in one launch per iteration, their
// state in panels of 8 dimensions.
//
// As in kernels_batch.cu a launch advances every swarm by one synchronous iteration
// over units handed to warps from a counter; as in kernels_panel.cu two lanes share
// a particle, lane j owning dimensions 8 q + 4 j .. + 3 of panel q, so that a warp's
// unit is 16 particles and a particle whose pbest row is pending writes it instead
// of reading it. D need not be a multiple of 8: the state holds whole panels, and the
// last panel's sum stops at D.
//
// Why beside the 128-particle units of kernels_batch.cu: those walk all dimension
// pairs of four particles per lane, so a unit lasts as long as its swarm has
// dimensions, and a batch of a few dozen swarms is over when its last 256-dimensional
// unit is -- 64 uneven swarms (N 64 .. 8192, D 8 .. 256) have 2100 such units for 2432
// resident warps. Units of 16 particles are an eighth of that: 258 us an iteration
// before and 150 now; 8 uneven swarms 53 and 31, 16 swarms of 8192 x 256 298 and 139, 512
// uneven ones, which fill the chip either way, 1077 and 1009. What bounds it at 512 is
// memory (20 bytes per particle and dimension: 0.82 ms at the copy's rate) with the issue
// slots half taken.
// Swarms of fewer than kBatchPanelMinD dimensions have too few panels for the ring's
// look-ahead and stay there, and so do those whose last panel's unused dimensions would be
// moved at a cost where memory bounds the batch (the rule stands in cupso_batch.cu). In batches of hundreds of swarms a ring of 6 stages (`deep`) is
// the faster one, 1046 and 1009 us at 512, and those of fewer than kBatchPanelDeepD dimensions
// stay there too; with 128 it is 276 and 282.
//
// Three CTAs of 256 threads an SM leave 80 registers a thread, and two of 128 were
// slower where the chip is full (1.29 against 1.13 ms). What a swarm's move needs
// (round keys, coefficients, bounds) is read from shared memory for every panel, where
// held it spilled (1.29 ms); gbest_pos comes through the ring too: loaded directly,
// every fourth panel waited for it (64 swarms of 8192 x 256 539 us, now 472).
#include <cuda_runtime.h>

#include <algorithm>

#include "cupso_device.cuh"
#include "cupso_internal.h"
#include "panel_common.cuh"
#include "stream_common.cuh"

namespace cupso {

namespace {

constexpr int kW = 8, kL = kW / 4;          // panel width, lanes per particle
constexpr uint32_t kPU = 32 / kL;           // particles per unit

struct PUnit {
    uint32_t sw, u;                         // swarm (0xFFFFFFFF: none), unit within it
};

// The unit at position k of the hand-out order.
__device__ __forceinline__ PUnit unit_at(const BatchDev& b, uint32_t k) {
    if (k >= b.nunits) return PUnit{0xFFFFFFFFu, 0u};
    const uint2 e = __ldg(b.units + k);
    return PUnit{e.x, e.y};
}

// Where a lane's values of a unit are: its four of panel 0 of pos, the next panel
// `step` on (in values of 16 bytes); the planes of vel and pbest_pos follow at one and
// two times (panels x step).
struct Feed {
    float4* x;
    uint32_t step;
    uint32_t g;         // gbest_pos of the swarm, panel 0 (values of 16 bytes into BatchDev::G)
    bool pending;       // the particle's pbest row is pending
};

__device__ __forceinline__ int panels_of(const BatchSwarm& w) { return (w.D + kW - 1) / kW; }

__device__ __forceinline__ Feed feed_of(const BatchSwarm& w, uint32_t u, int cur, int lane_id) {
    const uint32_t i = u * kPU + (uint32_t)(lane_id / kL);
    return Feed{reinterpret_cast<float4*>(w.x) + (size_t)i * (kW / 4) + lane_id % kL, (uint32_t)w.Np * (kW / 4),
                w.g16 + (uint32_t)(cur * (w.Gs / 4)), __ldcg(w.pflag + i) != 0};
}

// Copies panel q of `panels` into a stage of the rings (my: this lane's slots; gring: the
// warp's, of gbest_pos).
__device__ __forceinline__ void issue_panel(const BatchDev& b, const Feed& f, float4* my, float4* gring, int q,
                                            int panels, int stage, int lane_id) {
    float4* slot = my + (size_t)stage * 3 * kBlock;
    const float4* p = f.x + (size_t)q * f.step;
    const uint32_t plane = (uint32_t)panels * f.step;
    cp16(slot, reinterpret_cast<const float*>(p));
    cp16(slot + kBlock, reinterpret_cast<const float*>(p + plane));
    if (!f.pending) cp16(slot + 2 * kBlock, reinterpret_cast<const float*>(p + 2ull * plane));
    if (lane_id < kL) cp16(gring + stage * kL + lane_id, b.G + 4ull * (f.g + (uint32_t)(kL * q + lane_id)));
}

// The copies run STAGES - 1 panels ahead of the arithmetic, into the next unit.
struct PPipe {
    PUnit nxt;      // the unit that is being copied
    Feed feed;
    int iq;         // its panels copied
    int left;       // its panels still to copy; -1: there is no further unit
    int stage;      // ring stage of the panel being computed
};

// The first units go out CTA by CTA, so that every SM gets as many, and as long ones; the
// others come from the counter: nothing is drawn where every unit has its warp.
__device__ __forceinline__ void next_unit(const BatchDev& b, unsigned* work, PPipe& pp, bool first, int cur,
                                          int lane_id) {
    const uint32_t warps = gridDim.x * (kBlock / 32);
    uint32_t k = b.nunits;
    if (first) {
        k = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    } else if (b.nunits > warps) {
        if (lane_id == 0) k = warps + atomicAdd(work, 1u);
        k = __shfl_sync(0xFFFFFFFFu, k, 0);
    }
    pp.nxt = unit_at(b, k);
    pp.iq = 0;
    pp.left = -1;
    if (pp.nxt.sw != 0xFFFFFFFFu) {
        const BatchSwarm& w = b.swarms[pp.nxt.sw];
        pp.feed = feed_of(w, pp.nxt.u, cur, lane_id);
        pp.left = panels_of(w);
    }
}

__device__ __forceinline__ void issue_next(const BatchDev& b, PPipe& pp, float4* my, float4* gring, int stage,
                                           int lane_id) {
    if (pp.left > 0) {
        issue_panel(b, pp.feed, my, gring, pp.iq, pp.iq + pp.left, stage, lane_id);
        ++pp.iq;
        --pp.left;
    }
    cp_commit();   // an empty group when there is nothing left to copy
}

// One vector of the swarm's constants from the warp's shared memory. Read again for
// every panel: held in registers, the round keys alone would take 20 of the 80 that
// three CTAs an SM leave each thread.
__device__ __forceinline__ uint4 constants(uint32_t cst, int k) {
    uint4 r;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(cst + 16u * (uint32_t)k) : "memory");
    return r;
}

__device__ __forceinline__ void philox_round(uint4& c, uint32_t k0, uint32_t k1) {
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
    const uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
    const uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
}

struct MoveB { float w, c1, c2, vmax, lo, hi; };

template <bool FAST>
__device__ __forceinline__ void move_b(float& x, float& v, float pb, float g, uint32_t w1, uint32_t w2,
                                       const MoveB& m) {
    const float cognitive = __fsub_rn(pb, x);
    const float social = __fsub_rn(g, x);
    float vel = __fmul_rn(m.w, v);
    if constexpr (FAST) {
        vel = __fmaf_rn(__fmaf_rn(m.c1, hi24(w1), m.c1), cognitive, vel);
        vel = __fmaf_rn(__fmaf_rn(m.c2, hi24(w2), m.c2), social, vel);
        v = clampf_minmax(vel, -m.vmax, m.vmax);
        x = clampf_minmax(__fadd_rn(x, v), m.lo, m.hi);
    } else {
        vel = __fmaf_rn(__fmul_rn(m.c1, u01(w1)), cognitive, vel);
        vel = __fmaf_rn(__fmul_rn(m.c2, u01(w2)), social, vel);
        v = clampf(vel, -m.vmax, m.vmax);
        x = clampf(__fadd_rn(x, v), m.lo, m.hi);
    }
}

// Publishes a unit's candidate (below K) and counts the unit. The warp that completes
// the swarm sets gbest_pos of parity nxt: from the winner's pos, which is its
// pbest_pos, as it improved in this iteration, or from the other parity's where no key below K
// came. The winner's row is visible then: both lanes that own it have stored it before
// the __syncwarp, and lane 0 fences after that and before it counts the unit, as it does for
// every unit with a candidate; the completing warp's lane 0 fences after its count.
__device__ __forceinline__ void close_unit(const BatchSwarm& w, unsigned long long best, bool any_nan,
                                           unsigned long long K, int cur, int nxt, int lane_id) {
    __syncwarp();
    int last = 0;
    if (lane_id == 0) {
        if (best != kKeyNone) {
            atomicMin(w.gkey + nxt, best);
            __threadfence();
        }
        if (any_nan) atomicOr(w.status, kStatusNaN);
        last = atomicAdd(w.done, 1u) == w.nunits - 1u;
        if (last) __threadfence();
    }
    last = __shfl_sync(0xFFFFFFFFu, last, 0);
    if (last) {
        const unsigned long long knew = __ldcg(w.gkey + nxt);
        const size_t gi = (size_t)(knew & 0xFFFFFFFFull), Np = (size_t)w.Np;
        float* to = w.G + (size_t)nxt * w.Gs;
        const float* from = w.G + (size_t)cur * w.Gs;
        for (int d = lane_id; d < w.D; d += 32)
            to[d] = knew < K ? __ldcg(w.x + ((size_t)(d / kW) * Np + gi) * kW + d % kW) : __ldcg(from + d);
        __syncwarp();
        if (lane_id == 0) {
            w.gkey[cur] = knew;
            *w.done = 0u;
        }
    }
}

// One unit at iteration t: its first STAGES - 1 panels are in the ring (feed: its
// flags); keeps that many in flight, of the next unit once its own are issued.
template <int FIT, bool FAST, int STAGES>
__device__ __forceinline__ void run_unit(const BatchDev& b, unsigned* work, float4* my, float4* gring, uint32_t cst, PUnit cu,
                                         const Feed me, PPipe& pp, uint32_t t, int lane_id) {
    const BatchSwarm& w = b.swarms[cu.sw];
    __syncwarp();
    if (lane_id < 8)
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(cst + 16u * (uint32_t)lane_id),
                     "r"(w.cst[lane_id].x), "r"(w.cst[lane_id].y), "r"(w.cst[lane_id].z), "r"(w.cst[lane_id].w) : "memory");
    __syncwarp();
    const int D = w.D, Dq = panels_of(w), j = lane_id % kL;
    const uint32_t plane = (uint32_t)Dq * me.step;
    const int cur = (int)((t - 1u) & 1u), nxt = cur ^ 1;
    const uint32_t i = cu.u * kPU + (uint32_t)(lane_id / kL);
    const unsigned long long K = __ldcg(w.gkey + cur);
    const float pf = j == kL - 1 ? __ldcg(w.pf + i) : 0.0f;
    FitAcc<FIT> acc;
    float carry = 0.0f;
    for (int q = 0; q < Dq; ++q) {
        {
            __syncwarp();   // every lane has read the stage that is copied into
            int ws = pp.stage + STAGES - 1;
            if (ws >= STAGES) ws -= STAGES;
            // every unit has at least STAGES - 1 panels, so the look-ahead ends within the next one
            if (pp.left == 0) next_unit(b, work, pp, false, cur, lane_id);
            issue_next(b, pp, my, gring, ws, lane_id);
        }
        const int d0 = kW * q + 4 * j;
        cp_wait<STAGES - 1>();
        __syncwarp();   // lanes 0 and 1 copied gbest_pos
        const float4 g4 = gring[pp.stage * kL + j];
        const float4* slot = my + (size_t)pp.stage * 3 * kBlock;
        float4 X = slot[0], V = slot[kBlock];
        float4 Pb;
        float4* const to = me.x + (size_t)q * me.step;
        if (me.pending) {
            Pb = X;
            st4(reinterpret_cast<float*>(to + 2ull * plane), X);
        } else {
            Pb = slot[2 * kBlock];
        }
        const uint4 c1 = constants(cst, 6);
        uint4 r[2];
#pragma unroll
        for (int g = 0; g < 2; ++g) r[g] = make_uint4((uint32_t)((d0 >> 1) + g), i, t, c1.z);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const uint4 rk = constants(cst, k);
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                philox_round(r[g], rk.x, rk.y);
                philox_round(r[g], rk.z, rk.w);
            }
        }
        const uint4 c0 = constants(cst, 5);
        const MoveB m{__uint_as_float(c0.x), __uint_as_float(c0.y), __uint_as_float(c0.z), __uint_as_float(c0.w),
                      __uint_as_float(c1.x), __uint_as_float(c1.y)};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float xj = lane(X, k), vj = lane(V, k);
            move_b<FAST>(xj, vj, lane(Pb, k), lane(g4, k), word(r[k / 2], 2 * (k % 2)), word(r[k / 2], 2 * (k % 2) + 1),
                         m);
            set_lane(X, k, xj);
            set_lane(V, k, vj);
        }
        st4(reinterpret_cast<float*>(to), X);
        st4(reinterpret_cast<float*>(to + plane), V);
        if (q + 1 < Dq) panel_sum<FIT, kL, false, FAST>(acc, X, d0, D, j, lane_id, carry);
        else panel_sum<FIT, kL, true, FAST>(acc, X, d0, D, j, lane_id, carry);
        if (++pp.stage == STAGES) pp.stage = 0;
    }
    // Steps 4-5 in the particle's last lane, which holds the whole sum
    unsigned long long best = kKeyNone;
    bool nan = false;
    if (j == kL - 1) {
        const float f = acc.finish(D);
        const bool real = i < (uint32_t)w.N;
        nan = real && (f != f);
        uint32_t fl_new = 0u;
        if (real && f < pf) {
            fl_new = 1u;
            w.pf[i] = f;
            const unsigned long long k = pack_key(f, i);
            if (k < K) best = k;
        }
        if (fl_new != (uint32_t)me.pending) w.pflag[i] = (unsigned char)fl_new;
    }
    best = warp_min_u64(best);
    close_unit(w, best, __any_sync(0xFFFFFFFFu, nan), K, cur, nxt, lane_id);
}

// Step 1 of one unit: the single-swarm init kernel's arithmetic, every key competing.
template <int FIT>
__device__ __forceinline__ void init_unit(const BatchSwarm& wg, uint32_t u, int lane_id) {
    const BatchSwarm w = wg;
    const int D = w.D, Dq = (D + kW - 1) / kW, j = lane_id % kL;
    const float span = __fsub_rn(w.hi, w.lo), vspan = __fmul_rn(2.0f, w.vmax);
    const uint32_t i = u * kPU + (uint32_t)(lane_id / kL);
    FitAcc<FIT> acc;
    float carry = 0.0f;
    for (int q = 0; q < Dq; ++q) {
        const int d0 = kW * q + 4 * j;
        const size_t off = ((size_t)q * (size_t)w.Np + i) * kW + 4 * j;
        float4 X, V;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const uint4 r = philox4x32_10(make_uint4((uint32_t)((d0 >> 1) + g), i, 0u, w.swarm), w.key0, w.key1);
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                set_lane(X, 2 * g + hh, clampf(__fmaf_rn(u01(word(r, 2 * hh)), span, w.lo), w.lo, w.hi));
                set_lane(V, 2 * g + hh, clampf(__fmaf_rn(u01(word(r, 2 * hh + 1)), vspan, -w.vmax), -w.vmax, w.vmax));
            }
        }
        st4(w.x + off, X);
        st4(w.v + off, V);
        st4(w.pb + off, X);
        if (q + 1 < Dq) panel_sum<FIT, kL, false>(acc, X, d0, D, j, lane_id, carry);
        else panel_sum<FIT, kL, true>(acc, X, d0, D, j, lane_id, carry);
    }
    unsigned long long best = kKeyNone;
    bool nan = false;
    if (j == kL - 1) {
        const float f = acc.finish(D);
        w.pf[i] = f;
        if (i < (uint32_t)w.N) {
            best = pack_key(f, i);
            nan = f != f;
        }
    }
    best = warp_min_u64(best);
    // every particle competes; t = 0 lives in slot 0, and slot 1 gets the same key
    close_unit(w, best, __any_sync(0xFFFFFFFFu, nan), kKeyNone, 1, 0, lane_id);
}

}  // namespace

// Requires at least STAGES - 1 panels of every swarm of the batch and states of whole panels.
template <int STAGES>
__global__ void __launch_bounds__(kBlock, 3) batch_panel_kernel(const __grid_constant__ BatchDev b) {
    extern __shared__ float4 ring_p[];
    const uint32_t t = __ldcg(b.t_dev) + 1u;
    unsigned* work = b.work + (t & 1u);
    const int lane_id = threadIdx.x & 31;
    float4* my = ring_p + threadIdx.x;
    __shared__ uint4 s_cst[kBlock / 32][8];
    __shared__ float4 s_g[kBlock / 32][STAGES * kL];
    float4* gring = s_g[threadIdx.x >> 5];
    const uint32_t cst = (uint32_t)__cvta_generic_to_shared(s_cst[threadIdx.x >> 5]);

    PPipe pp;
    pp.stage = 0;
    pp.feed = Feed{};
    next_unit(b, work, pp, true, (int)((t - 1u) & 1u), lane_id);
#pragma unroll
    for (int k = 0; k < STAGES - 1; ++k) issue_next(b, pp, my, gring, k, lane_id);
    PUnit cu = pp.nxt;
    Feed me = pp.feed;
    while (cu.sw != 0xFFFFFFFFu) {
        const bool fast = b.swarms[cu.sw].fast != 0;
        switch (b.swarms[cu.sw].fid * 2 + (fast ? 1 : 0)) {
            case kSphere * 2 + 1: run_unit<kSphere, true, STAGES>(b, work, my, gring, cst, cu, me, pp, t, lane_id); break;
            case kSphere * 2: run_unit<kSphere, false, STAGES>(b, work, my, gring, cst, cu, me, pp, t, lane_id); break;
            case kRastrigin * 2 + 1: run_unit<kRastrigin, true, STAGES>(b, work, my, gring, cst, cu, me, pp, t, lane_id); break;
            case kRastrigin * 2: run_unit<kRastrigin, false, STAGES>(b, work, my, gring, cst, cu, me, pp, t, lane_id); break;
            case kAckley * 2 + 1: run_unit<kAckley, true, STAGES>(b, work, my, gring, cst, cu, me, pp, t, lane_id); break;
            case kAckley * 2: run_unit<kAckley, false, STAGES>(b, work, my, gring, cst, cu, me, pp, t, lane_id); break;
            case kRosenbrock * 2 + 1: run_unit<kRosenbrock, true, STAGES>(b, work, my, gring, cst, cu, me, pp, t, lane_id); break;
            case kRosenbrock * 2: run_unit<kRosenbrock, false, STAGES>(b, work, my, gring, cst, cu, me, pp, t, lane_id); break;
            case kCubicMax * 2 + 1: run_unit<kCubicMax, true, STAGES>(b, work, my, gring, cst, cu, me, pp, t, lane_id); break;
            default: run_unit<kCubicMax, false, STAGES>(b, work, my, gring, cst, cu, me, pp, t, lane_id); break;   // nothing else is admitted
        }
        cu = pp.nxt;        // every unit ends with the next one fetched
        me = pp.feed;
    }
    cp_wait<0>();
    // The last CTA rolls the batch forward: the next launch counts on the other counter.
    // Nothing of this launch reads what it sets once its CTA has arrived.
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) s_last = (atomicAdd(b.ticket, 1u) == gridDim.x - 1);
    __syncthreads();
    if (s_last && threadIdx.x == 0) {
        b.work[(t + 1u) & 1u] = 0u;
        *b.ticket = 0u;
        *b.t_dev = t;
    }
}

__global__ void __launch_bounds__(kBlock) batch_panel_init_kernel(const __grid_constant__ BatchDev b) {
    const int lane_id = threadIdx.x & 31;
    const unsigned nwarps = (gridDim.x * blockDim.x) >> 5;
    for (unsigned k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < b.nunits; k += nwarps) {
        const uint2 e = __ldg(b.units + k);
        const BatchSwarm& w = b.swarms[e.x];
        switch (w.fid) {
            case kSphere: init_unit<kSphere>(w, e.y, lane_id); break;
            case kRastrigin: init_unit<kRastrigin>(w, e.y, lane_id); break;
            case kAckley: init_unit<kAckley>(w, e.y, lane_id); break;
            case kRosenbrock: init_unit<kRosenbrock>(w, e.y, lane_id); break;
            default: init_unit<kCubicMax>(w, e.y, lane_id); break;   // nothing else is admitted
        }
    }
}

namespace {
static_assert(kBatchPanelMinD > kW * 3 && kBatchPanelDeepD > kW * 4, "rings of 5 and 6 stages: 4 and 5 panels");
constexpr size_t ring_bytes(int stages) { return sizeof(float4) * (size_t)stages * 3 * kBlock; }
}  // namespace

cudaError_t prepare_batch_panel() {
    cudaError_t e = cudaFuncSetAttribute(batch_panel_kernel<5>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)ring_bytes(5));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(batch_panel_kernel<6>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ring_bytes(6));
    return e;
}

int batch_panel_grid(unsigned int nunits, bool deep, int num_sms) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, deep ? batch_panel_kernel<6> : batch_panel_kernel<5>, kBlock,
                                                      ring_bytes(deep ? 6 : 5)) != cudaSuccess) {
        cudaGetLastError();
        n = 1;
    }
    const long long warps = (long long)num_sms * (kBlock / 32);
    const long long want = ((long long)nunits + warps - 1) / warps;   // CTAs per SM for a warp per unit
    return (int)std::min<long long>(num_sms * std::min<long long>(std::max(n, 1), want), nunits);
}

cudaError_t launch_batch_panel(const BatchDev& b, bool deep, int grid, cudaStream_t st) {
    if (deep) batch_panel_kernel<6><<<grid, kBlock, ring_bytes(6), st>>>(b);
    else batch_panel_kernel<5><<<grid, kBlock, ring_bytes(5), st>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_batch_panel_init(const BatchDev& b, int num_sms, cudaStream_t st) {
    const long long useful = ((long long)b.nunits + kBlock / 32 - 1) / (kBlock / 32);
    batch_panel_init_kernel<<<(int)std::min<long long>(useful, 8ll * num_sms), kBlock, 0, st>>>(b);
    return cudaGetLastError();
}

}  // namespace cupso
