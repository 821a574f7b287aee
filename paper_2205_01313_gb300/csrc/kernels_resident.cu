// kernels_resident.cu -- synchronous PSO with the whole swarm in the registers of
// all SMs: several iterations of one cupso_step call in one cooperative launch.
//
// A swarm of up to about a million particle-dimensions (65536 registers x 152
// SMs) needs no memory traffic per iteration. Each CTA owns P consecutive
// particles and has P x rows threads; thread (row, p) owns up to ITEMS dimension
// pairs (row, row + rows, ...) of particle p and keeps their pos, v and pbest_pos in
// registers for the whole launch. Per iteration
//   1. all warps: the end of Eq. 1 (the social term) and Eq. 2 on the items; pos
//      and the fitness terms to shared memory, one row per particle;
//   2. the first warps, one thread per particle: the terms added in the oracle's
//      order over d, pbest_fit (a register) compared, improvements flagged; then
//      the CTA's candidate (lowest improved key below gbest's), if any -- position
//      to its slot in global memory, key by an atomicMin -- and one arrival on
//      the grid barrier;
//   3. beside that and while the barrier completes: everything of the next
//      iteration that needs no gbest -- the Philox words, c1 r1 and c2 r2, then
//      (improved items having copied pos to pbest_pos) the inertia and cognitive
//      terms of Eq. 1. The other warps start on the words at once, the summing
//      warps after their arrival; the last warp, done first, polls the barrier;
//   4. if any CTA had a candidate, the agreed key and, if it is new, the winner's
//      position from its slot.
// What bounds an iteration is the chain 1-2-4: the ordered sum, one global round
// trip to arrive and see the last arrival, and two more only when gbest may have
// changed: the barrier word carries, beside its arrivals, how many candidates
// each parity has had, so an iteration without any ends with the poll. Keys,
// slots and counts are kept by parity: a CTA can be at most one iteration ahead of
// another, since every barrier needs all arrivals. A parity's key is never reset,
// it only falls: the new gbest is the lower of it and the one held.
// Philox is bound by its 20 wide multiplies (76 issue cycles per warp and call
// measured, 4 per multiply), more than all the rest: hence its place off the chain.
// Measured per iteration on one GB300 (calls of 1000; before: one launch of the
// tiled kernel, or one pass of the panel kernel, per iteration): 1024 x 32 sphere
// 5.0 -> 1.1 us, 20011 x 30 Ackley 8.7 -> 2.5, 20000 x 48 Rastrigin 10.4 -> 3.1,
// 8192 x 128 Rastrigin 10.2 -> 3.3, 60000 x 16 Rosenbrock 10.4 -> 3.9. Tried: warps of
// their own for sums and polling (20011 x 30 sphere 2.3 against 1.9 us: the
// workers' throughput counts more); the summing warps' first thread polling (2.2);
// an exchange without fences, every 64-bit word of a record tagged with its
// iteration and the candidates' CTAs named in the barrier words, so that a new
// gbest takes one round trip instead of two (1024 x 32 Rosenbrock 2.2 either way,
// and the iterations without a candidate 0.1 us longer).
//
// Same bits as the other SYNC kernels: the same operations per item, the same
// order of the sum, the lexicographic minimum of the same keys.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "cupso_device.cuh"
#include "cupso_internal.h"
#include "fit_terms.cuh"
#include "resident.h"
#include "stream_common.cuh"

namespace cupso {

namespace {

// Threads per CTA at most for ITEMS pairs per thread: what the register file
// holds at 10 registers per pair and about 45 others (whole warps per quarter SM).
constexpr int max_threads(int items) {
    return items <= 1 ? 1024 : (items <= 3 ? 768 : (items <= 4 ? 640 : (items <= 8 ? 512 : (items <= 12 ? 384 : 256))));
}
constexpr int kResItems[] = {1, 2, 3, 4, 5, 6, 8, 12, 16};   // instantiated
constexpr size_t kResSmem = 200u * 1024u;   // dynamic shared memory of a CTA at most

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// The part of Eq. 1 that needs no gbest, of two dimensions in move_one_fast's order: v
// becomes w v + c1 r1 (pbest - x); cr1 = c1 r1. Two IEEE operations per instruction
// (fma.rn.f32x2) here and in the cosines: Ackley 20000 x 48 3.55 us an iteration with
// single ones, now 3.37; sphere 3.11 and 2.98.
__device__ __forceinline__ void move_begin(const float (&x)[2], float (&v)[2], const float (&pb)[2],
                                           const float (&cr1)[2], const SwarmDev& s) {
    const f32x2 wv = mul2(both(s.w), pack2(v[0], v[1]));
    unpack2(fma2(pack2(cr1[0], cr1[1]), sub2(pack2(pb[0], pb[1]), pack2(x[0], x[1])), wv), v[0], v[1]);
}

// The rest: the social term, Eq. 2 and the clamps.
__device__ __forceinline__ void move_end(float (&x)[2], float (&v)[2], float2 g, const float (&cr2)[2],
                                         const SwarmDev& s) {
    const f32x2 xx = pack2(x[0], x[1]);
    unpack2(fma2(pack2(cr2[0], cr2[1]), sub2(pack2(g.x, g.y), xx), pack2(v[0], v[1])), v[0], v[1]);
    v[0] = clampf_minmax(v[0], -s.vmax, s.vmax);
    v[1] = clampf_minmax(v[1], -s.vmax, s.vmax);
    unpack2(add2(xx, pack2(v[0], v[1])), x[0], x[1]);
    x[0] = clampf_minmax(x[0], s.lo, s.hi);
    x[1] = clampf_minmax(x[1], s.lo, s.hi);
}

__device__ __forceinline__ size_t state_off(const SwarmDev& s, int panel, int d, uint32_t i) {
    return panel ? ((size_t)(d / panel) * (size_t)s.Np + i) * (size_t)panel + (size_t)(d % panel)
                 : (size_t)d * (size_t)s.Np + i;
}

// Four dimensions (d0 .. d0 + 3, of which the first `n` count) of the ordered
// fitness sum: x the positions, h the terms formed with them. Rosenbrock's terms
// pair neighbouring dimensions, which different threads own: they are formed here,
// off the chain of the sum, instead of after one more barrier.
template <int FIT>
__device__ __forceinline__ void fold4(FitAcc<FIT>& a, int d0, int n, const float4& x, const float4& h) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (e >= n) break;
        if constexpr (FIT == kSphere) {
            a.acc = __fmaf_rn(lane(x, e), lane(x, e), a.acc);
        } else if constexpr (FIT == kAckley) {
            a.acc = __fmaf_rn(lane(x, e), lane(x, e), a.acc);
            a.acc2 = __fadd_rn(a.acc2, lane(h, e));
        } else if constexpr (FIT == kRosenbrock) {
            a.add_c(d0 + e, lane(x, e), 0.0f);
        } else {
            a.acc = __fadd_rn(a.acc, lane(h, e));
        }
    }
}

// A particle's fitness from its rows of X and H (16-byte aligned).
template <int FIT>
__device__ __forceinline__ float row_fitness(const float* X, const float* H, int D) {
    constexpr bool kX = FIT == kSphere || FIT == kAckley || FIT == kRosenbrock;
    constexpr bool kH = FIT == kRastrigin || FIT == kAckley || FIT == kCubicMax;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    FitAcc<FIT> a;
    const int d4 = D & ~3;
#pragma unroll 4
    for (int d = 0; d < d4; d += 4)
        fold4<FIT>(a, d, 4, kX ? ld4(X + d) : zero, kH ? ld4(H + d) : zero);
    if (d4 < D) fold4<FIT>(a, d4, D - d4, kX ? ld4(X + d4) : zero, kH ? ld4(H + d4) : zero);
    return a.finish(D);
}

}  // namespace

// P particles per CTA, blockDim.x >= P * rows in whole warps, ITEMS * rows >=
// ceil(D / 2) pairs; S: floats per particle's row of X and H (a multiple of 4 whose
// quarter is odd, so that the summing threads' 16-byte reads spread over the
// banks; >= 2 ITEMS rows). State in `panel` layout (0: dimension-major), pending
// pbest rows (s.pflag) taken over and cleared. Requires s.fast_cr and s.fast_clamp (and, for a fitness with cos, bounds
// within kSmallX), a cooperative launch, *rb.bar, the word behind it and rb.key zero at launch: the CTA
// that leaves last clears them, so that a launch needs nothing before it (two memsets before
// each took 1.3 of the 3.5 us of host time of a call).
// rb.key holds complements, so that zero is "none".
// `expect`: arrivals that complete a barrier (gridDim.x; one more only to test that
// its bound works).
// *rb.bar: arrivals in bits 0..31, the candidates of even and odd iterations in
// bits 32..47 and 48..63 (each modulo 2^16; at most one per CTA in an iteration, so
// a change shows; the even count's carry moves the odd one by one now and then,
// which only costs a look at the key).
// Named barriers: 1 the summing warps; 2 the flags (summing warps arrive, the others
// wait). Barrier 0, all, separates the move from the sums and ends an iteration.
template <int FIT, int ITEMS>
__global__ void __launch_bounds__(max_threads(ITEMS), 1) resident_kernel(const __grid_constant__ SwarmDev s,
                                                                        const __grid_constant__ ResidentBufs rb, int P,
                                                                        int rows, int S, int panel, int iters,
                                                                        unsigned int expect) {
    constexpr bool kH = FIT == kRastrigin || FIT == kAckley || FIT == kCubicMax;   // terms formed with the move
    extern __shared__ __align__(16) float sm_res[];
    const int D = s.D, pairs = (D + 1) >> 1, T = (int)blockDim.x, tid = (int)threadIdx.x;
    float* X = sm_res;                                               // [P][S]
    float* H = X + (size_t)P * S;                                    // [P][S] if kH
    float2* Gs = reinterpret_cast<float2*>(H + (kH ? (size_t)P * S : 0));   // [ITEMS * rows] gbest_pos, then zeros
    unsigned char* imp = reinterpret_cast<unsigned char*>(Gs + ITEMS * rows);   // [P]
    __shared__ unsigned long long s_cand, s_key;
    __shared__ int s_ok;

    const uint32_t base = blockIdx.x * (uint32_t)P;
    const int n = min(P, s.N - (int)base);               // particles of this CTA (> 0)
    const int row = tid / P, p = tid - row * P;
    const uint32_t i = base + (uint32_t)p;
    // Threads past the last row do nothing; pairs past D and particles past N are
    // computed on zeros (their rows of X and H exist and are never summed).
    const bool active = row < rows;
    const int sum_threads = (P + 31) / 32 * 32;          // the summing warps
    const bool sums = tid < sum_threads;                 // uniform over a warp
    const int poller = T - 32;                           // the first thread of the last warp
    const uint32_t t_prev = __ldcg(s.t_dev);
    const int cur0 = (int)(t_prev & 1u);

    float x[ITEMS][2], v[ITEMS][2], pb[ITEMS][2], cr1[ITEMS][2], cr2[ITEMS][2];
    auto words = [&](uint32_t t) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint4 r = philox4x32_10_rk(make_uint4((uint32_t)(row + j * rows), i, t, s.swarm), s.rk0, s.rk1);
            unpack2(fma2(both(s.c1s), pack2(hi24(r.x), hi24(r.z)), both(s.c1s)), cr1[j][0], cr1[j][1]);
            unpack2(fma2(both(s.c2s), pack2(hi24(r.y), hi24(r.w)), both(s.c2s)), cr2[j][0], cr2[j][1]);
        }
    };
    auto begin = [&](bool up) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            if (up) {
                pb[j][0] = x[j][0];
                pb[j][1] = x[j][1];
            }
            move_begin(x[j], v[j], pb[j], cr1[j], s);
        }
    };
    const bool own = active && p < n;
    const bool lazy = own && s.pflag[i] != 0;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int g = row + j * rows;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            x[j][h] = v[j][h] = pb[j][h] = 0.0f;
            if (own && 2 * g + h < D) {
                const size_t off = state_off(s, panel, 2 * g + h, i);
                x[j][h] = s.x[off];
                v[j][h] = s.v[off];
                pb[j][h] = lazy ? x[j][h] : s.pb[off];
            }
        }
    }
    if (active) {
        words(t_prev + 1u);
        begin(false);
    }
    float pf = tid < n ? s.pf[base + tid] : 0.0f;
    if (tid < P) imp[tid] = 0;
    for (int d = tid; d < 2 * ITEMS * rows; d += T)
        reinterpret_cast<float*>(Gs)[d] = d < D ? s.G[(size_t)cur0 * D + d] : 0.0f;
    unsigned long long K = __ldcg(s.gkey + cur0);        // gbest's key, the same in every thread
    if (tid == 0) s_cand = kKeyNone;
    uint32_t seen = 0u;                                  // the poller: candidate counts by parity (16 bits each)
    float* const xo = X + (size_t)p * S + 2 * row;
    float* const ho = H + (size_t)p * S + 2 * row;
    __syncthreads();

    bool nan = false;
    int done = 0;
    for (int k = 0; k < iters; ++k) {
        const int par = k & 1;
        if (active) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                const float2 g = Gs[row + j * rows];
                move_end(x[j], v[j], g, cr2[j], s);
                *reinterpret_cast<float2*>(xo + 2 * j * rows) = make_float2(x[j][0], x[j][1]);
                if constexpr (kH)
                    *reinterpret_cast<float2*>(ho + 2 * j * rows) = FitTerms<FIT>::two(x[j][0], x[j][1]);
            }
        }
        __syncthreads();
        if (sums) {
            if (tid < n) {
                const float f = row_fitness<FIT>(X + (size_t)tid * S, H + (size_t)tid * S, D);
                nan |= (f != f);
                const bool better = f < pf;
                imp[tid] = better ? 1 : 0;
                if (better) {
                    pf = f;
                    const unsigned long long key = pack_key(f, base + (uint32_t)tid);
                    if (key < K) atomicMin(&s_cand, key);
                }
            }
            bar_sync(1, sum_threads);
            const unsigned long long cand = s_cand;
            if (cand != kKeyNone) {   // uniform over the summing warps
                const int pc = (int)((uint32_t)(cand & 0xFFFFFFFFull) - base);
                float* slot = rb.slots + ((size_t)par * gridDim.x + blockIdx.x) * (size_t)D;
                for (int d = tid; d < D; d += sum_threads) __stcg(slot + d, X[(size_t)pc * S + d]);
                bar_sync(1, sum_threads);
            }
            if (tid == 0) {
                // With a candidate the arrival releases its slot and key (written before the barrier
                // above). Without one the CTA has written nothing that others read, and a release
                // would wait about 0.3 us. That its reads of the last slots come before another
                // CTA's next writes of them, two iterations on, does not follow from a relaxed
                // arrival in the memory model; it holds because the loads have returned (their
                // values are in Gs) before the barriers of this iteration.
                if (cand != kKeyNone) {
                    atomicMax(rb.key + par, ~cand);
                    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(rb.bar),
                                 "l"(1ull + (1ull << (32 + 16 * par)))
                                 : "memory");
                } else {
                    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(rb.bar), "l"(1ull) : "memory");
                }
            }
            if (T > sum_threads) bar_arrive(2, T);   // the flags are written
        }
        const bool more = k + 1 < iters && active;
        if (more) words(t_prev + 2u + (uint32_t)k);
        if (!sums) bar_sync(2, T);
        if (more) begin(imp[p] != 0);
        if (tid == poller) {
            const unsigned int target = (unsigned int)(k + 1) * expect;
            int ok = 1;
            unsigned long long w = ld_relaxed_u64(rb.bar);
            if ((unsigned int)w < target) {
                const long long deadline = global_ns() + s.wait_limit_ns;
                while ((unsigned int)(w = ld_relaxed_u64(rb.bar)) < target) {
                    if (global_ns() > deadline) {
                        ok = 0;
                        atomicOr(s.status, kStatusTimeout);
                        break;
                    }
                }
            }
            // this parity's candidates: final for this iteration (the others are at most one ahead)
            const uint32_t mask = 0xFFFFu << (16 * par), now = (uint32_t)(w >> 32) & mask;
            unsigned long long key = kKeyNone;
            if (now != (seen & mask)) {   // acquire what the candidates' arrivals released
                asm volatile("fence.acq_rel.gpu;" ::: "memory");
                key = ~__ldcg(rb.key + par);
            }
            s_key = key;
            seen = (seen & ~mask) | now;
            s_ok = ok;
        }
        __syncthreads();
        if (!s_ok) break;
        if (tid == 0) s_cand = kKeyNone;   // read before this barrier, next written after the next one
        const unsigned long long best = s_key;
        if (best < K) {   // uniform
            const uint32_t c = (uint32_t)(best & 0xFFFFFFFFull) / (uint32_t)P;
            const float* slot = rb.slots + ((size_t)par * gridDim.x + c) * (size_t)D;
            for (int d = tid; d < D; d += T) reinterpret_cast<float*>(Gs)[d] = __ldcg(slot + d);
            K = best;
            __syncthreads();
        }
        done = k + 1;
    }

    // the state back to memory, pending pbest rows included
    const bool up = own && imp[p] != 0;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int g = row + j * rows;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (own && 2 * g + h < D) {
                const size_t off = state_off(s, panel, 2 * g + h, i);
                s.x[off] = x[j][h];
                s.v[off] = v[j][h];
                s.pb[off] = up ? x[j][h] : pb[j][h];
            }
        }
    }
    if (tid < n) {
        s.pf[base + tid] = pf;
        s.pflag[base + tid] = 0;
    }
    if (__syncthreads_or(nan) && tid == 0) atomicOr(s.status, kStatusNaN);
    if (tid == 0) {   // every thread of the CTA is done with the exchange
        unsigned int* gone = reinterpret_cast<unsigned int*>(rb.bar + 1);
        __threadfence();   // this CTA's arrivals and candidates before its leaving
        if (atomicAdd(gone, 1u) == gridDim.x - 1) {
            __threadfence();
            rb.key[0] = rb.key[1] = 0ull;
            *rb.bar = 0ull;
            *gone = 0u;
        }
    }
    if (blockIdx.x == 0) {
        const uint32_t t_end = t_prev + (uint32_t)done;
        const int out = (int)(t_end & 1u);
        for (int d = tid; d < D; d += T) s.G[(size_t)out * D + d] = reinterpret_cast<float*>(Gs)[d];
        if (tid == 0) {
            s.gkey[0] = K;
            s.gkey[1] = K;
            *s.t_dev = t_end;
        }
    }
}

namespace {

struct ResPlan {
    int P = 0, grid = 0, rows = 0, threads = 0, items = 0, S = 0;
    size_t smem = 0;
};

// P = N over the SMs, and of small swarms up to 128 (pair, particle) items, over at least 8 CTAs: more
// CTAs are no faster for one swarm (an iteration of 300 x 8 1.08 us in 150 CTAs, 0.78 in 10; 1000 x 2 1.03
// and 1.04), and cooperative launches of 150 CTAs hold up one another, so that swarms stepped on
// streams of their own no longer ran side by side (32 of 1000 x 2: 0.33 us per swarm and
// iteration, 0.10 on clusters, now 0.05; of 1024 x 16 0.16, 0.13 and 0.12). Then the fewest pairs
// per thread whose threads fit, and no more rows of threads than those pairs need.
bool res_plan(int N, int D, int num_sms, ResPlan* r) {
    const int pairs = (D + 1) / 2;
    const int small = std::min((N + 7) / 8, 128 / pairs);
    const int P = std::max((N + num_sms - 1) / num_sms, small);
    for (int items : kResItems) {
        const int rows = (pairs + items - 1) / items;
        const long long threads = ((long long)P * rows + 31) / 32 * 32;
        if (threads > max_threads(items)) continue;
        r->P = P;
        r->grid = (N + P - 1) / P;
        r->items = items;
        r->rows = rows;
        r->threads = (int)threads;
        const int q = (2 * items * rows + 3) / 4;   // quarter of the row stride, made odd
        r->S = 4 * (q | 1);
        r->smem = sizeof(float) * (2 * (size_t)P * r->S + 2 * (size_t)items * rows) + (size_t)P;
        return r->smem <= kResSmem;
    }
    return false;
}

template <int ITEMS>
const void* res_kernel_i(int fid) {
    switch (fid) {
        case kSphere: return (const void*)resident_kernel<kSphere, ITEMS>;
        case kRastrigin: return (const void*)resident_kernel<kRastrigin, ITEMS>;
        case kAckley: return (const void*)resident_kernel<kAckley, ITEMS>;
        case kRosenbrock: return (const void*)resident_kernel<kRosenbrock, ITEMS>;
        case kCubicMax: return (const void*)resident_kernel<kCubicMax, ITEMS>;
        default: return nullptr;
    }
}

const void* res_kernel(int items, int fid) {
    switch (items) {
        case 1: return res_kernel_i<1>(fid);
        case 2: return res_kernel_i<2>(fid);
        case 3: return res_kernel_i<3>(fid);
        case 4: return res_kernel_i<4>(fid);
        case 5: return res_kernel_i<5>(fid);
        case 6: return res_kernel_i<6>(fid);
        case 8: return res_kernel_i<8>(fid);
        case 12: return res_kernel_i<12>(fid);
        case 16: return res_kernel_i<16>(fid);
        default: return nullptr;
    }
}

}  // namespace

bool resident_fits(const SwarmDev& s, int fid, int num_sms) {
    ResPlan r;
    const bool has_cos = fid == kRastrigin || fid == kAckley;
    if (has_cos && !(std::fabs(s.lo) <= kSmallX && std::fabs(s.hi) <= kSmallX)) return false;
    return fid <= kCubicMax && s.fast_cr && s.fast_clamp && s.pflag && s.N >= 1 && res_plan(s.N, s.D, num_sms, &r);
}

size_t resident_bytes(int N, int D, int num_sms) {
    ResPlan r;
    if (!res_plan(N, D, num_sms, &r)) return 0;
    return 64 + sizeof(float) * 2 * (size_t)r.grid * (size_t)D;
}

ResidentBufs resident_bufs_at(void* base) {
    char* p = static_cast<char*>(base);
    return ResidentBufs{reinterpret_cast<unsigned long long*>(p), reinterpret_cast<unsigned long long*>(p + 32),
                        reinterpret_cast<float*>(p + 64)};
}

// Raises the shared-memory limit of this swarm's kernel. The limit belongs to the kernel,
// which other swarms run too, from other host threads as well: every swarm sets the same one,
// when it is created. (With each swarm's own before each of its launches, two threads with 77824 x 16
// and 20000 x 48 took it from one another and the larger one's launch was refused.)
cudaError_t prepare_resident(const SwarmDev& s, int fid, int num_sms) {
    ResPlan r;
    const void* k = res_plan(s.N, s.D, num_sms, &r) ? res_kernel(r.items, fid) : nullptr;
    if (!k) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmem);
}

cudaError_t launch_resident(const SwarmDev& s, const ResidentBufs& rb, int fid, int panel, int iters, bool stall_barrier,
                            int num_sms, cudaStream_t st) {
    ResPlan r;
    if (!resident_fits(s, fid, num_sms) || !rb.slots || iters < 1 || iters > kResidentMaxIters ||
        !res_plan(s.N, s.D, num_sms, &r))
        return cudaErrorInvalidValue;
    const void* k = res_kernel(r.items, fid);
    if (!k) return cudaErrorInvalidValue;
    unsigned int expect = (unsigned int)r.grid + (stall_barrier ? 1u : 0u);
    ResidentBufs b = rb;
    void* args[] = {const_cast<SwarmDev*>(&s), &b, &r.P, &r.rows, &r.S, &panel, &iters, &expect};
    return cudaLaunchCooperativeKernel(k, dim3(r.grid), dim3(r.threads), args, r.smem, st);
}

}  // namespace cupso
