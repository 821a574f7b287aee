// kernels_sync64.cu -- synchronous double-precision PSO, all iterations of a
// cupso_step call in one cooperative launch. CTA c of at most one per SM owns the particles
// c P .. c P + P - 1 and an iteration ends in a grid barrier on a counter.
//
//  * sync64_reg_kernel: the swarm in registers. Each CTA has P x rows threads;
//    thread (row, p) owns up to ITEMS dimensions (row, row + rows, ...) of particle p.
//    As kernels_resident.cu does it in single precision: after the move, the first
//    warps add the fitness terms in order, one thread per particle, and arrive on the
//    barrier, while the other warps form what the next iteration needs and no gbest
//    enters -- the uniforms, c1 r1 and c2 r2, the inertia and cognitive terms; the
//    last warp polls.
//  * sync64_mem_kernel: larger swarms, the state in memory (in L2 up to 126 MB), the
//    CTA's particles in tiles whose fitness terms fit shared memory.
//
// What bounds them is the FP64 pipe of a GB300: an instruction takes a warp's slot of
// 19 cycles of the SM's pipe (64 until its result) however many lanes are active. So
// the particles are spread evenly over the SMs, every FP64 instruction but the
// ordered sums runs with full warps, and those with 32 particles at a time: 16384 x
// 120 on 152 SMs is 405 x 8 + 4 x 120 instructions per SM, 34 us of the 39.6 an
// iteration takes. (Before: one launch per iteration of tiles of 16 particles, whose
// sums filled half a warp and a fifth of the pipe, and 7 tiles on some SMs, 6 on
// others: 60 us. The paper's one-dimensional swarms, 8192 particles: 1.5 us; with a
// launch and a last-block hand-off per iteration 4.8, in a persistent kernel with one
// particle per thread and everything between two barriers 3.3, on a cluster 4.2.)
//
// Step 5: a CTA with a candidate (lexicographically lowest improved key below
// gbest's) writes its key and position to its slot and releases them with its
// arrival, which also counts it; without one it arrives relaxed -- it has written
// nothing others read. If the count of the iteration's parity moved, every CTA
// reduces all slots; older slots hold keys that gbest has reached since, so they
// never win. Slots and counts are kept by parity: a CTA can be at most one iteration
// ahead of another. Every wait is bounded by s.wait_limit_ns: on expiry the timeout
// status is set and the CTA stops.
#include <cuda_runtime.h>

#include <algorithm>

#include "cupso_device.cuh"
#include "cupso_internal.h"
#include "fp64_common.cuh"
#include "paper_kernels.h"

namespace cupso {

namespace {

constexpr size_t kSync64Smem = 200u * 1024u;   // dynamic shared memory of a CTA at most
constexpr int kMemThreads = 512;
constexpr int kMemChunk = 4;   // items whose loads a thread issues together
// Particles of a tile at most: one per thread, and with few dimensions enough for two
// chunks of items per thread. With 512 whatever D, a one-dimensional tile was one item per thread
// between four barriers: 4 10^6 x 1 (sphere) 169 us an iteration, and 142 in a launch per iteration;
// now 128. 10^6 x 2 61 and 59, now 52; 4 10^6 x 3 330 and 313, now 299.
constexpr int mem_tile(int D) { return std::max(kMemThreads, 2 * kMemChunk * kMemThreads / D); }

// Threads per CTA at most for ITEMS dimensions per thread: what the register file
// holds at 10 registers per item (whole warps per quarter SM).
constexpr int max_threads64(int items) {
    return items <= 1 ? 1024 : (items <= 2 ? 768 : (items <= 4 ? 512 : (items <= 8 ? 384 : 256)));
}

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ PKey load_gkey64(const SwarmDev64& s, int par) {
    PKey k;
    k.k = __ldcg(&s.gkey[par].k);
    k.i = __ldcg(&s.gkey[par].i);
    k.pad = 0u;
    return k;
}

__device__ __forceinline__ PKey* slot_of(const Sync64Bufs& rb, int par, uint32_t cta, int D) {
    return reinterpret_cast<PKey*>(rb.slots + ((size_t)par * gridDim.x + cta) * sync64_slot_bytes(D));
}

// One arrival; `cand`: it carries a candidate of this parity, whose slot was written
// by threads that have passed a barrier with the caller since. `first`: the launch's first, which
// releases the cleared slots. A relaxed one does not order this CTA's reads of older slots
// before other CTAs' next writes of them in the memory model; that holds because the loads
// have returned, their values stored, before the CTA's barriers since.
__device__ __forceinline__ void arrive64(const Sync64Bufs& rb, int par, bool cand, bool first) {
    if (cand || first)
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(rb.bar),
                     "l"(1ull + (cand ? 1ull << (32 + 16 * par) : 0ull))
                     : "memory");
    else
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(rb.bar), "l"(1ull) : "memory");
}

// Waits until `target` arrivals; 0: expired, 1: done, 2: done and this parity's
// candidate count (bits 32..47 even, 48..63 odd, modulo 2^16) has moved since `seen`.
__device__ __forceinline__ int poll64(const SwarmDev64& s, const Sync64Bufs& rb, unsigned int target, int par, uint32_t& seen) {
    unsigned long long w = ld_relaxed_u64(rb.bar);
    if ((unsigned int)w < target) {
        const long long deadline = global_ns() + s.wait_limit_ns;
        while ((unsigned int)(w = ld_relaxed_u64(rb.bar)) < target)
            if (global_ns() > deadline) {
                atomicOr(s.status, kStatusTimeout);
                return 0;
            }
    }
    const uint32_t mask = 0xFFFFu << (16 * par), now = (uint32_t)(w >> 32) & mask;
    const bool moved = now != (seen & mask);
    seen = (seen & ~mask) | now;
    if (moved) asm volatile("fence.acq_rel.gpu;" ::: "memory");   // what the candidates' arrivals released
    return moved ? 2 : 1;
}

// Step 5 after a barrier with candidates: the lowest key of all slots and of K, and
// the winner's position to Gs if it is new. Every thread calls it.
__device__ __forceinline__ void take_gbest64(const Sync64Bufs& rb, int par, int P, int D, PKey& K, double* Gs, PKey* red) {
    PKey m = K;
    for (uint32_t r = threadIdx.x; r < gridDim.x; r += blockDim.x) {
        const PKey* sl = slot_of(rb, par, r, D);
        PKey c;
        c.k = __ldcg(&sl->k);
        c.i = __ldcg(&sl->i);
        c.pad = 0u;
        if (key_less(c, m)) m = c;
    }
    const PKey best = block_min_key(m, red);
    if (key_less(best, K)) {   // uniform
        const double* pos = reinterpret_cast<const double*>(slot_of(rb, par, best.i / (uint32_t)P, D) + 1);
        for (int d = threadIdx.x; d < D; d += blockDim.x) Gs[d] = __ldcg(pos + d);
        K = best;
        __syncthreads();
    }
}

// No candidate in this CTA's slots yet (thread 0, whose first arrival releases it).
__device__ __forceinline__ void clear_slots64(const Sync64Bufs& rb, int D) {
    for (int par = 0; par < 2; ++par) {
        PKey* slot = slot_of(rb, par, blockIdx.x, D);
        __stcg(&slot->k, ~0ull);
        __stcg(&slot->i, kNoIdx);
    }
}

// Thread 0, after a barrier of the CTA: it is done with the exchange. The CTA that leaves last
// clears the counters, so that a launch needs nothing before it (with two memsets before each, a
// PERSISTENT call of one iteration took 11.2 us, with the kernel it had before 10.3; now 8.4).
__device__ __forceinline__ void leave64(const Sync64Bufs& rb) {
    unsigned int* gone = reinterpret_cast<unsigned int*>(rb.bar + 1);
    __threadfence();   // this CTA's arrivals before its leaving
    if (atomicAdd(gone, 1u) == gridDim.x - 1) {
        __threadfence();
        *rb.bar = 0ull;
        *gone = 0u;
    }
}

// The end of a launch: gbest and the iteration counter (one CTA).
__device__ __forceinline__ void store_gbest64(const SwarmDev64& s, uint32_t t_end, const PKey& K, const double* Gs) {
    const int out = (int)(t_end & 1u);
    for (int d = threadIdx.x; d < s.D; d += blockDim.x) s.G[(size_t)out * s.D + d] = Gs[d];
    if (threadIdx.x == 0) {
        s.gkey[0] = K;
        s.gkey[1] = K;
        *s.t_dev = t_end;
    }
}

}  // namespace

// P particles per CTA, blockDim.x >= P * rows in whole warps, ITEMS * rows >= D; S:
// doubles per particle's row of X and H (odd, >= ITEMS * rows). rb.bar and the word behind
// it zero at launch. W1: s.w is 1. `expect`: arrivals that complete a barrier
// (gridDim.x; one more only to test that its bound works).
template <int FIT, bool W1, int ITEMS>
__global__ void __launch_bounds__(max_threads64(ITEMS), 1) sync64_reg_kernel(const __grid_constant__ SwarmDev64 s,
                                                                            const __grid_constant__ Sync64Bufs rb, int P,
                                                                            int rows, int S, int iters, unsigned int expect) {
    constexpr bool kNext = FitTerms64<FIT>::kNeedsNext;
    constexpr bool kH = FIT != kSphere;
    extern __shared__ __align__(16) double sm_s64[];
    const int D = s.D, T = (int)blockDim.x, tid = (int)threadIdx.x;
    double* X = sm_s64;                          // [P][S]
    double* H = X + (size_t)P * S;               // [P][S] if kH
    double* Gs = H + (kH ? (size_t)P * S : 0);   // [ITEMS * rows] gbest_pos, then zeros
    unsigned char* imp = reinterpret_cast<unsigned char*>(Gs + ITEMS * rows);   // [P]
    __shared__ PKey red[32], cred[32];
    __shared__ int s_state;

    const uint32_t base = blockIdx.x * (uint32_t)P;
    const int n = min(P, s.N - (int)base);
    const int row = tid / P, p = tid - row * P;
    const uint32_t i = base + (uint32_t)p;
    // threads past the last row do nothing; particles past N are computed on zeros
    // (their places in X and H exist and are never summed)
    const bool active = row < rows, own = active && p < n;
    const int sum_threads = (P + 31) / 32 * 32;
    const bool sums = tid < sum_threads;         // uniform over a warp
    const int poller = T - 32;
    const size_t Np = (size_t)s.Np;
    const uint32_t t_prev = __ldcg(s.t_dev);
    const int cur0 = (int)(t_prev & 1u);
    if (tid == 0) clear_slots64(rb, D);

    double x[ITEMS], v[ITEMS], pb[ITEMS], cr1[ITEMS], cr2[ITEMS];
    // dimensions past D are skipped: an FP64 instruction costs more than the test
    auto live = [&](int j) { return row + j * rows < D; };
    auto words = [&](uint32_t t) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            if (!live(j)) continue;
            const uint4 r = philox4x32_10(make_uint4((uint32_t)(row + j * rows), i, t, s.swarm), s.key0, s.key1);
            cr1[j] = c_times_u53(s.c1, s.c1_exp, r.x, r.y);
            cr2[j] = c_times_u53(s.c2, s.c2_exp, r.z, r.w);
        }
    };
    auto begin = [&](bool up) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            if (!live(j)) continue;
            if (up) pb[j] = x[j];
            v[j] = __fma_rn(cr1[j], __dsub_rn(pb[j], x[j]), W1 ? v[j] : __dmul_rn(s.w, v[j]));
        }
    };
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int d = row + j * rows;
        x[j] = v[j] = pb[j] = 0.0;
        if (own && d < D) {
            const size_t off = (size_t)d * Np + i;
            x[j] = s.x[off];
            v[j] = s.v[off];
            pb[j] = s.pb[off];
        }
    }
    if (active) {
        words(t_prev + 1u);
        begin(false);
    }
    double pf = tid < n ? s.pf[base + tid] : 0.0;
    if (tid < P) imp[tid] = 0;
    for (int d = tid; d < ITEMS * rows; d += T) Gs[d] = d < D ? s.G[(size_t)cur0 * D + d] : 0.0;
    PKey K = load_gkey64(s, cur0);               // the same in every thread
    uint32_t seen = 0u;                          // the poller: candidate counts by parity
    double* const xo = X + (size_t)p * S + row;
    double* const ho = H + (size_t)p * S + row;
    __syncthreads();

    bool nan = false;
    int done = 0;
    for (int k = 0; k < iters; ++k) {
        const int par = k & 1;
        if (active) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                if (!live(j)) continue;
                const double vel = __fma_rn(cr2[j], __dsub_rn(Gs[row + j * rows], x[j]), v[j]);
                v[j] = clamp64(vel, s.vlo, s.vmax, s.k_vlo, s.k_vhi, s.k_inf);
                x[j] = clamp64(__dadd_rn(x[j], v[j]), s.lo, s.hi, s.k_lo, s.k_hi, s.k_inf);
                xo[j * rows] = x[j];
                if constexpr (kH && !kNext) ho[j * rows] = FitTerms64<FIT>::term(x[j], 0.0);
            }
        }
        __syncthreads();
        if constexpr (kNext) {
            if (active) {
#pragma unroll
                for (int j = 0; j < ITEMS; ++j)
                    if (row + j * rows + 1 < D) ho[j * rows] = FitTerms64<FIT>::term(x[j], xo[j * rows + 1]);
            }
            __syncthreads();
        }
        if (sums) {
            PKey cand = key_none();
            if (tid < n) {
                const double* row_x = X + (size_t)tid * S;
                const double* row_h = H + (size_t)tid * S;
                double acc = 0.0;
                if constexpr (FIT == kSphere) {
#pragma unroll 8
                    for (int d = 0; d < D; ++d) acc = __fma_rn(row_x[d], row_x[d], acc);
                } else {
                    const int nt = kNext ? D - 1 : D;
#pragma unroll 8
                    for (int d = 0; d < nt; ++d) acc = __dadd_rn(acc, row_h[d]);
                }
                const double f = FIT == kCubicMax ? -acc : acc;
                nan |= (f != f);
                const bool better = f < pf;
                imp[tid] = better ? 1 : 0;
                if (better) {
                    pf = f;
                    const PKey c{fit_key64(f), base + (uint32_t)tid, 0u};
                    if (key_less(c, K)) cand = c;
                }
            }
            if (__any_sync(0xFFFFFFFFu, cand.i != kNoIdx)) cand = warp_min_key(cand);
            if ((tid & 31) == 0) cred[tid >> 5] = cand;
            bar_sync(1, sum_threads);
            PKey mine = cred[0];
            for (int w = 1; w < sum_threads / 32; ++w)
                if (key_less(cred[w], mine)) mine = cred[w];
            const bool has = mine.i != kNoIdx;   // uniform over the summing warps
            if (has) {
                PKey* slot = slot_of(rb, par, blockIdx.x, D);
                const double* pos = X + (size_t)(mine.i - base) * S;
                for (int d = tid; d < D; d += sum_threads) __stcg(reinterpret_cast<double*>(slot + 1) + d, pos[d]);
                if (tid == 0) {
                    __stcg(&slot->k, mine.k);
                    __stcg(&slot->i, mine.i);
                }
                bar_sync(1, sum_threads);
            }
            if (tid == 0) arrive64(rb, par, has, k == 0);
            if (T > sum_threads) bar_arrive(2, T);   // the flags are written
        }
        const bool more = k + 1 < iters && active;
        if (more) words(t_prev + 2u + (uint32_t)k);
        if (!sums) bar_sync(2, T);
        if (more) begin(imp[p] != 0);
        if (tid == poller) s_state = poll64(s, rb, (unsigned int)(k + 1) * expect, par, seen);
        __syncthreads();
        const int state = s_state;
        if (!state) break;
        if (state == 2) take_gbest64(rb, par, P, D, K, Gs, red);
        done = k + 1;
    }

    const bool up = own && imp[p] != 0;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int d = row + j * rows;
        if (own && d < D) {
            const size_t off = (size_t)d * Np + i;
            s.x[off] = x[j];
            s.v[off] = v[j];
            s.pb[off] = up ? x[j] : pb[j];
        }
    }
    if (tid < n) s.pf[base + tid] = pf;
    if (__syncthreads_or(nan) && tid == 0) atomicOr(s.status, kStatusNaN);
    if (tid == 0) leave64(rb);
    if (blockIdx.x == 0) store_gbest64(s, t_prev + (uint32_t)done, K, Gs);
}

// The state in memory: PC particles per CTA, taken in tiles of P (at most mem_tile(D)
// and what fits shared memory). A thread keeps its (dimension, particle) items of a
// tile in every iteration, issuing the loads of kMemChunk of them together.
template <int FIT, bool W1>
__global__ void __launch_bounds__(kMemThreads, 1) sync64_mem_kernel(const __grid_constant__ SwarmDev64 s,
                                                                   const __grid_constant__ Sync64Bufs rb, int PC, int P,
                                                                   int iters, unsigned int expect) {
    constexpr bool kNext = FitTerms64<FIT>::kNeedsNext;
    extern __shared__ __align__(16) double sm_s64[];
    const int D = s.D, T = (int)blockDim.x, tid = (int)threadIdx.x;
    double* Y = sm_s64;                               // [D][P] the terms summed (sphere: the positions)
    double* X = kNext ? Y + (size_t)D * P : Y;        // [D][P] positions, where terms pair neighbours
    double* Gs = X + (size_t)D * P;                   // [D]
    unsigned char* imp = reinterpret_cast<unsigned char*>(Gs + D);   // [P]
    __shared__ PKey red[32];
    __shared__ int s_state;

    const uint32_t first = blockIdx.x * (uint32_t)PC;
    const int mine_n = min(PC, s.N - (int)first);     // particles of this CTA (> 0)
    const size_t Np = (size_t)s.Np;
    const uint32_t t_prev = __ldcg(s.t_dev);
    const int cur0 = (int)(t_prev & 1u);
    if (tid == 0) clear_slots64(rb, D);
    for (int d = tid; d < D; d += T) Gs[d] = s.G[(size_t)cur0 * D + d];
    PKey K = load_gkey64(s, cur0);
    uint32_t seen = 0u;
    __syncthreads();

    bool nan = false;
    int done = 0;
    for (int k = 0; k < iters; ++k) {
        const uint32_t t = t_prev + 1u + (uint32_t)k;
        const int par = k & 1;
        PKey cand = key_none();
        for (int p0 = 0; p0 < mine_n; p0 += P) {
            const int n = min(P, mine_n - p0);
            const uint32_t base = first + (uint32_t)p0;
            const int items = n * D;
            // items e = d * n + p, from tid on in steps of T, without a division per item
            const int dstep = T / n, pstep = T - dstep * n;
            int d = tid / n, p = tid - d * n;
            auto next = [&]() {
                p += pstep;
                d += dstep;
                if (p >= n) {
                    p -= n;
                    ++d;
                }
            };
            for (int e0 = tid; e0 < items; e0 += kMemChunk * T) {
                double xs[kMemChunk], vs[kMemChunk], ps[kMemChunk];
                int dd[kMemChunk], pp[kMemChunk];
#pragma unroll
                for (int c = 0; c < kMemChunk; ++c) {
                    dd[c] = d;
                    pp[c] = p;
                    if (d < D) {
                        const size_t off = (size_t)d * Np + (base + (uint32_t)p);
                        xs[c] = s.x[off];
                        vs[c] = s.v[off];
                        ps[c] = s.pb[off];
                    }
                    next();
                }
#pragma unroll
                for (int c = 0; c < kMemChunk; ++c) {
                    if (dd[c] >= D) break;
                    const uint32_t i = base + (uint32_t)pp[c];
                    const size_t off = (size_t)dd[c] * Np + i;
                    const uint4 r = philox4x32_10(make_uint4((uint32_t)dd[c], i, t, s.swarm), s.key0, s.key1);
                    double xx = xs[c], vv = vs[c];
                    move_one64_t<W1>(xx, vv, ps[c], Gs[dd[c]], r, s);
                    s.x[off] = xx;
                    s.v[off] = vv;
                    const int at = dd[c] * P + pp[c];
                    if constexpr (FIT == kCubicMax) Y[at] = FitTerms64<FIT>::term(xx, 0.0);
                    else X[at] = xx;
                }
            }
            __syncthreads();
            if constexpr (kNext) {
                for (int dn = tid / n, pn = tid % n; dn + 1 < D;) {
                    Y[dn * P + pn] = FitTerms64<FIT>::term(X[dn * P + pn], X[(dn + 1) * P + pn]);
                    pn += pstep;
                    dn += dstep;
                    if (pn >= n) {
                        pn -= n;
                        ++dn;
                    }
                }
                __syncthreads();
            }
            for (int q = tid; q < n; q += T) {   // more than one each only where D < 2 kMemChunk
                const uint32_t i = base + (uint32_t)q;
                const double f = FitTerms64<FIT>::sum(Y, Y, P, q, D);
                nan |= (f != f);
                const bool better = f < s.pf[i];
                imp[q] = better ? 1 : 0;
                if (better) {
                    s.pf[i] = f;
                    const PKey c{fit_key64(f), i, 0u};
                    if (key_less(c, K) && key_less(c, cand)) cand = c;
                }
            }
            __syncthreads();
            // improved rows of pbest_pos, each thread from the positions it wrote itself
            d = tid / n;
            p = tid - d * n;
            while (d < D) {
                if (imp[p]) {
                    const size_t off = (size_t)d * Np + (base + (uint32_t)p);
                    s.pb[off] = s.x[off];
                }
                next();
            }
            __syncthreads();   // Y, X and imp are free for the next tile
        }
        const PKey best = block_min_key(cand, red);
        const bool has = best.i != kNoIdx;
        if (has) {
            PKey* slot = slot_of(rb, par, blockIdx.x, D);
            for (int d = tid; d < D; d += T) __stcg(reinterpret_cast<double*>(slot + 1) + d, s.x[(size_t)d * Np + best.i]);
            if (tid == 0) {
                __stcg(&slot->k, best.k);
                __stcg(&slot->i, best.i);
            }
            __syncthreads();
        }
        if (tid == 0) {
            arrive64(rb, par, has, k == 0);
            s_state = poll64(s, rb, (unsigned int)(k + 1) * expect, par, seen);
        }
        __syncthreads();
        const int state = s_state;
        if (!state) break;
        if (state == 2) take_gbest64(rb, par, PC, D, K, Gs, red);
        done = k + 1;
    }
    if (__syncthreads_or(nan) && tid == 0) atomicOr(s.status, kStatusNaN);
    if (tid == 0) leave64(rb);
    if (blockIdx.x == 0) store_gbest64(s, t_prev + (uint32_t)done, K, Gs);
}

namespace {

struct Plan64 {
    int P = 0, grid = 0, rows = 0, items = 0, threads = 0, S = 0, PC = 0;   // items 0: the state in memory
    size_t smem = 0;
};

bool plan64(int fid, int N, int D, int num_sms, Plan64* r) {
    // The particles spread over the SMs, but of small swarms up to 64 (dimension, particle) items to a
    // CTA, over at least 8 CTAs: one swarm is as fast or faster (an iteration of 300 x 2 1.53 and 1.09 us,
    // 8192 x 1 1.56 and 1.49), and many on streams of their own run side by side (64 of 2000 x 1: 0.24 us
    // per swarm and iteration, 0.09 on clusters, now 0.09). In one dimension whole warps instead, where a
    // part of one or a second one costs more than CTAs save: 32 particles to 32 CTAs, then 64 (128 x 1
    // 1.48 us with a CTA each, 1.52 with 16 to a CTA, 1.22-1.43 so; 1024 x 1 1.48, 1.49 with 64, 1.42; 2048 x 1
    // 1.48, 1.50 so, and with 32 1.41 but 64 of them 0.17).
    const int small = D == 1 ? std::min(std::max((N + 31) / 32, 32), 64) : std::min((N + 7) / 8, 64 / D);
    const int PC = std::max((N + num_sms - 1) / num_sms, small);
    r->PC = PC;
    r->grid = (N + PC - 1) / PC;
    for (int items = 1; items <= 16; items *= 2) {
        const int rows = (D + items - 1) / items;
        if ((long long)PC * rows > max_threads64(items)) continue;
        r->P = PC;
        r->items = items;
        r->rows = rows;
        r->threads = (PC * rows + 31) / 32 * 32;
        r->S = (items * rows) | 1;
        r->smem = sizeof(double) * (2 * (size_t)PC * r->S + (size_t)items * rows) + (size_t)PC;
        if (r->smem <= kSync64Smem) return true;
    }
    // tiles of equal size, as few as fit shared memory
    const size_t per = sizeof(double) * (size_t)D * (fid == kRosenbrock ? 2 : 1) + 1;
    const size_t room = kSync64Smem - std::min(kSync64Smem, sizeof(double) * (size_t)D);
    const int most = (int)std::min<size_t>(mem_tile(D), room / per);
    if (most < 1) return false;
    const int tiles = (PC + most - 1) / most;
    r->items = 0;
    r->P = (PC + tiles - 1) / tiles;
    r->threads = kMemThreads;
    r->smem = per * (size_t)r->P + sizeof(double) * (size_t)D;
    return true;
}

template <int FIT, bool W1>
const void* kernel64(int items) {
    switch (items) {
        case 0: return (const void*)sync64_mem_kernel<FIT, W1>;
        case 1: return (const void*)sync64_reg_kernel<FIT, W1, 1>;
        case 2: return (const void*)sync64_reg_kernel<FIT, W1, 2>;
        case 4: return (const void*)sync64_reg_kernel<FIT, W1, 4>;
        case 8: return (const void*)sync64_reg_kernel<FIT, W1, 8>;
        case 16: return (const void*)sync64_reg_kernel<FIT, W1, 16>;
        default: return nullptr;
    }
}

const void* kernel64(int fid, bool w1, int items) {
    switch (fid) {
        case kSphere: return w1 ? kernel64<kSphere, true>(items) : kernel64<kSphere, false>(items);
        case kRosenbrock: return w1 ? kernel64<kRosenbrock, true>(items) : kernel64<kRosenbrock, false>(items);
        case kCubicMax: return w1 ? kernel64<kCubicMax, true>(items) : kernel64<kCubicMax, false>(items);
        default: return nullptr;
    }
}

}  // namespace

size_t sync64_bytes(int fid, int N, int D, int num_sms) {
    Plan64 r;
    return plan64(fid, N, D, num_sms, &r) ? 64 + 2 * (size_t)r.grid * sync64_slot_bytes(D) : 0;
}

Sync64Bufs sync64_bufs_at(void* base) {
    return Sync64Bufs{static_cast<unsigned long long*>(base), static_cast<unsigned char*>(base) + 64};
}

// Raises the shared-memory limit of this swarm's kernel, to the same value for every swarm (it
// belongs to the kernel, which swarms of other sizes run from other host threads).
cudaError_t prepare_sync64(const SwarmDev64& s, int fid, int num_sms) {
    Plan64 r;
    const void* k = plan64(fid, s.N, s.D, num_sms, &r) ? kernel64(fid, s.w_one != 0, r.items) : nullptr;
    if (!k) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSync64Smem);
}

cudaError_t launch_sync64(const SwarmDev64& s, const Sync64Bufs& rb, int fid, int iters, int per_launch, bool stall_barrier,
                          int num_sms, cudaStream_t st) {
    Plan64 r;
    if (!rb.slots || iters < 1 || per_launch < 1 || per_launch > kSync64MaxIters || !plan64(fid, s.N, s.D, num_sms, &r)) return cudaErrorInvalidValue;
    const void* k = kernel64(fid, s.w_one != 0, r.items);
    if (!k) return cudaErrorInvalidValue;
    unsigned int expect = (unsigned int)r.grid + (stall_barrier ? 1u : 0u);
    cudaError_t e = cudaSuccess;
    for (int left = iters; e == cudaSuccess && left > 0;) {
        int n = std::min(left, per_launch);
        left -= n;
        SwarmDev64 sa = s;
        Sync64Bufs ba = rb;
        void* reg_args[] = {&sa, &ba, &r.P, &r.rows, &r.S, &n, &expect};
        void* mem_args[] = {&sa, &ba, &r.PC, &r.P, &n, &expect};
        e = cudaLaunchCooperativeKernel(k, dim3(r.grid), dim3(r.threads), r.items ? reg_args : mem_args, r.smem, st);
    }
    return e;
}

}  // namespace cupso
