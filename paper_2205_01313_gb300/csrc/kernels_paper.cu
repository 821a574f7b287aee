// kernels_paper.cu -- the paper's own GPU designs, one particle per thread,
// and the double-precision swarm.
//
// The paper maps one particle to one thread (Sec. 2.2) and compares four ways
// of finding the global best after Steps 2-4:
//  * reduction (Sec. 2.2, Fig. 1): every block reduces its particles' pbest
//    to one entry of an auxiliary array, a second kernel reduces that array;
//  * loop unrolling (Sec. 2.2): the same with the reduction loop unrolled;
//  * queue (Sec. 3.1, Alg. 2): only particles that beat the global best enter
//    a shared-memory queue through an atomic add, thread 0 scans the queue into
//    the block's auxiliary entry, and the second kernel does the same over the
//    blocks;
//  * queue lock (Sec. 3.2, Alg. 3): thread 0 takes a global lock and updates
//    the global best itself, so the second kernel disappears. The update is in
//    place: blocks that run later in the same launch already see it.
// Here they are rebuilt for both precisions, as comparison baselines beside
// the library's own kernels. The candidate order is lexicographic on
// (fitness key, index), so every variant but the queue lock gives the
// synchronous result exactly. Iterations read the counter from device memory
// (graph-capturable); the one-kernel variants roll it from the last block.
//
// The double-precision swarm runs the paper's workload in its precision:
// binary64 state, 53-bit uniforms, sphere / Rosenbrock / the cubic of Eq. 3.
// Besides the four designs above it has a fused one-launch synchronous step
// (block argmin, a short candidate list, the last block gathers gbest) and an
// on-chip kernel that keeps a small swarm in one CTA's shared memory for many
// iterations.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "cupso_device.cuh"
#include "cupso_internal.h"
#include "fp64_common.cuh"
#include "paper_kernels.h"
#include "pdl.cuh"
#include "stream_common.cuh"

namespace cg = cooperative_groups;

namespace cupso {

namespace {

// Appends a block's candidate to the list; a push beyond the capacity is
// dropped and reported (launchers never start more blocks than list_cap).
__device__ __forceinline__ void push_candidate(const PaperBufs& b, const PKey& k, unsigned int* status) {
    const unsigned int slot = atomicAdd(b.list_n, 1u);
    if (slot < b.list_cap) b.list[slot] = k;
    else atomicOr(status, kStatusBadArg);
}

__device__ __forceinline__ unsigned long long ld_volatile_u64(const unsigned long long* p) {
    return *reinterpret_cast<const volatile unsigned long long*>(p);
}

// ---------------------------------------------------------------------------
// Precision adapters: what the generic kernels need from each swarm type.
// ---------------------------------------------------------------------------
struct Fp32 {
    using Dev = SwarmDev;
    using T = float;

    // Steps 2-3 for particle i at iteration t: one Philox call per dimension pair.
    template <int FIT>
    __device__ static float step_particle(const SwarmDev& s, uint32_t i, uint32_t t, const float* G) {
        const size_t Np = (size_t)s.Np;
        FitAcc<FIT> acc;
        for (int d0 = 0; d0 < s.D; d0 += 2) {
            const uint4 r = philox4x32_10(make_uint4((uint32_t)(d0 >> 1), i, t, s.swarm), s.key0, s.key1);
            for (int h = 0; h < 2 && d0 + h < s.D; ++h) {
                const int d = d0 + h;
                const size_t off = (size_t)d * Np + i;
                float x = s.x[off], v = s.v[off];
                move_one(x, v, s.pb[off], G[d], u01(word(r, 2 * h)), u01(word(r, 2 * h + 1)), s);
                s.x[off] = x;
                s.v[off] = v;
                acc.add(d, x);
            }
        }
        return acc.finish(s.D);
    }
    __device__ static PKey key(float f, uint32_t i) { return PKey{(unsigned long long)fit_key(f), i, 0u}; }
    // fitness part of the current gbest key (a single 64-bit load)
    __device__ static unsigned long long gk(const SwarmDev& s, int par) { return ld_volatile_u64(s.gkey + par) >> 32; }
    __device__ static PKey load_gkey(const SwarmDev& s, int par) {
        const unsigned long long k = ld_volatile_u64(s.gkey + par);
        return PKey{k >> 32, (uint32_t)(k & 0xFFFFFFFFull), 0u};
    }
    __device__ static void store_gkey(const SwarmDev& s, int par, PKey k) {
        *reinterpret_cast<volatile unsigned long long*>(s.gkey + par) = (k.k << 32) | (unsigned long long)k.i;
    }
};

struct Fp64 {
    using Dev = SwarmDev64;
    using T = double;

    // Steps 2-3 for particle i at iteration t: one Philox call per dimension.
    template <int FIT>
    __device__ static double step_particle(const SwarmDev64& s, uint32_t i, uint32_t t, const double* G) {
        const size_t Np = (size_t)s.Np;
        FitAcc64<FIT> acc;
        for (int d = 0; d < s.D; ++d) {
            const uint4 r = philox4x32_10(make_uint4((uint32_t)d, i, t, s.swarm), s.key0, s.key1);
            const size_t off = (size_t)d * Np + i;
            double x = s.x[off], v = s.v[off];
            move_one64(x, v, s.pb[off], G[d], r, s);
            s.x[off] = x;
            s.v[off] = v;
            acc.add(d, x);
        }
        return acc.finish();
    }
    __device__ static PKey key(double f, uint32_t i) { return PKey{fit_key64(f), i, 0u}; }
    __device__ static unsigned long long gk(const SwarmDev64& s, int par) { return ld_volatile_u64(&s.gkey[par].k); }
    __device__ static PKey load_gkey(const SwarmDev64& s, int par) {
        const volatile PKey* p = s.gkey + par;
        return PKey{p->k, p->i, 0u};
    }
    __device__ static void store_gkey(const SwarmDev64& s, int par, PKey k) {
        volatile PKey* p = s.gkey + par;
        p->i = k.i;
        p->k = k.k;
    }
};

// ---------------------------------------------------------------------------
// Alg. 3: thread 0 of a block with a candidate takes the global lock (a
// bounded wait: on expiry the timeout status is set and the update skipped),
// re-checks against the global best and, if it is better, writes gbest_pos
// (from the candidate's pbest row: index first, position after) and the key.
// ---------------------------------------------------------------------------
template <class A>
__device__ void locked_update(const typename A::Dev& s, const PaperBufs& b, int cur, PKey best) {
    const long long deadline = global_ns() + s.wait_limit_ns;
    bool got = false;
    for (;;) {
        if (atomicCAS(b.lock, 0u, 1u) == 0u) {
            got = true;
            break;
        }
        if (global_ns() > deadline) break;
        __nanosleep(64);
    }
    if (!got) {
        atomicOr(s.status, kStatusTimeout);
        return;
    }
    __threadfence();
    const PKey K = A::load_gkey(s, cur);
    if (key_less(best, K)) {
        const size_t Np = (size_t)s.Np;
        for (int d = 0; d < s.D; ++d) s.G[(size_t)cur * s.D + d] = __ldcg(s.pb + (size_t)d * Np + best.i);
        __threadfence();
        A::store_gkey(s, cur, best);
        __threadfence();
    }
    atomicExch(b.lock, 0u);
}

// ---------------------------------------------------------------------------
// One iteration's first (or only) kernel: Steps 2-4 for one particle per
// thread, then the block's part of Step 5 in the chosen design.
// ---------------------------------------------------------------------------
template <class A, int FIT, int AGG>
__global__ void __launch_bounds__(kPaperBlock) paper_step_kernel(const __grid_constant__ typename A::Dev s,
                                                                 const __grid_constant__ PaperBufs b) {
    using T = typename A::T;
    __shared__ PKey red[kPaperBlock];   // tree operands, or the queue
    __shared__ unsigned int qn;
    __shared__ int s_last;
    pdl_wait();
    pdl_launch_next();
    const uint32_t t_prev = __ldcg(s.t_dev);
    const uint32_t t = t_prev + 1u;
    const int cur = (int)(t_prev & 1u), nxt = cur ^ 1;
    const int tid = threadIdx.x;
    const uint32_t i = blockIdx.x * (uint32_t)kPaperBlock + (uint32_t)tid;
    const size_t Np = (size_t)s.Np;
    if (tid == 0) qn = 0u;
    __syncthreads();

    PKey mine = key_none();
    bool nan = false;
    if (i < (uint32_t)s.N) {
        const T f = A::template step_particle<FIT>(s, i, t, s.G + (size_t)cur * s.D);   // Steps 2-3
        nan = (f != f);
        const T pf = s.pf[i];
        const bool imp = f < pf;                                                         // Step 4
        if (imp) {
            s.pf[i] = f;
            for (int d = 0; d < s.D; ++d) s.pb[(size_t)d * Np + i] = s.x[(size_t)d * Np + i];
        }
        if constexpr (AGG == kAggReduce || AGG == kAggReduceUnrolled) {
            mine = A::key(imp ? f : pf, i);              // the reduction takes every particle
        } else if (imp) {
            // Sec. 3.1: only a particle that improved and can beat the global best
            // competes. Comparing the fitness key alone (<=) keeps every particle
            // that could win a tie on its index.
            const PKey k = A::key(f, i);
            if (k.k <= A::gk(s, cur)) mine = k;
        }
    }

    if constexpr (AGG == kAggReduce) {
        red[tid] = mine;
        __syncthreads();
        for (int st = kPaperBlock / 2; st > 0; st >>= 1) {
            if (tid < st && key_less(red[tid + st], red[tid])) red[tid] = red[tid + st];
            __syncthreads();
        }
        if (tid == 0) b.aux[blockIdx.x] = red[0];
    } else if constexpr (AGG == kAggReduceUnrolled) {
        red[tid] = mine;
        __syncthreads();
#pragma unroll
        for (int st = kPaperBlock / 2; st > 32; st >>= 1) {
            if (tid < st && key_less(red[tid + st], red[tid])) red[tid] = red[tid + st];
            __syncthreads();
        }
        if (tid < 32) {
            PKey k = red[tid];
            if (key_less(red[tid + 32], k)) k = red[tid + 32];
            k = warp_min_key(k);
            if (tid == 0) b.aux[blockIdx.x] = k;
        }
    } else if constexpr (AGG == kAggQueue || AGG == kAggQueueLock) {
        // Alg. 2: the rare candidates enter the block's queue in atomic order
        if (mine.i != kNoIdx) red[atomicAdd(&qn, 1u)] = mine;
        __syncthreads();
        if (tid == 0) {
            PKey best = key_none();
            const unsigned int n = qn;
            for (unsigned int j = 0; j < n; ++j)
                if (key_less(red[j], best)) best = red[j];
            if constexpr (AGG == kAggQueue) {
                b.aux[blockIdx.x] = best;
            } else if (best.i != kNoIdx) {
                locked_update<A>(s, b, cur, best);   // Alg. 3
            }
        }
    } else {  // kAggSyncList
        const PKey k = block_min_key(mine, red);
        if (tid == 0 && k.i != kNoIdx) push_candidate(b, k, s.status);
    }
    if (__syncthreads_or(nan) && tid == 0) atomicOr(s.status, kStatusNaN);

    if constexpr (AGG == kAggQueueLock || AGG == kAggSyncList) {
        // The last block to finish closes the iteration.
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = (atomicAdd(b.ticket, 1u) == gridDim.x - 1);
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        if constexpr (AGG == kAggQueueLock) {
            // the in-place gbest of this iteration is the next iteration's
            for (int d = tid; d < s.D; d += blockDim.x)
                s.G[(size_t)nxt * s.D + d] = __ldcg(s.G + (size_t)cur * s.D + d);
            if (tid == 0) A::store_gkey(s, nxt, A::load_gkey(s, cur));
        } else {
            const unsigned int n = min(__ldcg(b.list_n), b.list_cap);
            PKey k = tid == 0 ? A::load_gkey(s, cur) : key_none();
            for (unsigned int j = tid; j < n; j += blockDim.x) {
                PKey c;
                c.k = __ldcg(&b.list[j].k);
                c.i = __ldcg(&b.list[j].i);
                c.pad = 0u;
                if (key_less(c, k)) k = c;
            }
            const PKey best = block_min_key(k, red);
            if (best.i < (uint32_t)s.N)
                for (int d = tid; d < s.D; d += blockDim.x)
                    s.G[(size_t)nxt * s.D + d] = __ldcg(s.pb + (size_t)d * Np + best.i);
            if (tid == 0) {
                A::store_gkey(s, nxt, best);
                A::store_gkey(s, cur, best);
                *b.list_n = 0u;
            }
        }
        __syncthreads();
        if (tid == 0) {
            *b.ticket = 0u;
            *s.t_dev = t;
        }
    }
}

// ---------------------------------------------------------------------------
// Second kernel (one block): over the blocks' auxiliary entries. REDUCE and
// REDUCE_UNROLLED reduce all of them (every particle's pbest took part);
// QUEUE runs Alg. 2 once more: entries that beat the global best enter a
// queue that thread 0 scans. ADVANCE: this closes iteration t_prev + 1
// (gbest into the next parity, counter rolled); otherwise it sets the gbest
// of the current iteration (after the initialisation or a loaded state).
// ---------------------------------------------------------------------------
template <class A, int AGG, bool ADVANCE>
__global__ void __launch_bounds__(1024) paper_finish_kernel(const __grid_constant__ typename A::Dev s,
                                                            const __grid_constant__ PaperBufs b, int nblocks) {
    __shared__ PKey red[1024];
    __shared__ unsigned int qn;
    pdl_wait();
    pdl_launch_next();
    const int tid = threadIdx.x;
    const uint32_t t_prev = __ldcg(s.t_dev);
    const int cur = (int)(t_prev & 1u);
    const int out = ADVANCE ? (cur ^ 1) : cur;
    PKey k = key_none();
    for (int j = tid; j < nblocks; j += blockDim.x) {
        PKey c;
        c.k = __ldcg(&b.aux[j].k);
        c.i = __ldcg(&b.aux[j].i);
        c.pad = 0u;
        if (key_less(c, k)) k = c;
    }
    PKey best;
    if constexpr (AGG == kAggQueue) {
        if (tid == 0) qn = 0u;
        __syncthreads();
        const PKey K = A::load_gkey(s, cur);
        if (k.i != kNoIdx && key_less(k, K)) red[atomicAdd(&qn, 1u)] = k;
        __syncthreads();
        if (tid == 0) {
            PKey m = K;
            const unsigned int n = qn;
            for (unsigned int j = 0; j < n; ++j)
                if (key_less(red[j], m)) m = red[j];
            red[0] = m;
        }
        __syncthreads();
        best = red[0];
    } else {
        red[tid] = k;
        __syncthreads();
        const int lim = AGG == kAggReduceUnrolled ? 32 : 0;
        for (int st = blockDim.x / 2; st > lim; st >>= 1) {
            if (tid < st && key_less(red[tid + st], red[tid])) red[tid] = red[tid + st];
            __syncthreads();
        }
        if (AGG == kAggReduceUnrolled && tid < 32) {
            PKey m = red[tid];
            if (key_less(red[tid + 32], m)) m = red[tid + 32];
            m = warp_min_key(m);
            if (tid == 0) red[0] = m;
        }
        __syncthreads();
        best = red[0];
    }
    const size_t Np = (size_t)s.Np;
    if (best.i < (uint32_t)s.N)
        for (int d = tid; d < s.D; d += blockDim.x) s.G[(size_t)out * s.D + d] = __ldcg(s.pb + (size_t)d * Np + best.i);
    if (tid == 0) {
        A::store_gkey(s, 0, best);
        A::store_gkey(s, 1, best);
        if (ADVANCE) *s.t_dev = t_prev + 1u;
    }
}

// ---------------------------------------------------------------------------
// FP64 Step 1 (t = 0) and the gbest of a loaded state.
// ---------------------------------------------------------------------------
template <int FIT>
__global__ void __launch_bounds__(kPaperBlock) init64_kernel(const __grid_constant__ SwarmDev64 s,
                                                             const __grid_constant__ PaperBufs b) {
    __shared__ PKey red[32];
    const uint32_t i = blockIdx.x * (uint32_t)kPaperBlock + threadIdx.x;
    const size_t Np = (size_t)s.Np;
    PKey mine = key_none();
    bool nan = false;
    if (i < (uint32_t)s.N) {
        const double span = __dsub_rn(s.hi, s.lo);
        const double vspan = __dmul_rn(2.0, s.vmax);
        FitAcc64<FIT> acc;
        for (int d = 0; d < s.D; ++d) {
            const uint4 r = philox4x32_10(make_uint4((uint32_t)d, i, 0u, s.swarm), s.key0, s.key1);
            const double x = clamp64(__fma_rn(u53(r.x, r.y), span, s.lo), s.lo, s.hi, s.k_lo, s.k_hi, s.k_inf);
            const double v = clamp64(__fma_rn(u53(r.z, r.w), vspan, -s.vmax), -s.vmax, s.vmax, s.k_vlo, s.k_vhi, s.k_inf);
            const size_t off = (size_t)d * Np + i;
            s.x[off] = x;
            s.v[off] = v;
            s.pb[off] = x;
            acc.add(d, x);
        }
        const double f = acc.finish();
        s.pf[i] = f;
        nan = (f != f);
        mine = Fp64::key(f, i);
    }
    const PKey k = block_min_key(mine, red);
    if (threadIdx.x == 0) b.aux[blockIdx.x] = k;
    if (__syncthreads_or(nan) && threadIdx.x == 0) atomicOr(s.status, kStatusNaN);
}

__global__ void __launch_bounds__(kPaperBlock) pbest_min64_kernel(const __grid_constant__ SwarmDev64 s,
                                                                  const __grid_constant__ PaperBufs b) {
    __shared__ PKey red[32];
    const uint32_t i = blockIdx.x * (uint32_t)kPaperBlock + threadIdx.x;
    PKey mine = key_none();
    bool nan = false;
    if (i < (uint32_t)s.N) {
        const double f = s.pf[i];
        nan = (f != f);
        mine = Fp64::key(f, i);
    }
    const PKey k = block_min_key(mine, red);
    if (threadIdx.x == 0) b.aux[blockIdx.x] = k;
    if (__syncthreads_or(nan) && threadIdx.x == 0) atomicOr(s.status, kStatusNaN);
}

// ---------------------------------------------------------------------------
// On-chip FP64 swarm: a cluster of C CTAs (1 <= C <= 16). CTA r keeps the
// particles [r P, r P + n_r) -- x, v, pbest_pos and the fitness terms
// ([D][P]), pbest_fit and its copy of gbest -- in shared memory for `iters`
// iterations. Per iteration every CTA pushes its best candidate (key and
// position) into slot [parity][r] of every CTA of the cluster through
// distributed shared memory (index first, position after, Sec. 4.3); one
// cluster barrier replaces the paper's kernel boundary (Sec. 2.2), and every
// CTA reduces the same slots in the same order, so all hold the same gbest.
// ---------------------------------------------------------------------------
constexpr int kOnchip64Threads = 1024;
constexpr int kMaxCluster64 = 16;

struct Onchip64Layout {
    int P;                                  // particles per CTA
    size_t o_x, o_v, o_pb, o_h, o_pf, o_G, o_red, o_slots, slot, bytes;
};

__host__ __device__ inline size_t al16(size_t x) { return (x + 15) / 16 * 16; }

__host__ __device__ inline Onchip64Layout onchip64_layout(int N, int D, int C) {
    Onchip64Layout L;
    L.P = (N + C - 1) / C;
    const size_t plane = sizeof(double) * (size_t)L.P * (size_t)D;
    size_t o = 0;
    L.o_x = o; o = al16(o + plane);
    L.o_v = o; o = al16(o + plane);
    L.o_pb = o; o = al16(o + plane);
    L.o_h = o; o = al16(o + plane);
    L.o_pf = o; o = al16(o + sizeof(double) * (size_t)L.P);
    L.o_G = o; o = al16(o + sizeof(double) * (size_t)D);
    L.o_red = o; o = al16(o + sizeof(PKey) * 32);
    L.slot = al16(sizeof(PKey) + sizeof(double) * (size_t)D);
    L.o_slots = o; o += 2 * (size_t)C * L.slot;
    L.bytes = o;
    return L;
}

template <int FIT>
__global__ void __launch_bounds__(kOnchip64Threads) onchip64_kernel(const __grid_constant__ SwarmDev64 s, int iters) {
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int N = s.N, D = s.D;
    const Onchip64Layout L = onchip64_layout(N, D, C);
    const int P = L.P;
    const int base = rank * P;
    const int n = max(0, min(P, N - base));       // particles of this CTA
    double* x = reinterpret_cast<double*>(smem + L.o_x);    // [D][P]
    double* v = reinterpret_cast<double*>(smem + L.o_v);
    double* pb = reinterpret_cast<double*>(smem + L.o_pb);
    double* H = reinterpret_cast<double*>(smem + L.o_h);
    double* pf = reinterpret_cast<double*>(smem + L.o_pf);
    double* G = reinterpret_cast<double*>(smem + L.o_G);
    PKey* red = reinterpret_cast<PKey*>(smem + L.o_red);
    unsigned char* slots = smem + L.o_slots;
    const size_t Np = (size_t)s.Np;
    const int tid = threadIdx.x;
    const uint32_t t_prev = __ldcg(s.t_dev);
    const int cur0 = (int)(t_prev & 1u);
    const int nD = n * D;

    for (int e = tid; e < nD; e += blockDim.x) {
        const int d = e / n, p = e - d * n;
        const size_t g = (size_t)d * Np + (size_t)(base + p);
        x[d * P + p] = s.x[g];
        v[d * P + p] = s.v[g];
        pb[d * P + p] = s.pb[g];
    }
    for (int p = tid; p < n; p += blockDim.x) pf[p] = s.pf[base + p];
    for (int d = tid; d < D; d += blockDim.x) G[d] = s.G[(size_t)cur0 * D + d];
    PKey K = Fp64::load_gkey(s, cur0);
    __syncthreads();

    bool nan = false;
    for (int k = 0; k < iters; ++k) {
        const uint32_t t = t_prev + 1u + (uint32_t)k;
        // Step 2 for every (dimension, particle); the fitness terms that need only x_d
        for (int e = tid; e < nD; e += blockDim.x) {
            const int d = e / n, p = e - d * n;
            const int j = d * P + p;
            const uint4 r = philox4x32_10(make_uint4((uint32_t)d, (uint32_t)(base + p), t, s.swarm), s.key0, s.key1);
            double xx = x[j], vv = v[j];
            move_one64(xx, vv, pb[j], G[d], r, s);
            x[j] = xx;
            v[j] = vv;
            if constexpr (!FitTerms64<FIT>::kNeedsNext && FIT != kSphere) H[j] = FitTerms64<FIT>::term(xx, 0.0);
        }
        __syncthreads();
        if constexpr (FitTerms64<FIT>::kNeedsNext) {
            for (int e = tid; e < nD; e += blockDim.x) {
                const int d = e / n, p = e - d * n;
                if (d + 1 < D) H[d * P + p] = FitTerms64<FIT>::term(x[d * P + p], x[(d + 1) * P + p]);
            }
            __syncthreads();
        }
        // Steps 3-4 per particle; this CTA's Step-5 candidate
        PKey cand = key_none();
        for (int p = tid; p < n; p += blockDim.x) {
            const double f = FitTerms64<FIT>::sum(x, H, P, p, D);
            nan |= (f != f);
            if (f < pf[p]) {
                pf[p] = f;
                for (int d = 0; d < D; ++d) pb[d * P + p] = x[d * P + p];
                const PKey c = Fp64::key(f, (uint32_t)(base + p));
                if (key_less(c, K) && key_less(c, cand)) cand = c;
            }
        }
        const PKey best = block_min_key(cand, red);   // barriers inside
        // push (key, position) into slot [par][rank] of every CTA
        const int par = k & 1;
        const size_t my_slot = ((size_t)par * C + rank) * L.slot;
        if (tid < C) {
            unsigned char* remote = cluster.map_shared_rank(slots, tid);
            *reinterpret_cast<PKey*>(remote + my_slot) = best;
        }
        if (best.i != kNoIdx) {
            const int pc = (int)best.i - base;
            for (int e = tid; e < C * D; e += blockDim.x) {
                const int r = e / D, d = e - r * D;
                unsigned char* remote = cluster.map_shared_rank(slots, r);
                reinterpret_cast<double*>(remote + my_slot + sizeof(PKey))[d] = pb[d * P + pc];
            }
        }
        cluster.sync();
        // Step 5: the same reduction over the slots in every CTA
        PKey bk = K;
        int win = -1;
        for (int r = 0; r < C; ++r) {
            const PKey kk = *reinterpret_cast<const PKey*>(slots + ((size_t)par * C + r) * L.slot);
            if (key_less(kk, bk)) {
                bk = kk;
                win = r;
            }
        }
        if (win >= 0) {
            const double* row = reinterpret_cast<const double*>(slots + ((size_t)par * C + win) * L.slot + sizeof(PKey));
            for (int d = tid; d < D; d += blockDim.x) G[d] = row[d];
            K = bk;
        }
        __syncthreads();
    }
    for (int e = tid; e < nD; e += blockDim.x) {
        const int d = e / n, p = e - d * n;
        const size_t g = (size_t)d * Np + (size_t)(base + p);
        s.x[g] = x[d * P + p];
        s.v[g] = v[d * P + p];
        s.pb[g] = pb[d * P + p];
    }
    for (int p = tid; p < n; p += blockDim.x) s.pf[base + p] = pf[p];
    if (__syncthreads_or(nan) && tid == 0) atomicOr(s.status, kStatusNaN);
    if (rank == 0) {
        const int out = (int)((t_prev + (uint32_t)iters) & 1u);
        for (int d = tid; d < D; d += blockDim.x) s.G[(size_t)out * D + d] = G[d];
        if (tid == 0) {
            Fp64::store_gkey(s, 0, K);
            Fp64::store_gkey(s, 1, K);
            *s.t_dev = t_prev + (uint32_t)iters;
        }
    }
    // no CTA leaves while another may still read its shared memory
    cluster.sync();
}

// ---------------------------------------------------------------------------
// FP64 synchronous step for many dimensions: a block takes a tile of P
// particles with all D dimensions and spreads its (dimension, particle) pairs
// over the threads (the one-particle-per-thread designs leave most SMs idle
// when N is small and D large). The fitness terms are formed in parallel, the
// ordered sum by one thread per particle; pbest rows are written by all
// threads. Step 5 as in the fused one-particle-per-thread step: block argmin,
// candidate list, the last block gathers gbest.
// ---------------------------------------------------------------------------
constexpr int kTileItems = 2048;     // P * D per block at most (32 KB of x' and terms)
constexpr int kTileMinD = 16;        // below this the one-particle-per-thread step is used
constexpr int kChunk64 = 1;          // items whose loads a thread issues together (more only costs occupancy: FP64-bound)

template <int FIT>
__global__ void __launch_bounds__(256) sync64_tile_kernel(const __grid_constant__ SwarmDev64 s,
                                                         const __grid_constant__ PaperBufs b, int P) {
    __shared__ double X[kTileItems];
    __shared__ double H[kTileItems];
    __shared__ PKey red[32];
    __shared__ int imp[32];
    __shared__ int s_last;
    pdl_wait();
    pdl_launch_next();
    const uint32_t t_prev = __ldcg(s.t_dev);
    const uint32_t t = t_prev + 1u;
    const int cur = (int)(t_prev & 1u), nxt = cur ^ 1;
    const int tid = threadIdx.x;
    const int D = s.D;
    const size_t Np = (size_t)s.Np;
    const int base = blockIdx.x * P;
    const int n = min(P, s.N - base);
    const int nD = n * D;
    const double* G = s.G + (size_t)cur * D;

    // a thread loads the rows of kChunk64 items before it computes any of them
    for (int e0 = tid; e0 < nD; e0 += kChunk64 * blockDim.x) {
        double xs[kChunk64], vs[kChunk64], ps[kChunk64];
#pragma unroll
        for (int c = 0; c < kChunk64; ++c) {
            const int e = e0 + c * blockDim.x;
            if (e < nD) {
                const int d = e / n, p = e - d * n;
                const size_t off = (size_t)d * Np + (size_t)(base + p);
                xs[c] = s.x[off];
                vs[c] = s.v[off];
                ps[c] = s.pb[off];
            }
        }
#pragma unroll
        for (int c = 0; c < kChunk64; ++c) {
            const int e = e0 + c * blockDim.x;
            if (e >= nD) break;
            const int d = e / n, p = e - d * n;
            const uint32_t i = (uint32_t)(base + p);
            const size_t off = (size_t)d * Np + i;
            const uint4 r = philox4x32_10(make_uint4((uint32_t)d, i, t, s.swarm), s.key0, s.key1);
            double xx = xs[c], vv = vs[c];
            move_one64(xx, vv, ps[c], G[d], r, s);
            s.x[off] = xx;
            s.v[off] = vv;
            X[d * P + p] = xx;
            if constexpr (!FitTerms64<FIT>::kNeedsNext && FIT != kSphere) H[d * P + p] = FitTerms64<FIT>::term(xx, 0.0);
        }
    }
    __syncthreads();
    if constexpr (FitTerms64<FIT>::kNeedsNext) {
        for (int e = tid; e < nD; e += blockDim.x) {
            const int d = e / n, p = e - d * n;
            if (d + 1 < D) H[d * P + p] = FitTerms64<FIT>::term(X[d * P + p], X[(d + 1) * P + p]);
        }
        __syncthreads();
    }
    PKey cand = key_none();
    bool nan = false;
    if (tid < n) {
        const uint32_t i = (uint32_t)(base + tid);
        const double f = FitTerms64<FIT>::sum(X, H, P, tid, D);
        nan = (f != f);
        const bool better = f < s.pf[i];
        imp[tid] = better ? 1 : 0;
        if (better) {
            s.pf[i] = f;
            const PKey c = Fp64::key(f, i);
            if (c.k <= Fp64::gk(s, cur)) cand = c;
        }
    }
    __syncthreads();
    for (int e = tid; e < nD; e += blockDim.x) {
        const int d = e / n, p = e - d * n;
        if (imp[p]) s.pb[(size_t)d * Np + (size_t)(base + p)] = X[d * P + p];
    }
    const PKey k = block_min_key(cand, red);
    if (tid == 0 && k.i != kNoIdx) push_candidate(b, k, s.status);
    if (__syncthreads_or(nan) && tid == 0) atomicOr(s.status, kStatusNaN);

    // the last block to finish closes the iteration
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(b.ticket, 1u) == gridDim.x - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const unsigned int nl = min(__ldcg(b.list_n), b.list_cap);
    PKey m = tid == 0 ? Fp64::load_gkey(s, cur) : key_none();
    for (unsigned int j = tid; j < nl; j += blockDim.x) {
        PKey c;
        c.k = __ldcg(&b.list[j].k);
        c.i = __ldcg(&b.list[j].i);
        c.pad = 0u;
        if (key_less(c, m)) m = c;
    }
    const PKey best = block_min_key(m, red);
    if (best.i < (uint32_t)s.N)
        for (int d = tid; d < D; d += blockDim.x)
            s.G[(size_t)nxt * D + d] = __ldcg(s.pb + (size_t)d * Np + best.i);
    __syncthreads();
    if (tid == 0) {
        Fp64::store_gkey(s, nxt, best);
        Fp64::store_gkey(s, cur, best);
        *b.list_n = 0u;
        *b.ticket = 0u;
        *s.t_dev = t;
    }
}

// Particles per tile of sync64_tile_kernel: a power of two, at most 32 and
// kTileItems / D, and small enough that the tiles cover the SMs twice over.
int tile_particles(int N, int D, int num_sms) {
    int P = 32;
    while (P > 1 && (P * D > kTileItems || (long long)N < 2ll * num_sms * P)) P >>= 1;
    return P;
}

#define CUPSO_DISPATCH_FIT32(fid, CALL)            \
    switch (fid) {                                 \
        case kSphere: { constexpr int F = kSphere; CALL; break; }         \
        case kRastrigin: { constexpr int F = kRastrigin; CALL; break; }   \
        case kAckley: { constexpr int F = kAckley; CALL; break; }         \
        case kRosenbrock: { constexpr int F = kRosenbrock; CALL; break; } \
        case kCubicMax: { constexpr int F = kCubicMax; CALL; break; }     \
        default: return cudaErrorInvalidValue;     \
    }

#define CUPSO_DISPATCH_FIT64(fid, CALL)            \
    switch (fid) {                                 \
        case kSphere: { constexpr int F = kSphere; CALL; break; }         \
        case kRosenbrock: { constexpr int F = kRosenbrock; CALL; break; } \
        case kCubicMax: { constexpr int F = kCubicMax; CALL; break; }     \
        default: return cudaErrorInvalidValue;     \
    }

size_t al256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

size_t paper_bufs_bytes(int Np, int list_cap) {
    const size_t nb = (size_t)paper_blocks(Np);
    return al256(sizeof(PKey) * nb) + al256(sizeof(PKey) * (size_t)list_cap) + 256;
}

PaperBufs paper_bufs_at(void* base, int Np, int list_cap) {
    const size_t nb = (size_t)paper_blocks(Np);
    char* p = static_cast<char*>(base);
    PaperBufs b;
    b.aux = reinterpret_cast<PKey*>(p);
    p += al256(sizeof(PKey) * nb);
    b.list = reinterpret_cast<PKey*>(p);
    b.list_cap = (unsigned int)list_cap;
    p += al256(sizeof(PKey) * (size_t)list_cap);
    unsigned int* w = reinterpret_cast<unsigned int*>(p);
    b.lock = w;
    b.ticket = w + 1;
    b.list_n = w + 2;
    return b;
}

cudaError_t launch_queue_step(const SwarmDev& s, const PaperBufs& b, int fid, bool lock, cudaStream_t st) {
    const int nb = paper_blocks(s.N);
    if (lock) {
        CUPSO_DISPATCH_FIT32(fid, return launch_pdl(paper_step_kernel<Fp32, F, kAggQueueLock>, dim3(nb),
                                                    dim3(kPaperBlock), 0, st, s, b));
    }
    cudaError_t e = cudaSuccess;
    CUPSO_DISPATCH_FIT32(fid, e = launch_pdl(paper_step_kernel<Fp32, F, kAggQueue>, dim3(nb), dim3(kPaperBlock), 0, st,
                                             s, b));
    if (e != cudaSuccess) return e;
    return launch_pdl(paper_finish_kernel<Fp32, kAggQueue, true>, dim3(1), dim3(1024), 0, st, s, b, nb);
}

bool fp64_fitness_supported(int fid) { return fid == kSphere || fid == kRosenbrock || fid == kCubicMax; }

cudaError_t launch_init64(const SwarmDev64& s, const PaperBufs& b, int fid, cudaStream_t st) {
    const int nb = paper_blocks(s.N);
    CUPSO_DISPATCH_FIT64(fid, (init64_kernel<F><<<nb, kPaperBlock, 0, st>>>(s, b)));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    paper_finish_kernel<Fp64, kAggReduce, false><<<1, 1024, 0, st>>>(s, b, nb);
    return cudaGetLastError();
}

cudaError_t launch_recompute64(const SwarmDev64& s, const PaperBufs& b, cudaStream_t st) {
    const int nb = paper_blocks(s.N);
    pbest_min64_kernel<<<nb, kPaperBlock, 0, st>>>(s, b);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    paper_finish_kernel<Fp64, kAggReduce, false><<<1, 1024, 0, st>>>(s, b, nb);
    return cudaGetLastError();
}

cudaError_t launch_step64(const SwarmDev64& s, const PaperBufs& b, int fid, int agg, int num_sms, cudaStream_t st) {
    const int nb = paper_blocks(s.N);
    if ((unsigned int)nb > b.list_cap) return cudaErrorInvalidConfiguration;
    if (agg == kAggSyncList && s.D >= kTileMinD && s.D <= kTileItems) {
        const int P = tile_particles(s.N, s.D, num_sms);
        const int tiles = (s.N + P - 1) / P;
        if ((unsigned int)tiles > b.list_cap) return cudaErrorInvalidConfiguration;
        const int threads = P * s.D >= 256 ? 256 : (P * s.D + 31) / 32 * 32;
        CUPSO_DISPATCH_FIT64(fid, return launch_pdl(sync64_tile_kernel<F>, dim3(tiles), dim3(threads), 0, st, s, b, P));
    }
    const dim3 g1(nb), b1(kPaperBlock), g2(1), b2(1024);
    cudaError_t e = cudaSuccess;
    switch (agg) {
        case kAggReduce:
            CUPSO_DISPATCH_FIT64(fid, e = launch_pdl(paper_step_kernel<Fp64, F, kAggReduce>, g1, b1, 0, st, s, b));
            if (e != cudaSuccess) return e;
            return launch_pdl(paper_finish_kernel<Fp64, kAggReduce, true>, g2, b2, 0, st, s, b, nb);
        case kAggReduceUnrolled:
            CUPSO_DISPATCH_FIT64(fid, e = launch_pdl(paper_step_kernel<Fp64, F, kAggReduceUnrolled>, g1, b1, 0, st, s, b));
            if (e != cudaSuccess) return e;
            return launch_pdl(paper_finish_kernel<Fp64, kAggReduceUnrolled, true>, g2, b2, 0, st, s, b, nb);
        case kAggQueue:
            CUPSO_DISPATCH_FIT64(fid, e = launch_pdl(paper_step_kernel<Fp64, F, kAggQueue>, g1, b1, 0, st, s, b));
            if (e != cudaSuccess) return e;
            return launch_pdl(paper_finish_kernel<Fp64, kAggQueue, true>, g2, b2, 0, st, s, b, nb);
        case kAggQueueLock:
            CUPSO_DISPATCH_FIT64(fid, return launch_pdl(paper_step_kernel<Fp64, F, kAggQueueLock>, g1, b1, 0, st, s, b));
        case kAggSyncList:
            CUPSO_DISPATCH_FIT64(fid, return launch_pdl(paper_step_kernel<Fp64, F, kAggSyncList>, g1, b1, 0, st, s, b));
        default:
            return cudaErrorInvalidValue;
    }
}

namespace {

// Dynamic shared memory that a CTA of the on-chip kernel may take: the device's limit less
// room for the static shared arrays.
int max_onchip64_smem() {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return 0;
    return v - 1024;
}

int threads_for(int P, int D) {
    const long long work = (long long)P * D;
    int th = (int)((work + 31) / 32 * 32);
    return th < 32 ? 32 : (th > kOnchip64Threads ? kOnchip64Threads : th);
}

// The same limits whatever the swarm: they belong to the kernel, which swarms of other sizes
// run from other host threads.
template <int FIT>
cudaError_t set_onchip64_attrs(int C) {
    cudaError_t e = cudaFuncSetAttribute(onchip64_kernel<FIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_onchip64_smem());
    if (e == cudaSuccess && C > 8)
        e = cudaFuncSetAttribute(onchip64_kernel<FIT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

cudaLaunchConfig_t onchip64_config(int C, int threads, size_t smem, cudaStream_t st, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C, 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

bool cluster64_schedulable(int N, int D, int C) {
    const Onchip64Layout L = onchip64_layout(N, D, C);
    if (set_onchip64_attrs<kSphere>(C) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = onchip64_config(C, threads_for(L.P, D), L.bytes, nullptr, attr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, onchip64_kernel<kSphere>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n > 0;
}

}  // namespace

// CTAs of the on-chip cluster for (N, D), or 0 if the swarm does not fit: the
// power of two that gives each CTA about 128 (particle, dimension) pairs (so
// the FP64 work of an iteration spreads over that many SMs), at least the
// smallest count whose shared memory fits, at most 16.
int onchip64_cluster(int N, int D) {
    const int limit = max_onchip64_smem();
    if (limit <= 0) return 0;
    const long long pd = (long long)N * D;
    int C = 1;
    while (C < kMaxCluster64 && pd > 128ll * C && C < N) C *= 2;
    while (C <= kMaxCluster64 && onchip64_layout(N, D, C).bytes > (size_t)limit) C *= 2;
    if (C > kMaxCluster64) return 0;
    const int C_min = C;
    while (C >= 1 && !cluster64_schedulable(N, D, C)) C /= 2;
    if (C < 1 || onchip64_layout(N, D, C).bytes > (size_t)limit) return 0;
    (void)C_min;
    return C;
}

bool onchip64_fits(int N, int D) { return onchip64_cluster(N, D) > 0; }

cudaError_t launch_onchip64(const SwarmDev64& s, int fid, int iters, cudaStream_t st) {
    const int C = onchip64_cluster(s.N, s.D);
    if (C <= 0) return cudaErrorInvalidConfiguration;
    const Onchip64Layout L = onchip64_layout(s.N, s.D, C);
    const int threads = threads_for(L.P, s.D);
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = onchip64_config(C, threads, L.bytes, st, attr);
    switch (fid) {
        case kSphere: {
            cudaError_t e = set_onchip64_attrs<kSphere>(C);
            return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, onchip64_kernel<kSphere>, s, iters);
        }
        case kRosenbrock: {
            cudaError_t e = set_onchip64_attrs<kRosenbrock>(C);
            return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, onchip64_kernel<kRosenbrock>, s, iters);
        }
        case kCubicMax: {
            cudaError_t e = set_onchip64_attrs<kCubicMax>(C);
            return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, onchip64_kernel<kCubicMax>, s, iters);
        }
        default:
            return cudaErrorInvalidValue;
    }
}

}  // namespace cupso
