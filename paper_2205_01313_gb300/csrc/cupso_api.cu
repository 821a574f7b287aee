// cupso_api.cu -- the C ABI declared in include/cupso.h.
//
// Host-side control only (Sec. 2.2 splits PSO into host control and device
// work): argument checks, one device arena per swarm, stream and CUDA-graph
// management, and the launch of the kernels (kernels_*.cu). A handle holds
// either a single-precision swarm or a double-precision one (the paper's
// precision, kernels_paper.cu). Every step of the iteration runs on the GPU.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/cupso.h"
#include "cupso_device.cuh"
#include "cupso_internal.h"
#include "lsq_internal.h"
#include "paper_kernels.h"
#include "resident.h"
#include "tiled_kernels.h"

using namespace cupso;

namespace {

thread_local char g_last_error[512] = "";

int fail(int code, const char* fmt, const char* detail = "") {
    std::snprintf(g_last_error, sizeof(g_last_error), fmt, detail);
    return code;
}

int cuda_fail(cudaError_t e, const char* where) {
    std::snprintf(g_last_error, sizeof(g_last_error), "%s: %s", where, cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? CUPSO_ERR_OOM : CUPSO_ERR_CUDA;
}

#define CUPSO_CUDA(call, where)                      \
    do {                                             \
        cudaError_t e_ = (call);                     \
        if (e_ != cudaSuccess) return cuda_fail(e_, where); \
    } while (0)

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

}  // namespace

void cupso::set_last_error(const char* msg) { std::snprintf(g_last_error, sizeof(g_last_error), "%s", msg); }

struct cupso_swarm {
    SwarmDev dev{};
    bool fp64 = false;              // a double-precision swarm: dev64 instead of dev
    SwarmDev64 dev64{};
    PaperBufs pbufs{};              // one-particle-per-thread designs (QUEUE, QUEUE_LOCK, FP64 modes)
    ResidentBufs rbufs{};           // the resident SYNC kernel's exchange (slots null: it does not fit)
    Sync64Bufs s64bufs{};           // the FP64 one-launch steps' exchange (slots null: D too large)
    bool onchip64 = false;          // the FP64 swarm fits the on-chip kernel
    int N = 0, D = 0, Np = 0, fid = 0;
    uint64_t seed = 0;
    uint32_t swarm = 0;
    void* arena = nullptr;
    size_t arena_bytes = 0;
    cudaStream_t own = nullptr;     // the handle's non-blocking stream
    cudaStream_t stream = nullptr;  // where work is queued (own or the caller's)
    cudaStream_t capture = nullptr; // graphs are captured here, launched on `stream`
    int device = 0, num_sms = 1;
    int mode = CUPSO_MODE_AUTO;
    int graph_chunk = 16;
    cudaGraphExec_t graph = nullptr;
    int graph_mode = -1, graph_len = 0;
    uint32_t t_host = 0;
    int hold_lock = 0;
    int stall_barrier = 0;          // test hook: the cooperative multi-iteration launches wait for one CTA more
    int iters_per_launch = 0;       // panel SYNC step: iterations per launch, 0 = automatic
    int lsq_rescore = 0;            // CUPSO_OPT_LSQ_RESCORE: 0 float-float, 1 FP64
    int grid_override = 0;
    int onchip_cluster = 0;
    int sync_kernel = 0;            // CUPSO_SYNC_KERNEL_*
    int ppt_option = 0;             // particles per thread of the pipelined kernel, 0 = automatic
    bool pipelined_ok = false;      // shared-memory limit raised for the pipelined kernels
    bool panel_ok = false;          // the same for the panel kernels (D % 8 == 0)
    int panel = 0;                  // x, v, pb in the panel layout of this width (kernels_panel.cu), 0: dimension-major
    bool lazy_pending = false;      // the pipelined step may have left pbest rows unwritten
    // least-squares fitness (fitness_id CUPSO_LSQ), set by cupso_set_lsq
    struct Lsq {
        const float* A = nullptr;   // [M][D], borrowed
        const float* b = nullptr;   // [M], borrowed
        int M = 0, precision = 0;
        LsqTcState tc;              // BF16 / FP8 operands and plan
        void* buf = nullptr;        // f [Np] | cand [lists*16 + 16 + ticket] | partial [16 * chunks] | g64 | exact_ws
        void* exact_ws = nullptr;   // FP32 / FP64 fitness: residual workspace
        size_t ws_most = 0;         // and its limit
        float* f = nullptr;
        unsigned long long* cand = nullptr;
        double* partial = nullptr;
        double* g64 = nullptr;
        unsigned int* flags = nullptr;   // [Np / 4]: improved this iteration (one byte per particle)
        int chunks = 32;                 // pieces of the FP64 rescoring per candidate (set with A)
        LsqGram gram;                    // A^T A etc. for the Gram-form rescoring when D <= M
        void* gram_buf = nullptr;
        bool time_fitness = false;       // CUPSO_OPT_TIME_FITNESS
        // the residual offsets of a new gbest are computed on a side stream while the
        // next move runs (fork and join events, also inside captured graphs)
        cudaStream_t side = nullptr;
        cudaEvent_t fork = nullptr, join = nullptr;
        std::vector<cudaEvent_t> ev;     // pairs around the fitness phase
        double fitness_ms_sum = 0.0;
        int fitness_timed = 0;
    };
    Lsq* lsq = nullptr;
    // staged rows of get_state / set_state (allocated on first use, at most
    // kStageBytes unless one particle's row is larger)
    bool no_staging = false;        // test hook: there is no device memory for it
    void* stage = nullptr;
    size_t stage_bytes = 0;
    std::vector<char> head_copy;    // host copy of a gbest read: the arena's head and gbest_pos
    // result slots of cupso_gbest_post / _wait (allocated on first use): a
    // device record and a pinned host copy per slot, the copy stream, and per
    // slot the events of the snapshot and of its copy
    char* rec_dev = nullptr;
    char* rec_host = nullptr;
    cudaStream_t rec_stream = nullptr;
    cudaEvent_t rec_ev[2] = {nullptr, nullptr};
    cudaEvent_t rec_done[2] = {nullptr, nullptr};
    bool rec_posted[2] = {false, false};
};

namespace {

int resolved_mode(const cupso_swarm* h) {
    if (h->mode != CUPSO_MODE_AUTO) return h->mode;
    if (h->fp64) return h->onchip64 ? CUPSO_MODE_ONCHIP : CUPSO_MODE_SYNC;
    return h->onchip_cluster > 0 ? CUPSO_MODE_ONCHIP : CUPSO_MODE_SYNC;
}

// Particles per tile when the tiled SYNC kernel runs, else 0. AUTO takes it
// for D >= 8 up to the crossover measured on a GB300 against the pipelined
// kernel (which runs over d inside each thread and needs many particles per
// SM to hide its row latency), tiled and pipelined in us per iteration from captured graphs and,
// where the pipelined one costs about 2 us more and the tiled one 1, from launches one by one:
// sphere 93703 x 30 17.4 and 17.1, 16.6 and 17.5; 110000 x 12 10.7 and 10.2, 11.0 and 12.3; 80000 x
// 80 32.7 and 34.4, 33.1 and 36.8; 60000 x 201 75 and 64. Rosenbrock, whose terms need the next
// dimension's value too, 80000 x 30 18.7 and 17.4, 18.0 and 18.6; 60000 x 63 26.6 and 25.5, 27 and 28.
int sync_tile(const cupso_swarm* h) {
    if (h->fp64) return 0;
    if (h->sync_kernel == CUPSO_SYNC_KERNEL_TILED) return tiled_particles(h->N, h->D, h->num_sms);
    if (h->sync_kernel != CUPSO_SYNC_KERNEL_AUTO || h->D < 8) return 0;
    if (h->panel_ok && h->D % 8 == 0) {
        // against the panel kernel running each cupso_step call in one cooperative
        // launch (sweep on one GB300, N = 4096 .. 262144, D = 16 .. 256, Rosenbrock and
        // Rastrigin, steps of 96 iterations): the tiled kernel is the faster one only
        // below 2^17 particle-dimensions
        const long long pd = (long long)h->N * h->D;
        return pd < (1ll << 17) ? tiled_particles(h->N, h->D, h->num_sms) : 0;
    }
    const int D = h->D;
    const long long per_sm = h->fid == CUPSO_ROSENBROCK ? (D <= 32 ? 560 : D <= 64 ? 390 : 224)
                                                        : (D <= 16 ? 780 : D <= 64 ? 680 : D <= 128 ? 560 : 330);
    if ((long long)h->N > per_sm * h->num_sms) return 0;
    return tiled_particles(h->N, h->D, h->num_sms);
}

// Blocks of the tiled kernel: one wave of resident blocks (or the grid option).
int tiled_grid(const cupso_swarm* h, int P) {
    if (h->grid_override > 0) return h->grid_override;
    return h->num_sms * tiled_blocks_per_sm(h->fid, P, h->D);
}

// Ring depth of the pipelined SYNC kernel, or 0 for the register kernel.
int sync_stages(const cupso_swarm* h) {
    int want = 0;
    switch (h->sync_kernel) {
        case CUPSO_SYNC_KERNEL_REGISTER: return 0;
        case CUPSO_SYNC_KERNEL_PIPELINED3: want = 3; break;
        case CUPSO_SYNC_KERNEL_PIPELINED4: want = 4; break;
        default:  // deepest ring the dimension count allows
            if (h->pipelined_ok && pipelined_supported(4, h->D)) return 4;
            want = 3;
            break;
    }
    return (h->pipelined_ok && pipelined_supported(want, h->D)) ? want : 0;
}

// The panel SYNC kernel (the state in the panel layout) when it runs: its
// panel width and ring depth (5 panels where the panels allow, else 3); width
// 0 when the dimension-major kernels run. AUTO takes the panel kernel for
// D % 8 == 0 wherever the tiled kernel is not the faster one; 16-dimension
// panels for D >= 128 or up to 8192 particles, 8-dimension panels otherwise
// (Rosenbrock 2^20 x 64: a tie, 0.239 ms per iteration either way).
struct PanelCfg {
    int width = 0, stages = 0;
};
PanelCfg panel_cfg(const cupso_swarm* h) {
    PanelCfg c;
    if (h->fp64 || !h->panel_ok || h->fid == CUPSO_LSQ) return c;
    int widths[2] = {0, 0};
    switch (h->sync_kernel) {
        case CUPSO_SYNC_KERNEL_PANEL8: widths[0] = 8; break;
        case CUPSO_SYNC_KERNEL_PANEL16: widths[0] = 16; break;
        case CUPSO_SYNC_KERNEL_AUTO:
            if (sync_tile(h)) return c;
            // 16-dimension panels (units of 8 particles) for long particles (D >= 128)
            // and for swarms of up to 8192 particles, 8 otherwise (the same sweep; where
            // the other width wins, by at most 10 %, the units divide unevenly over
            // the warps)
            if (h->D % 16 == 0 && (h->D >= 128 || h->N <= 8192)) widths[0] = 16;
            widths[1] = 8;
            break;
        default: return c;
    }
    for (int w : widths) {
        if (!w) continue;
        for (int st : {5, 3})
            if (panel_supported(w, st, h->D)) {
                c.width = w;
                c.stages = st;
                return c;
            }
    }
    return c;
}

// Particles per thread of the pipelined kernel: fewer make more and shorter units, more
// share the Philox calls' latency and their copies' instructions. Sweep on one GB300 (us
// per iteration with 1, 2 and 4): 2000 x 7 6.9, 7.1, 7.8; 35000 x 65 22.8, 20.2, 24.5; 80000
// x 127 66, 53, 56; 100000 x 127 74, 65, 57; 300000 x 63 93, 87, 83; 10^6 x 7 46, 32, 28.
int sync_ppt(const cupso_swarm* h) {
    if (h->ppt_option) return h->ppt_option;
    if ((long long)h->Np >= 640ll * h->num_sms) return 4;
    if ((long long)h->Np >= 128ll * h->num_sms) return 2;
    return 1;
}

// CTAs of a kernel whose warps take units, the first ones CTA by CTA: the same number on
// every SM, at most `per_sm`, as few as hold a warp per unit. (With the units' own number
// of CTAs some SMs had two and most one: 40000 x 32 in panels 11.1 us an iteration, now
// 8.5; 20000 x 128 15.2 and 12.9.)
int even_grid(const cupso_swarm* h, int units, int per_sm) {
    const int warps = kBlock / 32;
    if (h->grid_override > 0) return std::min(h->grid_override, (units + warps - 1) / warps);
    const int want = (int)(((long long)units + (long long)warps * h->num_sms - 1) / ((long long)warps * h->num_sms));
    return std::min(h->num_sms * std::min(per_sm, want), units);
}

int sync_grid(const cupso_swarm* h) {
    const PanelCfg pc = panel_cfg(h);
    if (pc.width) {
        // persistent: warps pull units of 128 / width particles from a counter
        const int units = h->Np / (128 / pc.width);
        return even_grid(h, units, panel_blocks_per_sm(pc.width, pc.stages, h->fid, h->D));
    }
    const int stages = sync_stages(h);
    if (stages) {
        // persistent: warps pull units of 32 * ppt particles from a counter
        const int ppt = sync_ppt(h);
        const int units = h->Np / (32 * ppt);
        // of a few dozen units the CTAs' last one waits for the fewer, the better: 846 x 5 8.2 us
        // in 28 CTAs and 6.2 in 4
        if (3 * units <= h->num_sms && h->grid_override == 0) return (units + kBlock / 32 - 1) / (kBlock / 32);
        return even_grid(h, units, pipelined_blocks_per_sm(stages, h->fid, h->D, ppt));
    }
    const int ntiles = tiles_of(h->Np);
    int g = h->grid_override > 0 ? h->grid_override : h->num_sms * sync_blocks_per_sm(h->fid, h->D);
    return g < ntiles ? g : ntiles;
}

// Iterations per launch of the panel SYNC step: the option, else all of a
// cupso_step call up to kPanelMaxIters.
int panel_iters_per_launch(const cupso_swarm* h) {
    return h->iters_per_launch > 0 ? h->iters_per_launch : kPanelMaxIters;
}

// Whether an iteration of a swarm that waits for all CTAs ends well within the wait limit: a
// millisecond, and 0.12 ns per particle-dimension (double precision in memory takes 0.02).
// A shorter limit is meant for other waits; the kernels of single iterations have none.
bool limit_ample(const cupso_swarm* h) {
    return h->dev.wait_limit_ns >= 1000000ll + (long long)h->N * h->D / 8;
}

// The iterations of a call from which they run in the resident kernel
// (kernels_resident.cu), 0: never. Synchronous swarm, AUTO kernel choice, default grid,
// several iterations per launch allowed.
//  * SYNC: loading and storing the registers costs as much as one or two iterations
//    of the kernels that keep the state in memory; measured per iteration against
//    them at 2, 3 and 4 iterations: 1024 x 32 6.4, 4.6, 4.2 us against 5.4, 5.3, 5.2;
//    20000 x 48 11.2, 8.6, 7.2 against 11.3, 10.6, 10.2; one more where the state is
//    in panels, whose loads are strided here.
//  * AUTO, where the swarm also fits one cluster's shared memory: an iteration takes
//    1.0 to 1.5 us (2.2 while gbest improves) whatever the swarm, against 1.1 us (32 x
//    1) to 4.7 (2048 x 32) on the cluster, whose launch costs less: 2048 x 32 at 4
//    iterations 4.0 against 6.7 us, 1000 x 2 3.1 against 2.8; 300 x 8 (Rosenbrock)
//    at 100 1.95 against 1.68, at 1000 1.51 against 1.58. The cluster's time grows with D
//    and the line by N leaves that out: below 1000 particles long ones stay on the cluster
//    where registers would be faster (64 x 30 in calls of 100 1.2 to 2.5 against 2.3 to 3.1,
//    512 x 16 1.1 to 1.4 against 1.7 to 2.2, but Rosenbrock there 2.2 against 2.0).
int resident_from(const cupso_swarm* h, int mode) {
    if (!h->rbufs.slots || h->sync_kernel != CUPSO_SYNC_KERNEL_AUTO || h->grid_override != 0 || h->iters_per_launch == 1 ||
        !limit_ample(h))
        return 0;
    if (mode == CUPSO_MODE_SYNC) return h->panel ? 4 : 3;
    if (mode != CUPSO_MODE_ONCHIP || h->mode != CUPSO_MODE_AUTO) return 0;
    return h->N >= 1000 ? 5 : (long long)h->N * h->D >= 1000 ? 300 : 0;
}

// The iterations of a call from which those of an FP64 swarm run in one cooperative
// launch (kernels_sync64.cu), 0: never. Its start and end cost as much as two to five iterations of the
// kernels with a launch per iteration (SYNC; us per iteration at 2 and 10: 32 x 1 5.6
// and 2.3 against 4.6 and 4.5, 131072 x 1 10.7 and 6.3 against 9.2, 30000 x 10 at 10
// 11.9 against 15.8), and more than those of the cluster (AUTO where the swarm
// fits one: 512 x 1 at 10 and 200 2.4 and 1.55 against 2.3 and 1.8, 8192 x 1 2.6 and
// 1.6 against 4.7 and 4.2).
int sync64_from(const cupso_swarm* h, int mode) {
    if (!h->s64bufs.slots) return 0;
    if (mode == CUPSO_MODE_PERSISTENT) return 1;
    if (h->iters_per_launch == 1 || !limit_ample(h)) return 0;
    const long long pd = (long long)h->N * h->D;
    if (mode == CUPSO_MODE_SYNC) return pd >= (1 << 18) ? 5 : 3;
    return mode == CUPSO_MODE_ONCHIP && h->mode == CUPSO_MODE_AUTO ? (pd >= 2000 ? 10 : 50) : 0;
}

// The same for either precision.
int one_launch_from(const cupso_swarm* h, int mode) { return h->fp64 ? sync64_from(h, mode) : resident_from(h, mode); }

// CTAs of a multi-iteration panel launch: the SYNC grid, at most what the SMs
// hold at once (a cooperative launch).
int panel_persist_grid(const cupso_swarm* h, const PanelCfg& pc) {
    const int resident = h->num_sms * panel_blocks_per_sm(pc.width, pc.stages, h->fid, h->D);
    return std::min(sync_grid(h), resident);
}

// ASYNC uses small CTAs when the swarm is small, so that it still spreads
// over many independently running CTAs.
int async_block(const cupso_swarm* h) {
    return (h->Np / kTile >= 2 * h->num_sms) ? kBlock : 32;
}

// Particles per tile of the tiled asynchronous kernel (0: the streaming one),
// tiles up to about 896 particles per SM (224 with narrow tiles and a cheap fitness),
// else the streaming layout, which large swarms fill.
int async_tile(const cupso_swarm* h) {
    if (h->fp64 || h->D < 2) return 0;
    const bool has_cos = h->fid == CUPSO_RASTRIGIN || h->fid == CUPSO_ACKLEY;
    const long long per_sm = (has_cos || h->D <= 64) ? 896 : 224;
    if ((long long)h->N > per_sm * h->num_sms) return 0;
    return tiled_particles(h->N, h->D, h->num_sms);
}

int async_grid(const cupso_swarm* h) {
    if (const int P = async_tile(h)) {
        const int tiles = (h->N + P - 1) / P;
        const int g = h->grid_override > 0 ? h->grid_override : h->num_sms * async_tiled_blocks_per_sm(P, h->D);
        return g < tiles ? g : tiles;
    }
    const int tile = async_block(h) * kPerThread;
    const int ntiles = (h->Np + tile - 1) / tile;
    const int per_sm = async_blocks_per_sm(h->fid, h->D) * (kBlock / async_block(h));
    int g = h->grid_override > 0 ? h->grid_override : h->num_sms * per_sm;
    return g < ntiles ? g : ntiles;
}

void drop_graph(cupso_swarm* h) {
    if (h->graph) cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
    h->graph_mode = -1;
    h->graph_len = 0;
}

constexpr int kModeLsq = 100;   // internal: one least-squares iteration

// The tensor-core precisions: approximate fitness, FP64-verified gbest.
bool lsq_approx(int precision) { return precision == CUPSO_LSQ_BF16 || precision == CUPSO_LSQ_FP8; }

cudaError_t launch_lsq_iteration(cupso_swarm* h, cudaStream_t st) {
    cupso_swarm::Lsq& L = *h->lsq;
    const int grid = h->num_sms * 8;   // grid-stride over (particle group, dimension) items
    if (!lsq_approx(L.precision)) {
        cudaError_t e = lsq_launch_move(h->dev, grid, st);
        if (e == cudaSuccess)
            e = lsq_exact_launch(h->dev.x, h->Np, h->N, h->D, L.A, L.b, L.M, L.precision == CUPSO_LSQ_FP64, L.f,
                                 L.exact_ws, L.ws_most, h->num_sms, st);
        if (e != cudaSuccess) return e;
        return lsq_launch_select_exact(h->dev, L.f, L.flags, grid, st);
    }
    // The residual offsets of the gbest this iteration moves towards (recomputed
    // only if the last acceptance moved it) run beside the move, which is
    // bound by HBM; the product, which adds them, waits for both. The move
    // writes the tensor-core operand too; the fitness is then the product alone.
    cudaError_t e = cudaEventRecord(L.fork, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(L.side, L.fork, 0);
    if (e == cudaSuccess) e = lsq_launch_offsets(h->dev, L.A, L.b, L.M, L.tc.roff, L.tc.roff_stale, h->num_sms, L.side);
    if (e == cudaSuccess) e = cudaEventRecord(L.join, L.side);
    if (e == cudaSuccess)
        e = lsq_launch_move_q(h->dev, L.tc.tmMove, L.tc.Xq, L.tc.Kp, L.tc.fp8, L.tc.sx, h->num_sms, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, L.join, 0);
    if (e != cudaSuccess) return e;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (L.time_fitness) {
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        cudaEventRecord(e0, st);
    }
    // the product leaves partial sums; the selection kernel adds them
    if (lsq_eval_tc_partials(&L.tc, st) != CUPSO_OK) return cudaErrorLaunchFailure;
    if (L.time_fitness) {
        cudaEventRecord(e1, st);
        L.ev.push_back(e0);
        L.ev.push_back(e1);
    }
    // offsets for the gbest this iteration accepts: at the start of the next one
    return lsq_launch_gbest_approx(h->dev, nullptr, L.tc.part, lsq_tc_partials(L.tc.plan), 0, true, L.A, L.b, L.M,
                                   L.cand, L.partial, L.chunks, L.g64, reinterpret_cast<unsigned int*>(h->dev.pflag),
                                   grid, L.gram, nullptr, L.tc.roff_stale, h->num_sms, st);
}

// gbest of an approximate-fitness swarm from scratch, with `fit` (device, [Np])
// as every particle's approximate fitness: the 16 lowest are rescored
// and the best becomes gbest (and the reference point of the tensor-core
// fitness, whose offsets are recomputed). t_dev ends at t.
cudaError_t lsq_reset_gbest(cupso_swarm* h, const float* fit, uint32_t t, cudaStream_t st) {
    cupso_swarm::Lsq& L = *h->lsq;
    const double inf = INFINITY;
    cudaError_t e = cudaMemcpyAsync(L.g64, &inf, sizeof(double), cudaMemcpyHostToDevice, st);
    // the accept kernel advances t: start one below and let it land on t
    if (e == cudaSuccess) e = lsq_launch_set_t(h->dev, t - 1u, st);
    if (e == cudaSuccess)
        e = lsq_launch_gbest_approx(h->dev, fit, nullptr, 0, 1, true, L.A, L.b, L.M, L.cand, L.partial, L.chunks,
                                    L.g64, reinterpret_cast<unsigned int*>(h->dev.pflag), h->num_sms * 8, L.gram,
                                    L.tc.roff, L.tc.roff_stale, h->num_sms, st);
    return e;
}

cudaError_t launch_one64(cupso_swarm* h, int mode, cudaStream_t st) {
    switch (mode) {
        case CUPSO_MODE_SYNC: return launch_step64(h->dev64, h->pbufs, h->fid, kAggSyncList, h->num_sms, st);
        case CUPSO_MODE_TREE: return launch_step64(h->dev64, h->pbufs, h->fid, kAggReduce, h->num_sms, st);
        case CUPSO_MODE_TREE_UNROLLED: return launch_step64(h->dev64, h->pbufs, h->fid, kAggReduceUnrolled, h->num_sms, st);
        case CUPSO_MODE_QUEUE: return launch_step64(h->dev64, h->pbufs, h->fid, kAggQueue, h->num_sms, st);
        case CUPSO_MODE_QUEUE_LOCK: return launch_step64(h->dev64, h->pbufs, h->fid, kAggQueueLock, h->num_sms, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_one(cupso_swarm* h, int mode, cudaStream_t st) {
    if (h->fp64) return launch_one64(h, mode, st);
    switch (mode) {
        case kModeLsq: return launch_lsq_iteration(h, st);
        case CUPSO_MODE_SYNC: {
            const PanelCfg pc = panel_cfg(h);
            if (pc.width) return launch_sync_panel(h->dev, h->fid, pc.width, pc.stages, sync_grid(h), 1, false, st);
            if (const int P = sync_tile(h))
                return launch_sync_tiled(h->dev, h->fid, P, tiled_grid(h, P), st);
            const int stages = sync_stages(h);
            if (stages) return launch_sync_pipelined(h->dev, h->fid, stages, sync_ppt(h), sync_grid(h), st);
            return launch_sync_step(h->dev, h->fid, sync_grid(h), st);
        }
        case CUPSO_MODE_TREE: return launch_tree_step(h->dev, h->fid, false, st);
        case CUPSO_MODE_TREE_UNROLLED: return launch_tree_step(h->dev, h->fid, true, st);
        case CUPSO_MODE_QUEUE: return launch_queue_step(h->dev, h->pbufs, h->fid, false, st);
        case CUPSO_MODE_QUEUE_LOCK: return launch_queue_step(h->dev, h->pbufs, h->fid, true, st);
        default: return cudaErrorInvalidValue;
    }
}

// Before any kernel that reads pbest_pos directly: write back the rows the
// pipelined step left pending.
int ensure_materialized(cupso_swarm* h) {
    if (h->fp64 || !h->lazy_pending) return CUPSO_OK;
    cudaError_t e;
    if (h->panel) {
        const int grid = std::max(1, std::min(h->num_sms * 8, (h->Np + kBlock - 1) / kBlock));
        e = launch_materialize_panel(h->dev, h->panel, grid, h->stream);
    } else {
        const int grid = std::max(1, std::min(h->num_sms * 8, (h->Np / 4 + kBlock - 1) / kBlock));
        e = launch_materialize(h->dev, grid, h->stream);
    }
    if (e != cudaSuccess) return cuda_fail(e, "materialize launch");
    h->lazy_pending = false;
    return CUPSO_OK;
}

// Puts pos, v and pbest_pos in the layout the next kernel reads: the panel
// layout of width `want` (8 or 16) for the panel SYNC kernel, the
// dimension-major one (want 0) for every other kernel. Pending pbest rows are
// written back first; each array goes through a temporary copy (one array's
// size, freed again). Not for stream capture.
int ensure_layout(cupso_swarm* h, int want) {
    if (h->fp64 || h->panel == want) return CUPSO_OK;
    int rc = ensure_materialized(h);
    if (rc) return rc;
    drop_graph(h);
    const size_t bytes = sizeof(float) * (size_t)h->D * (size_t)h->Np;
    void* tmp = nullptr;
    CUPSO_CUDA(cudaMalloc(&tmp, bytes), "cudaMalloc (relayout)");
    float* arrays[3] = {h->dev.x, h->dev.v, h->dev.pb};
    const int grid = h->num_sms * 8;
    cudaError_t e = cudaSuccess;
    // at most two passes: out of the current panel width, into the wanted one
    const int passes[2][2] = {{h->panel, 0}, {want, 1}};
    for (const auto& ps : passes) {
        if (!ps[0]) continue;
        for (int a = 0; a < 3 && e == cudaSuccess; ++a) {
            e = launch_relayout(arrays[a], static_cast<float*>(tmp), h->D, h->Np, ps[0], ps[1] != 0, grid, h->stream);
            if (e == cudaSuccess) e = cudaMemcpyAsync(arrays[a], tmp, bytes, cudaMemcpyDeviceToDevice, h->stream);
        }
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    cudaFree(tmp);
    if (e != cudaSuccess) return cuda_fail(e, "relayout");
    h->panel = want;
    return CUPSO_OK;
}

// A graph of `len` iterations. The kernels read the iteration counter from
// device memory, so one captured graph serves every later chunk.
int ensure_graph(cupso_swarm* h, int mode, int len) {
    if (h->graph && h->graph_mode == mode && h->graph_len == len) return CUPSO_OK;
    drop_graph(h);
    if (!h->capture) CUPSO_CUDA(cudaStreamCreateWithFlags(&h->capture, cudaStreamNonBlocking), "cudaStreamCreate");
    CUPSO_CUDA(cudaStreamBeginCapture(h->capture, cudaStreamCaptureModeThreadLocal), "cudaStreamBeginCapture");
    cudaError_t le = cudaSuccess;
    for (int k = 0; k < len && le == cudaSuccess; ++k) le = launch_one(h, mode, h->capture);
    cudaGraph_t g = nullptr;
    cudaError_t ee = cudaStreamEndCapture(h->capture, &g);
    if (le != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return cuda_fail(le, "kernel launch during capture");
    }
    if (ee != cudaSuccess) return cuda_fail(ee, "cudaStreamEndCapture");
    cudaError_t ie = cudaGraphInstantiate(&h->graph, g, 0);
    cudaGraphDestroy(g);
    if (ie != cudaSuccess) {
        h->graph = nullptr;
        return cuda_fail(ie, "cudaGraphInstantiate");
    }
    h->graph_mode = mode;
    h->graph_len = len;
    return CUPSO_OK;
}

}  // namespace

int cupso::check_problem_args(int D, int N, const cupso_bounds* b, float w, float c1, float c2, int fid) {
    if (D < 1 || N < 1) return fail(CUPSO_ERR_INVALID_ARG, "D and N must be >= 1%s");
    if ((long long)N > (long long)0x7FFFFFFF - kPad) return fail(CUPSO_ERR_INVALID_ARG, "N too large%s");
    const long long Np = ((long long)N + kPad - 1) / kPad * kPad;
    if (Np * (long long)D >= (1ll << 31)) return fail(CUPSO_ERR_INVALID_ARG, "N * D must be < 2^31%s");
    if (!b) return fail(CUPSO_ERR_INVALID_ARG, "bounds is NULL%s");
    if (!std::isfinite(b->min_pos) || !std::isfinite(b->max_pos) || !std::isfinite(b->max_v))
        return fail(CUPSO_ERR_INVALID_ARG, "bounds must be finite%s");
    if (!(b->min_pos < b->max_pos)) return fail(CUPSO_ERR_INVALID_ARG, "min_pos must be < max_pos%s");
    if (!(b->max_v > 0.0f)) return fail(CUPSO_ERR_INVALID_ARG, "max_v must be > 0%s");
    if (!std::isfinite(w) || !std::isfinite(c1) || !std::isfinite(c2))
        return fail(CUPSO_ERR_INVALID_ARG, "w, c1, c2 must be finite%s");
    if (fid < CUPSO_SPHERE || fid > CUPSO_LSQ) return fail(CUPSO_ERR_INVALID_ARG, "unknown fitness_id%s");
    return CUPSO_OK;
}

namespace {
// What a gbest read needs stands together in the arena, so that one copy brings it: the
// keys of both parities, the counters and words with the sticky status, and from kHeadBytes
// gbest_pos of both parities.
constexpr size_t kHeadBytes = 128, kHeadStatus = 40, kHeadStatus64 = 36;
}

// The fast arithmetic path's constants and whether it gives the same bits:
// c * 2^-24 is exact unless it would be subnormal (checked by scaling back), and
// the min/max clamps need bounds that are not zero.
void cupso::set_fast_paths(SwarmDev* s) {
    s->c1s = std::ldexp(s->c1, -24);
    s->c2s = std::ldexp(s->c2, -24);
    s->fast_cr = (std::ldexp(s->c1s, 24) == s->c1 && std::ldexp(s->c2s, 24) == s->c2 &&
                  (s->c1 == 0.0f || std::fabs(s->c1s) >= FLT_MIN) && (s->c2 == 0.0f || std::fabs(s->c2s) >= FLT_MIN))
                     ? 1 : 0;
    s->fast_clamp = (s->lo != 0.0f && s->hi != 0.0f) ? 1 : 0;
}

namespace {

int create_swarm(int D, int N, const cupso_bounds* b, float w, float c1, float c2, int fid, uint64_t seed,
                 uint32_t swarm, cudaStream_t user_stream, cupso_handle* out) {
    if (!out) return fail(CUPSO_ERR_INVALID_ARG, "out is NULL%s");
    *out = nullptr;
    int rc = check_problem_args(D, N, b, w, c1, c2, fid);
    if (rc) return rc;
    cupso_swarm* h = new (std::nothrow) cupso_swarm();
    if (!h) return fail(CUPSO_ERR_OOM, "host allocation failed%s");
    h->N = N;
    h->D = D;
    h->Np = (N + kPad - 1) / kPad * kPad;
    h->fid = fid;
    h->seed = seed;
    h->swarm = swarm;
    auto bail = [&](int code) {
        cupso_destroy(h);
        return code;
    };
    cudaError_t e = cudaGetDevice(&h->device);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaGetDevice"));
    e = cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaDeviceGetAttribute"));
    e = cudaStreamCreateWithFlags(&h->own, cudaStreamNonBlocking);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaStreamCreate"));
    h->stream = user_stream ? user_stream : h->own;

    // One arena: x, v, pb [D][Np]; pf [Np]; words, G [2][D]; Grec [D]; aux; ...
    const size_t A = 256;
    const size_t plane = sizeof(float) * (size_t)D * (size_t)h->Np;
    const size_t ntiles = (size_t)tiles_of(h->Np);
    size_t off = 0;
    const size_t o_x = off; off = align_up(off + plane, A);
    const size_t o_v = off; off = align_up(off + plane, A);
    const size_t o_pb = off; off = align_up(off + plane, A);
    const size_t o_pf = off; off = align_up(off + sizeof(float) * (size_t)h->Np, A);
    const size_t o_words = off; off += kHeadBytes;
    const size_t o_G = off; off = align_up(off + sizeof(float) * 2 * (size_t)D, A);
    const size_t o_Grec = off; off = align_up(off + sizeof(float) * (size_t)D, A);
    const size_t o_aux = off; off = align_up(off + sizeof(unsigned long long) * ntiles, A);
    const size_t o_flag = off; off = align_up(off + (size_t)h->Np, A);
    const int list_cap = paper_blocks(h->Np);      // one candidate per block of the queue designs
    const size_t o_paper = off; off = align_up(off + paper_bufs_bytes(h->Np, list_cap), A);
    const size_t res_bytes = fid == CUPSO_LSQ ? 0 : resident_bytes(N, D, h->num_sms);
    const size_t o_res = off; off = align_up(off + res_bytes, A);
    h->arena_bytes = off;
    e = cudaMalloc(&h->arena, h->arena_bytes);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaMalloc"));
    char* base = static_cast<char*>(h->arena);
    SwarmDev& s = h->dev;
    s.x = reinterpret_cast<float*>(base + o_x);
    s.v = reinterpret_cast<float*>(base + o_v);
    s.pb = reinterpret_cast<float*>(base + o_pb);
    s.pf = reinterpret_cast<float*>(base + o_pf);
    s.G = reinterpret_cast<float*>(base + o_G);
    s.Grec = reinterpret_cast<float*>(base + o_Grec);
    s.aux = reinterpret_cast<unsigned long long*>(base + o_aux);
    s.pflag = reinterpret_cast<unsigned char*>(base + o_flag);
    unsigned long long* w64 = reinterpret_cast<unsigned long long*>(base + o_words);
    s.gkey = w64;        // [2]
    s.claim = w64 + 2;
    s.reckey = w64 + 3;
    unsigned int* w32 = reinterpret_cast<unsigned int*>(w64 + 4);
    s.ticket = w32 + 0;
    s.t_dev = w32 + 1;
    s.status = w32 + 2;   // kHeadStatus
    s.lock = w32 + 3;
    s.seq = w32 + 4;
    s.work = w32 + 5;
    s.bar = reinterpret_cast<unsigned long long*>(w32 + 6);
    s.phase = w32 + 10;
    s.N = N;
    s.D = D;
    s.Np = h->Np;
    s.lo = b->min_pos;
    s.hi = b->max_pos;
    s.vmax = b->max_v;
    s.w = w;
    s.c1 = c1;
    s.c2 = c2;
    s.key0 = (uint32_t)(seed & 0xFFFFFFFFull);
    s.key1 = (uint32_t)(seed >> 32);
    philox_round_keys(s.key0, s.key1, s.rk0, s.rk1);
    s.swarm = swarm;
    s.wait_limit_ns = 2000000000ll;
    h->pbufs = paper_bufs_at(base + o_paper, h->Np, list_cap);
    set_fast_paths(&s);
    if (res_bytes && resident_fits(s, fid, h->num_sms) && prepare_resident(s, fid, h->num_sms) == cudaSuccess)
        h->rbufs = resident_bufs_at(base + o_res);

    int cl = 0, per = 0;
    h->onchip_cluster = (fid != CUPSO_LSQ && onchip_fits(N, D, &cl, &per)) ? cl : 0;
    h->pipelined_ok = prepare_pipelined(fid, fast_form(s, fid)) == cudaSuccess;
    h->panel_ok = fid != CUPSO_LSQ && panel_supported(8, 3, D) && prepare_panel(fid, fast_form(s, fid)) == cudaSuccess;
    cudaGetLastError();

    e = cudaMemsetAsync(base + o_words, 0, kHeadBytes, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s.pflag, 0, (size_t)h->Np, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s.gkey, 0xFF, 2 * sizeof(unsigned long long), h->stream);
    // the queue designs' storage and the words of the resident kernel's exchange behind it
    const size_t res_words = std::min<size_t>(res_bytes, 64);
    if (e == cudaSuccess) e = cudaMemsetAsync(base + o_paper, 0, o_res + res_words - o_paper, h->stream);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaMemsetAsync"));
    const int grid = std::min(tiles_of(h->Np), h->num_sms * 4);
    e = launch_init(s, fid, grid, h->stream);
    if (e != cudaSuccess) return bail(cuda_fail(e, "init launch"));
    e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return bail(cuda_fail(e, "init"));
    *out = h;
    return CUPSO_OK;
}

// k when c = 2^k exactly with |k| <= 512 (c r is then an exponent shift of a
// uniform in (2^-53, 1], which stays normal), else kNoExp.
int pow2_exponent(double c) {
    if (!(c > 0.0) || !std::isfinite(c)) return kNoExp;
    int e = 0;
    const double m = std::frexp(c, &e);   // c = m 2^e, m in [0.5, 1)
    if (m != 0.5) return kNoExp;
    const int k = e - 1;
    return (k >= -512 && k <= 512) ? k : kNoExp;
}

// A double-precision swarm: arena x, v, pb [D][Np], pf [Np], G [2][D]
// (binary64) behind the gbest keys and counters, and the working storage of the
// one-particle-per-thread kernels.
int create_swarm64(int D, int N, const cupso_bounds_f64* b, double w, double c1, double c2, int fid, uint64_t seed,
                   cupso_handle* out) {
    if (!out) return fail(CUPSO_ERR_INVALID_ARG, "out is NULL%s");
    *out = nullptr;
    if (D < 1 || N < 1) return fail(CUPSO_ERR_INVALID_ARG, "D and N must be >= 1%s");
    if ((long long)N > (long long)0x7FFFFFFF - kPad) return fail(CUPSO_ERR_INVALID_ARG, "N too large%s");
    const long long Npl = ((long long)N + kPad - 1) / kPad * kPad;
    if (Npl * (long long)D >= (1ll << 31)) return fail(CUPSO_ERR_INVALID_ARG, "N * D must be < 2^31%s");
    if (!b) return fail(CUPSO_ERR_INVALID_ARG, "bounds is NULL%s");
    if (!std::isfinite(b->min_pos) || !std::isfinite(b->max_pos) || !std::isfinite(b->max_v))
        return fail(CUPSO_ERR_INVALID_ARG, "bounds must be finite%s");
    if (!(b->min_pos < b->max_pos)) return fail(CUPSO_ERR_INVALID_ARG, "min_pos must be < max_pos%s");
    if (!(b->max_v > 0.0)) return fail(CUPSO_ERR_INVALID_ARG, "max_v must be > 0%s");
    if (!std::isfinite(w) || !std::isfinite(c1) || !std::isfinite(c2))
        return fail(CUPSO_ERR_INVALID_ARG, "w, c1, c2 must be finite%s");
    if (fid < CUPSO_SPHERE || fid > CUPSO_LSQ) return fail(CUPSO_ERR_INVALID_ARG, "unknown fitness_id%s");
    if (!fp64_fitness_supported(fid))
        return fail(CUPSO_ERR_UNSUPPORTED, "double precision supports sphere, Rosenbrock and the cubic%s");
    cupso_swarm* h = new (std::nothrow) cupso_swarm();
    if (!h) return fail(CUPSO_ERR_OOM, "host allocation failed%s");
    h->fp64 = true;
    h->N = N;
    h->D = D;
    h->Np = (int)Npl;
    h->fid = fid;
    h->seed = seed;
    auto bail = [&](int code) {
        cupso_destroy(h);
        return code;
    };
    cudaError_t e = cudaGetDevice(&h->device);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaGetDevice"));
    e = cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaDeviceGetAttribute"));
    e = cudaStreamCreateWithFlags(&h->own, cudaStreamNonBlocking);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaStreamCreate"));
    h->stream = h->own;

    const size_t A = 256;
    const size_t plane = sizeof(double) * (size_t)D * (size_t)h->Np;
    size_t off = 0;
    const size_t o_x = off; off = align_up(off + plane, A);
    const size_t o_v = off; off = align_up(off + plane, A);
    const size_t o_pb = off; off = align_up(off + plane, A);
    const size_t o_pf = off; off = align_up(off + sizeof(double) * (size_t)h->Np, A);
    const size_t o_key = off;
    const size_t o_words = off + 2 * sizeof(PKey); off += kHeadBytes;
    const size_t o_G = off; off = align_up(off + sizeof(double) * 2 * (size_t)D, A);
    const int list_cap = h->Np;   // the tiled step may run up to one block per particle
    const size_t o_paper = off; off = align_up(off + paper_bufs_bytes(h->Np, list_cap), A);
    const size_t s64_bytes = sync64_bytes(fid, N, D, h->num_sms);
    const size_t o_s64 = off; off = align_up(off + s64_bytes, A);
    h->arena_bytes = off;
    e = cudaMalloc(&h->arena, h->arena_bytes);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaMalloc"));
    char* base = static_cast<char*>(h->arena);
    SwarmDev64& s = h->dev64;
    s.x = reinterpret_cast<double*>(base + o_x);
    s.v = reinterpret_cast<double*>(base + o_v);
    s.pb = reinterpret_cast<double*>(base + o_pb);
    s.pf = reinterpret_cast<double*>(base + o_pf);
    s.G = reinterpret_cast<double*>(base + o_G);
    s.gkey = reinterpret_cast<PKey*>(base + o_key);
    unsigned int* w32 = reinterpret_cast<unsigned int*>(base + o_words);
    s.t_dev = w32 + 0;
    s.status = w32 + 1;   // kHeadStatus64
    s.N = N;
    s.D = D;
    s.Np = h->Np;
    s.lo = b->min_pos;
    s.hi = b->max_pos;
    s.vmax = b->max_v;
    s.w = w;
    s.c1 = c1;
    s.c2 = c2;
    s.key0 = (uint32_t)(seed & 0xFFFFFFFFull);
    s.key1 = (uint32_t)(seed >> 32);
    s.swarm = 0u;
    s.wait_limit_ns = 2000000000ll;
    s.w_one = (w == 1.0) ? 1 : 0;
    s.c1_exp = pow2_exponent(c1);
    s.c2_exp = pow2_exponent(c2);
    s.k_lo = order_key64(b->min_pos);
    s.k_hi = order_key64(b->max_pos);
    s.k_vlo = order_key64(-b->max_v);
    s.k_vhi = order_key64(b->max_v);
    s.k_inf = order_key64((double)INFINITY);
    s.vlo = -b->max_v;
    h->dev.wait_limit_ns = s.wait_limit_ns;
    h->dev.status = s.status;
    h->pbufs = paper_bufs_at(base + o_paper, h->Np, list_cap);
    if (s64_bytes && prepare_sync64(s, fid, h->num_sms) == cudaSuccess) h->s64bufs = sync64_bufs_at(base + o_s64);
    h->onchip_cluster = onchip64_cluster(N, D);
    h->onchip64 = h->onchip_cluster > 0;
    cudaGetLastError();

    e = cudaMemsetAsync(base + o_words, 0, 64, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s.gkey, 0xFF, 2 * sizeof(PKey), h->stream);
    // the queue designs' storage and the words of the one-launch steps' exchange behind it
    const size_t s64_words = std::min<size_t>(s64_bytes, 64);
    if (e == cudaSuccess) e = cudaMemsetAsync(base + o_paper, 0, o_s64 + s64_words - o_paper, h->stream);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaMemsetAsync"));
    e = launch_init64(s, h->pbufs, fid, h->stream);
    if (e != cudaSuccess) return bail(cuda_fail(e, "init launch"));
    e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return bail(cuda_fail(e, "init"));
    *out = h;
    return CUPSO_OK;
}

// The staging buffer for rows of `row` bytes, N of them: all at once, or chunks
// of up to kStageBytes; fewer when memory is short, down to one row. Kept as it is once
// there. Leaves h->stage null where not even one row fits: the rows then go through host
// memory (host_planes), which needs none on the device.
constexpr size_t kStageBytes = 32u << 20;
int ensure_stage(cupso_swarm* h, size_t row, size_t N) {
    if (h->stage || h->no_staging) return CUPSO_OK;
    size_t want = std::min(row * N, std::max(row, kStageBytes));
    cudaError_t e;
    while ((e = cudaMalloc(&h->stage, want)) == cudaErrorMemoryAllocation && want > row) {
        cudaGetLastError();
        want = std::max(row, want / 4);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        h->stage = nullptr;
        return e == cudaErrorMemoryAllocation ? CUPSO_OK : cuda_fail(e, "cudaMalloc (state staging)");
    }
    h->stage_bytes = want;
    return CUPSO_OK;
}

// Element (d, i) of a plane in `panel` layout (0: dimension-major).
size_t plane_at(size_t d, size_t i, size_t Np, size_t panel) {
    return panel ? ((d / panel) * Np + i) * panel + d % panel : d * Np + i;
}

template <typename T>
void unpack_plane(const cupso_swarm* h, const T* plane, int panel, T* out) {
    const size_t N = (size_t)h->N, D = (size_t)h->D, Np = (size_t)h->Np;
    for (size_t i = 0; i < N; ++i)
        for (size_t d = 0; d < D; ++d) out[i * D + d] = plane[plane_at(d, i, Np, (size_t)panel)];
}

// `count` bytes of host memory for whole planes.
int host_planes(std::vector<char>* mem, size_t count) {
    try {
        mem->resize(count);
    } catch (...) {
        return fail(CUPSO_ERR_OOM, "host allocation failed%s");
    }
    return CUPSO_OK;
}

// out[i][d], i < N, from a device array in `panel` layout; queued on the
// handle's stream (the caller waits).
template <typename T>
int download_rows(cupso_swarm* h, const T* src, int panel, T* out) {
    const size_t D = (size_t)h->D, row = sizeof(T) * D;
    if (D == 1) {   // one row either way
        CUPSO_CUDA(cudaMemcpyAsync(out, src, sizeof(T) * (size_t)h->N, cudaMemcpyDeviceToHost, h->stream), "cudaMemcpyAsync");
        return CUPSO_OK;
    }
    int rc = ensure_stage(h, row, (size_t)h->N);
    if (rc) return rc;
    if (!h->stage) {
        std::vector<char> mem;
        rc = host_planes(&mem, row * (size_t)h->Np);
        if (rc) return rc;
        CUPSO_CUDA(cudaMemcpyAsync(mem.data(), src, mem.size(), cudaMemcpyDeviceToHost, h->stream), "cudaMemcpyAsync");
        CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
        unpack_plane(h, reinterpret_cast<const T*>(mem.data()), panel, out);
        return CUPSO_OK;
    }
    const int per = (int)std::min<size_t>((size_t)h->N, h->stage_bytes / row);
    for (int i0 = 0; i0 < h->N; i0 += per) {
        const int n = std::min(per, h->N - i0);
        CUPSO_CUDA(launch_unpack_rows(src, static_cast<T*>(h->stage), h->D, h->Np, panel, i0, n, h->stream), "unpack launch");
        CUPSO_CUDA(cudaMemcpyAsync(out + (size_t)i0 * D, h->stage, row * (size_t)n, cudaMemcpyDeviceToHost, h->stream),
                   "cudaMemcpyAsync");
        if (n == h->N - i0) break;
    }
    return CUPSO_OK;
}

// The whole state to the host, waited for: `planes` = {x, v, pb}, which pf follows in the arena.
// Of a small swarm as one copy, rearranged on the host: 90 x 26 52 us with a copy per array,
// 62 with a kernel and a copy per array, so 26; 300 x 26, near the line, 66, 59 and 42.
constexpr size_t kSmallState = 512u << 10, kSmallValues = 10000;
template <typename T>
int download_state(cupso_swarm* h, const T* const (&planes)[3], const T* pf, int panel, T* const (&outs)[3], T* pf_out) {
    const size_t N = (size_t)h->N;
    const char* const from = reinterpret_cast<const char*>(planes[0]);
    const size_t bytes = (size_t)(reinterpret_cast<const char*>(pf + N) - from);
    if (h->D > 1 && bytes <= kSmallState && N * (size_t)h->D <= kSmallValues) {
        std::vector<char> mem;
        const int rc = host_planes(&mem, bytes);
        if (rc) return rc;
        CUPSO_CUDA(cudaMemcpyAsync(mem.data(), from, bytes, cudaMemcpyDeviceToHost, h->stream), "cudaMemcpyAsync");
        CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
        auto copy_of = [&](const T* p) {
            return reinterpret_cast<const T*>(mem.data() + (reinterpret_cast<const char*>(p) - from));
        };
        for (int a = 0; a < 3; ++a)
            if (outs[a]) unpack_plane(h, copy_of(planes[a]), panel, outs[a]);
        if (pf_out) std::memcpy(pf_out, copy_of(pf), sizeof(T) * N);
        return CUPSO_OK;
    }
    for (int a = 0; a < 3; ++a) {
        if (!outs[a]) continue;
        const int rc = download_rows(h, planes[a], panel, outs[a]);
        if (rc) return rc;
    }
    if (pf_out)
        CUPSO_CUDA(cudaMemcpyAsync(pf_out, pf, sizeof(T) * N, cudaMemcpyDeviceToHost, h->stream), "cudaMemcpyAsync");
    CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
    return CUPSO_OK;
}

// The reverse of download_rows: a device array in `panel` layout from in[i][d], zeros in the
// padding. ensure_stage comes before, so that a state is not left half loaded; without a
// stage `host` holds a plane.
template <typename T>
int upload_rows(cupso_swarm* h, const T* in, int panel, T* dst, std::vector<char>& host) {
    const size_t D = (size_t)h->D, row = sizeof(T) * D;
    const int pad = h->Np - h->N;
    if (D == 1) {
        CUPSO_CUDA(cudaMemcpyAsync(dst, in, sizeof(T) * (size_t)h->N, cudaMemcpyHostToDevice, h->stream), "cudaMemcpyAsync");
        CUPSO_CUDA(cudaMemsetAsync(dst + h->N, 0, sizeof(T) * (size_t)pad, h->stream), "cudaMemsetAsync");
        return CUPSO_OK;
    }
    if (!h->stage) {
        T* plane = reinterpret_cast<T*>(host.data());
        std::fill(plane, plane + D * (size_t)h->Np, T(0));
        for (size_t i = 0; i < (size_t)h->N; ++i)
            for (size_t d = 0; d < D; ++d) plane[plane_at(d, i, (size_t)h->Np, (size_t)panel)] = in[i * D + d];
        CUPSO_CUDA(cudaMemcpyAsync(dst, plane, row * (size_t)h->Np, cudaMemcpyHostToDevice, h->stream), "cudaMemcpyAsync");
        CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
        return CUPSO_OK;
    }
    const int per = (int)std::min<size_t>((size_t)h->N, h->stage_bytes / row);
    for (int i0 = 0; i0 < h->N; i0 += per) {
        const int n = std::min(per, h->N - i0);
        const bool last = n == h->N - i0;
        CUPSO_CUDA(cudaMemcpyAsync(h->stage, in + (size_t)i0 * D, row * (size_t)n, cudaMemcpyHostToDevice, h->stream),
                   "cudaMemcpyAsync");
        CUPSO_CUDA(launch_pack_rows(static_cast<const T*>(h->stage), dst, h->D, h->Np, panel, i0, n, last ? n + pad : n,
                                    h->stream),
                   "pack launch");
        if (last) break;
    }
    return CUPSO_OK;
}

// pos, v and pbest_pos into the arena.
template <typename T>
int upload_state(cupso_swarm* h, const T* const (&ins)[3], int panel, T* const (&dsts)[3]) {
    std::vector<char> host;
    if (h->D > 1) {
        const size_t row = sizeof(T) * (size_t)h->D;
        int rc = ensure_stage(h, row, (size_t)h->N);
        if (rc == CUPSO_OK && !h->stage) rc = host_planes(&host, row * (size_t)h->Np);
        if (rc) return rc;
    }
    for (int a = 0; a < 3; ++a) {
        const int rc = upload_rows(h, ins[a], panel, dsts[a], host);
        if (rc) return rc;
    }
    return CUPSO_OK;
}

int status_code(unsigned st) {
    if (st & kStatusBadArg) return CUPSO_ERR_CUDA;   // a device-side bound check dropped work
    if (st & kStatusTimeout) return CUPSO_ERR_DEVICE_TIMEOUT;
    if (st & kStatusNaN) return CUPSO_ERR_NAN;
    return CUPSO_OK;
}

double key_to_fit64(unsigned long long key) {
    if (key == ~0ull) return NAN;
    const unsigned long long bits = (key >> 63) ? (key & 0x7FFFFFFFFFFFFFFFull) : ~key;
    double f;
    std::memcpy(&f, &bits, 8);
    return f;
}

float key_to_fit(unsigned long long key) {
    const uint32_t k = (uint32_t)(key >> 32);
    if (k == 0xFFFFFFFFu) return NAN;
    const uint32_t bits = (k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k;
    float f;
    std::memcpy(&f, &bits, 4);
    return f;
}

}  // namespace

// One problem solved through its own handle: create, `iters` steps, gbest.
int cupso::solve_one_plain(const cupso_problem& p, int iters, cupso_result& r, cudaStream_t stream) {
    cupso_handle h = nullptr;
    int rc = create_swarm(p.D, p.N, &p.bounds, p.w, p.c1, p.c2, p.fitness_id, p.seed, p.swarm_id, stream, &h);
    if (rc == CUPSO_OK) rc = cupso_step(h, iters);
    if (rc == CUPSO_OK) rc = cupso_get_gbest(h, &r.fit, r.pos, &r.idx);
    r.status = rc;
    if (h) cupso_destroy(h);
    return rc;
}

void cupso::set_cuda_error(cudaError_t e, const char* where) { cuda_fail(e, where); }

namespace {

// A posted result's record: the gbest key at 0, the sticky status at 16, gbest_pos from 32.
constexpr size_t kRecStatus = 16, kRecPos = 32;
size_t rec_bytes(int D) { return align_up(kRecPos + sizeof(float) * (size_t)D, 256); }

// The current gbest into a contiguous record, a snapshot that later steps do not change.
__global__ void gbest_record_kernel(const uint32_t* __restrict__ key, const unsigned* __restrict__ status,
                                    const uint32_t* __restrict__ G, int D, uint32_t* __restrict__ rec) {
    for (int e = threadIdx.x; e < D; e += blockDim.x) rec[kRecPos / 4 + e] = __ldcg(G + e);
    if (threadIdx.x < 2) rec[threadIdx.x] = __ldcg(key + threadIdx.x);
    if (threadIdx.x == 32) rec[kRecStatus / 4] = __ldcg(status);
}

cudaError_t queue_record(const cupso_swarm* h, char* rec) {
    const size_t cur = h->t_host & 1u, D = (size_t)h->D;
    gbest_record_kernel<<<1, 256, 0, h->stream>>>(reinterpret_cast<const uint32_t*>(h->dev.gkey + cur), h->dev.status,
                                                  reinterpret_cast<const uint32_t*>(h->dev.G + cur * D), (int)D,
                                                  reinterpret_cast<uint32_t*>(rec));
    return cudaGetLastError();
}

// The arena's head in h->head_copy, and *pos, unless null, at the current gbest_pos in it: one copy
// into ordinary memory and one wait (14 us through the Python binding, as with a copy per
// field into pinned memory, which took 130 us to allocate with the first read and 120 to free with the
// handle; with a kernel that gathers a record first 19). It takes both parities' positions
// along where the current one comes second, unless they are long.
int read_head(cupso_swarm* h, const char** pos) {
    const size_t cur = h->t_host & 1u, row = (h->fp64 ? sizeof(double) : sizeof(float)) * (size_t)h->D;
    const bool apart = pos && cur && row > (64u << 10);
    const size_t tail = !pos || apart ? 0 : (cur + 1) * row;
    try {
        h->head_copy.resize(kHeadBytes + (apart ? row : tail));
    } catch (...) {
        return fail(CUPSO_ERR_OOM, "host allocation failed%s");
    }
    char* const to = h->head_copy.data();
    const char* const head = h->fp64 ? reinterpret_cast<const char*>(h->dev64.gkey) : reinterpret_cast<const char*>(h->dev.gkey);
    CUPSO_CUDA(cudaMemcpyAsync(to, head, kHeadBytes + tail, cudaMemcpyDeviceToHost, h->stream), "cudaMemcpyAsync");
    if (apart)
        CUPSO_CUDA(cudaMemcpyAsync(to + kHeadBytes, head + kHeadBytes + row, row, cudaMemcpyDeviceToHost, h->stream),
                   "cudaMemcpyAsync");
    CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
    if (pos) *pos = to + kHeadBytes + (apart ? 0 : cur * row);
    return CUPSO_OK;
}

int ensure_records(cupso_swarm* h) {
    if (h->rec_dev) return CUPSO_OK;
    const size_t bytes = 2 * rec_bytes(h->D);
    CUPSO_CUDA(cudaMalloc(&h->rec_dev, bytes), "cudaMalloc (gbest records)");
    CUPSO_CUDA(cudaMallocHost(&h->rec_host, bytes), "cudaMallocHost (gbest records)");
    CUPSO_CUDA(cudaStreamCreateWithFlags(&h->rec_stream, cudaStreamNonBlocking), "cudaStreamCreate");
    for (int k = 0; k < 2; ++k) {
        CUPSO_CUDA(cudaEventCreateWithFlags(&h->rec_ev[k], cudaEventDisableTiming), "cudaEventCreate");
        CUPSO_CUDA(cudaEventCreateWithFlags(&h->rec_done[k], cudaEventDisableTiming), "cudaEventCreate");
    }
    return CUPSO_OK;
}

}  // namespace

extern "C" {

int cupso_create(int D, int N, const cupso_bounds* bounds, float w, float c1, float c2, int fitness_id,
                 uint64_t seed, cupso_handle* out) {
    return create_swarm(D, N, bounds, w, c1, c2, fitness_id, seed, 0u, nullptr, out);
}

int cupso_set_stream(cupso_handle h, void* cuda_stream) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    h->stream = cuda_stream ? static_cast<cudaStream_t>(cuda_stream) : h->own;
    return CUPSO_OK;
}

int cupso_set_option(cupso_handle h, int key, long long value) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    switch (key) {
        case CUPSO_OPT_MODE:
            if (value < CUPSO_MODE_AUTO || value > CUPSO_MODE_PERSISTENT)
                return fail(CUPSO_ERR_INVALID_ARG, "unknown mode%s");
            if (value == CUPSO_MODE_PERSISTENT && (!h->fp64 || h->D > 4096))
                return fail(CUPSO_ERR_UNSUPPORTED, "the persistent mode serves double-precision swarms with D <= 4096%s");
            if (h->fp64) {
                if (value == CUPSO_MODE_ASYNC)
                    return fail(CUPSO_ERR_UNSUPPORTED, "double-precision swarms have no ASYNC mode%s");
                if (value == CUPSO_MODE_ONCHIP && !h->onchip64)
                    return fail(CUPSO_ERR_UNSUPPORTED, "swarm does not fit in one CTA's shared memory%s");
                h->mode = (int)value;
                return CUPSO_OK;
            }
            if (h->fid == CUPSO_LSQ && value != CUPSO_MODE_AUTO && value != CUPSO_MODE_SYNC)
                return fail(CUPSO_ERR_UNSUPPORTED, "least-squares swarms run the synchronous iteration only%s");
            if (value == CUPSO_MODE_ONCHIP && h->onchip_cluster == 0)
                return fail(CUPSO_ERR_UNSUPPORTED, "swarm does not fit in one cluster's shared memory%s");
            h->mode = (int)value;
            return CUPSO_OK;
        case CUPSO_OPT_GRAPH_CHUNK:
            if (value < 0 || value > 4096) return fail(CUPSO_ERR_INVALID_ARG, "graph chunk out of range%s");
            h->graph_chunk = (int)value;
            drop_graph(h);
            return CUPSO_OK;
        case CUPSO_OPT_WAIT_LIMIT_NS:
            if (value < 1000 || value > 60000000000ll) return fail(CUPSO_ERR_INVALID_ARG, "wait limit out of range%s");
            h->dev.wait_limit_ns = value;
            h->dev64.wait_limit_ns = value;
            drop_graph(h);
            return CUPSO_OK;
        case CUPSO_OPT_CLEAR_STATUS:
            // with the status, the counters a wait that expired may have left behind
            // (a double-precision swarm has none: each launch clears its own barrier)
            CUPSO_CUDA(cudaMemsetAsync(h->dev.status, 0, sizeof(unsigned), h->stream), "cudaMemsetAsync");
            if (h->fp64) return CUPSO_OK;
            CUPSO_CUDA(cudaMemsetAsync(h->dev.ticket, 0, sizeof(unsigned), h->stream), "cudaMemsetAsync");
            CUPSO_CUDA(cudaMemsetAsync(h->dev.work, 0, 6 * sizeof(unsigned), h->stream), "cudaMemsetAsync");
            return CUPSO_OK;
        case CUPSO_OPT_GRID:
            if (value < 0 || value > (1 << 20)) return fail(CUPSO_ERR_INVALID_ARG, "grid out of range%s");
            h->grid_override = (int)value;
            drop_graph(h);
            return CUPSO_OK;
        case CUPSO_OPT_SYNC_KERNEL:
            if (value < CUPSO_SYNC_KERNEL_AUTO || value > CUPSO_SYNC_KERNEL_PANEL16)
                return fail(CUPSO_ERR_INVALID_ARG, "unknown sync kernel%s");
            h->sync_kernel = (int)value;
            drop_graph(h);
            return CUPSO_OK;
        case CUPSO_OPT_TIME_FITNESS:
            if (!h->lsq) return fail(CUPSO_ERR_INVALID_ARG, "timing applies to least-squares swarms after cupso_set_lsq%s");
            h->lsq->time_fitness = value != 0;
            drop_graph(h);
            return CUPSO_OK;
        case CUPSO_OPT_PARTICLES_PER_THREAD:
            if (value != 0 && value != 1 && value != 2 && value != 4)
                return fail(CUPSO_ERR_INVALID_ARG, "particles per thread must be 0 (automatic), 1, 2 or 4%s");
            h->ppt_option = (int)value;
            drop_graph(h);
            return CUPSO_OK;
        case CUPSO_OPT_ITERS_PER_LAUNCH:
            if (value < 0 || value > kPanelMaxIters)
                return fail(CUPSO_ERR_INVALID_ARG, "iterations per launch out of range%s");
            h->iters_per_launch = (int)value;
            return CUPSO_OK;
        case CUPSO_OPT_LSQ_RESCORE:
            if (value != 0 && value != 1) return fail(CUPSO_ERR_INVALID_ARG, "rescoring: 0 (float-float) or 1 (FP64)%s");
            h->lsq_rescore = (int)value;
            if (h->lsq) h->lsq->gram.ff = value == 0;
            drop_graph(h);
            return CUPSO_OK;
        case CUPSO_OPT_FAULT_HOLD_LOCK:
            h->hold_lock = value ? 1 : 0;
            return CUPSO_OK;
        case CUPSO_OPT_FAULT_STALL_BARRIER:
            h->stall_barrier = value ? 1 : 0;
            return CUPSO_OK;
        case CUPSO_OPT_FAULT_NO_STAGING:
            h->no_staging = value != 0;
            return CUPSO_OK;
        default:
            return fail(CUPSO_ERR_INVALID_ARG, "unknown option%s");
    }
}

int cupso_step(cupso_handle h, int iters) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    if (iters < 0) return fail(CUPSO_ERR_INVALID_ARG, "iters must be >= 0%s");
    if (iters == 0) return CUPSO_OK;
    if ((uint64_t)h->t_host + (uint64_t)iters > 0xFFFFFFFFull)
        return fail(CUPSO_ERR_INVALID_ARG, "iteration counter would overflow%s");
    if (h->fid == CUPSO_LSQ) {
        if (!h->lsq) return fail(CUPSO_ERR_INVALID_ARG, "least-squares swarm: call cupso_set_lsq first%s");
        int left = iters;
        const int L = h->lsq->time_fitness ? 0 : h->graph_chunk;
        if (L > 1 && left >= L) {
            int rc = ensure_graph(h, kModeLsq, L);
            if (rc) return rc;
            while (left >= L) {
                cudaError_t e = cudaGraphLaunch(h->graph, h->stream);
                if (e != cudaSuccess) return cuda_fail(e, "cudaGraphLaunch");
                left -= L;
            }
        }
        for (; left > 0; --left) {
            cudaError_t e = launch_lsq_iteration(h, h->stream);
            if (e != cudaSuccess) return cuda_fail(e, "least-squares iteration");
        }
        // the tensor-core iteration leaves improved pbest rows to the next move
        if (lsq_approx(h->lsq->precision)) h->lazy_pending = true;
        h->t_host += (uint32_t)iters;
        return CUPSO_OK;
    }
    const int mode = resolved_mode(h);
    const int from = one_launch_from(h, mode);
    bool one_launch = from > 0 && iters >= from;
    // A stream that may use only some of the SMs (a green context's) refuses a launch whose CTAs
    // would not all be resident: the call then runs as a shorter one would.
    auto refused = [&](cudaError_t e) {
        if (e != cudaErrorCooperativeLaunchTooLarge || mode == CUPSO_MODE_PERSISTENT) return false;
        cudaGetLastError();
        one_launch = false;
        return true;
    };
    if (h->fp64 && one_launch) {
        // PERSISTENT: one launch by definition
        const int most = mode != CUPSO_MODE_PERSISTENT && h->iters_per_launch > 0 ? h->iters_per_launch : kSync64MaxIters;
        const cudaError_t e = launch_sync64(h->dev64, h->s64bufs, h->fid, iters, most, h->stall_barrier != 0, h->num_sms,
                                            h->stream);
        if (e != cudaSuccess && !refused(e)) return cuda_fail(e, "one-launch step");
        if (e == cudaSuccess) {
            h->t_host += (uint32_t)iters;
            return CUPSO_OK;
        }
    }
    if (h->fp64 && mode == CUPSO_MODE_ONCHIP) {
        cudaError_t e = launch_onchip64(h->dev64, h->fid, iters, h->stream);
        if (e != cudaSuccess) return cuda_fail(e, "on-chip launch");
        h->t_host += (uint32_t)iters;
        return CUPSO_OK;
    }
    if (!h->fp64 && one_launch) {
        // any layout, pending pbest rows included; a launch's iterations as for the panel step
        const int most = h->iters_per_launch > 0 ? h->iters_per_launch : kResidentMaxIters;
        for (int left = iters; one_launch && left > 0;) {
            const int n = std::min(left, most);
            const cudaError_t e = launch_resident(h->dev, h->rbufs, h->fid, h->panel, n, h->stall_barrier != 0, h->num_sms,
                                                  h->stream);
            if (e != cudaSuccess && (left < iters || !refused(e))) return cuda_fail(e, "resident launch");
            left -= n;
        }
        if (one_launch) {
            h->lazy_pending = false;
            h->t_host += (uint32_t)iters;
            return CUPSO_OK;
        }
    }
    const int panel = (!h->fp64 && mode == CUPSO_MODE_SYNC) ? panel_cfg(h).width : 0;
    {
        const int rc = ensure_layout(h, panel);
        if (rc) return rc;
    }
    const bool pipelined =
        panel != 0 || (!h->fp64 && mode == CUPSO_MODE_SYNC && sync_tile(h) == 0 && sync_stages(h) > 0);
    if (!pipelined) {
        const int rc = ensure_materialized(h);
        if (rc) return rc;
    }
    cudaError_t e = cudaSuccess;
    if (mode == CUPSO_MODE_ASYNC) {
        if (const int P = async_tile(h))
            e = launch_async_tiled(h->dev, h->fid, P, async_grid(h), h->t_host + 1u, iters, h->hold_lock, h->stream);
        else
            e = launch_async(h->dev, h->fid, async_grid(h), async_block(h), h->t_host + 1u, iters, h->hold_lock,
                             h->stream);
        if (e != cudaSuccess) return cuda_fail(e, "async launch");
    } else if (mode == CUPSO_MODE_ONCHIP) {
        e = launch_onchip(h->dev, h->fid, iters, h->stream);
        if (e != cudaSuccess) return cuda_fail(e, "on-chip launch");
    } else {
        int left = iters;
        const int P = panel ? panel_iters_per_launch(h) : 1;
        if (P > 1 && left > 1) {
            // several iterations per cooperative launch, a grid barrier between them
            const PanelCfg pc = panel_cfg(h);
            const int grid = panel_persist_grid(h, pc);
            while (left > 1) {
                const int n = std::min(left, P);
                e = cudaMemsetAsync(h->dev.work, 0, 6 * sizeof(unsigned), h->stream);
                if (e == cudaSuccess)
                    e = launch_sync_panel(h->dev, h->fid, pc.width, pc.stages, grid, n, h->stall_barrier != 0,
                                          h->stream);
                if (e != cudaSuccess) return cuda_fail(e, "panel launch");
                left -= n;
            }
        }
        const int L = h->graph_chunk;
        if (L > 1 && left >= L) {
            int rc = ensure_graph(h, mode, L);
            if (rc) return rc;
            while (left >= L) {
                e = cudaGraphLaunch(h->graph, h->stream);
                if (e != cudaSuccess) return cuda_fail(e, "cudaGraphLaunch");
                left -= L;
            }
        }
        for (; left > 0; --left) {
            e = launch_one(h, mode, h->stream);
            if (e != cudaSuccess) return cuda_fail(e, "step launch");
        }
    }
    if (pipelined) h->lazy_pending = true;
    h->t_host += (uint32_t)iters;
    return CUPSO_OK;
}

int cupso_get_gbest(cupso_handle h, float* fit_out, float* pos_out, int64_t* idx_out) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    if (h->fp64) return fail(CUPSO_ERR_UNSUPPORTED, "double-precision swarm: use the _fp64 functions%s");
    const char* pos = nullptr;
    int rc = read_head(h, pos_out ? &pos : nullptr);
    if (rc) return rc;
    unsigned long long key = 0;
    unsigned st = 0;
    std::memcpy(&key, h->head_copy.data() + sizeof(key) * (h->t_host & 1u), sizeof(key));
    std::memcpy(&st, h->head_copy.data() + kHeadStatus, sizeof(st));
    if (pos_out) std::memcpy(pos_out, pos, sizeof(float) * (size_t)h->D);
    if (fit_out) *fit_out = key_to_fit(key);
    if (idx_out) *idx_out = (int64_t)(key & 0xFFFFFFFFull);
    rc = status_code(st);
    if (rc) fail(rc, "device status set: %s", cupso_status_string(rc));
    return rc;
}

int cupso_gbest_post(cupso_handle h, int slot) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    if (h->fp64) return fail(CUPSO_ERR_UNSUPPORTED, "double-precision swarm: use the _fp64 functions%s");
    if (slot != 0 && slot != 1) return fail(CUPSO_ERR_INVALID_ARG, "slot must be 0 or 1%s");
    if (h->rec_posted[slot]) return fail(CUPSO_ERR_INVALID_ARG, "slot already holds a result; wait for it first%s");
    int rc = ensure_records(h);
    if (rc) return rc;
    const size_t rb = rec_bytes(h->D);
    char* dev = h->rec_dev + (size_t)slot * rb;
    // the snapshot follows the queued steps on the handle's stream; the next
    // step cannot change what it copies (a step rewrites these words only
    // after the stream reaches it). Its copy to the host runs on the second
    // stream, beside the next steps.
    CUPSO_CUDA(queue_record(h, dev), "gbest record launch");
    CUPSO_CUDA(cudaEventRecord(h->rec_ev[slot], h->stream), "cudaEventRecord");
    CUPSO_CUDA(cudaStreamWaitEvent(h->rec_stream, h->rec_ev[slot], 0), "cudaStreamWaitEvent");
    CUPSO_CUDA(cudaMemcpyAsync(h->rec_host + (size_t)slot * rb, dev, rb, cudaMemcpyDeviceToHost, h->rec_stream),
               "cudaMemcpyAsync");
    CUPSO_CUDA(cudaEventRecord(h->rec_done[slot], h->rec_stream), "cudaEventRecord");
    h->rec_posted[slot] = true;
    return CUPSO_OK;
}

int cupso_gbest_wait(cupso_handle h, int slot, float* fit_out, float* pos_out, int64_t* idx_out) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    if (slot != 0 && slot != 1) return fail(CUPSO_ERR_INVALID_ARG, "slot must be 0 or 1%s");
    if (!h->rec_posted[slot]) return fail(CUPSO_ERR_INVALID_ARG, "nothing posted to this slot%s");
    CUPSO_CUDA(cudaEventSynchronize(h->rec_done[slot]), "cudaEventSynchronize");
    h->rec_posted[slot] = false;
    const char* rec = h->rec_host + (size_t)slot * rec_bytes(h->D);
    unsigned long long key = 0;
    unsigned st = 0;
    std::memcpy(&key, rec, 8);
    std::memcpy(&st, rec + kRecStatus, 4);
    if (pos_out) std::memcpy(pos_out, rec + kRecPos, sizeof(float) * (size_t)h->D);
    if (fit_out) *fit_out = key_to_fit(key);
    if (idx_out) *idx_out = (int64_t)(key & 0xFFFFFFFFull);
    const int rc = status_code(st);
    if (rc) fail(rc, "device status set: %s", cupso_status_string(rc));
    return rc;
}

int cupso_get_state(cupso_handle h, float* pos, float* v, float* pbest_pos, float* pbest_fit, uint32_t* t_out) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    if (h->fp64) return fail(CUPSO_ERR_UNSUPPORTED, "double-precision swarm: use the _fp64 functions%s");
    const int mrc = ensure_materialized(h);
    if (mrc) return mrc;
    float* const outs[3] = {pos, v, pbest_pos};
    const float* const planes[3] = {h->dev.x, h->dev.v, h->dev.pb};
    const int rc = download_state(h, planes, static_cast<const float*>(h->dev.pf), h->panel, outs, pbest_fit);
    if (rc) return rc;
    if (t_out) *t_out = h->t_host;
    return CUPSO_OK;
}

int cupso_set_state(cupso_handle h, const float* pos, const float* v, const float* pbest_pos,
                    const float* pbest_fit, uint32_t t) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    if (h->fp64) return fail(CUPSO_ERR_UNSUPPORTED, "double-precision swarm: use the _fp64 functions%s");
    if (!pos || !v || !pbest_pos || !pbest_fit) return fail(CUPSO_ERR_INVALID_ARG, "state array is NULL%s");
    CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
    // straight into the layout that the next step reads
    const int panel = resolved_mode(h) == CUPSO_MODE_SYNC ? panel_cfg(h).width : 0;
    const float* const ins[3] = {pos, v, pbest_pos};
    float* const dsts[3] = {h->dev.x, h->dev.v, h->dev.pb};
    const int rc = upload_state(h, ins, panel, dsts);
    if (rc) return rc;
    CUPSO_CUDA(cudaMemcpyAsync(h->dev.pf, pbest_fit, sizeof(float) * (size_t)h->N, cudaMemcpyHostToDevice, h->stream),
               "cudaMemcpyAsync");
    CUPSO_CUDA(cudaMemsetAsync(h->dev.pflag, 0, (size_t)h->Np, h->stream), "cudaMemsetAsync");
    h->lazy_pending = false;
    if (h->panel != panel) drop_graph(h);
    h->panel = panel;
    if (h->lsq && lsq_approx(h->lsq->precision)) {
        // the given pbest_fit are approximate values: gbest only from the rescoring
        CUPSO_CUDA(lsq_reset_gbest(h, h->dev.pf, t, h->stream), "lsq gbest");
    } else {
        CUPSO_CUDA(launch_recompute(h->dev, t, panel, true, h->stream), "recompute launch");
    }
    CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
    h->t_host = t;
    return CUPSO_OK;
}

int cupso_set_lsq(cupso_handle h, const float* A_dev, const float* b_dev, int M, int precision) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    if (h->fp64) return fail(CUPSO_ERR_UNSUPPORTED, "double-precision swarm: use the _fp64 functions%s");
    if (h->fid != CUPSO_LSQ) return fail(CUPSO_ERR_INVALID_ARG, "swarm was not created with CUPSO_LSQ%s");
    if (!A_dev || !b_dev || M < 1) return fail(CUPSO_ERR_INVALID_ARG, "A, b must be device arrays and M >= 1%s");
    if (precision < CUPSO_LSQ_FP32 || precision > CUPSO_LSQ_FP64) return fail(CUPSO_ERR_INVALID_ARG, "unknown precision%s");
    if (lsq_approx(precision) && !lsq_tc_available())
        return fail(CUPSO_ERR_UNSUPPORTED, "tensor-core least squares needs cuTensorMapEncodeTiled%s");
    int rc = ensure_materialized(h);
    if (rc) return rc;
    CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
    drop_graph(h);
    if (h->lsq) {
        for (cudaEvent_t ev : h->lsq->ev) cudaEventDestroy(ev);
        if (h->lsq->fork) cudaEventDestroy(h->lsq->fork);
        if (h->lsq->join) cudaEventDestroy(h->lsq->join);
        if (h->lsq->side) cudaStreamDestroy(h->lsq->side);
        lsq_free_tc(&h->lsq->tc);
        if (h->lsq->buf) cudaFree(h->lsq->buf);
        if (h->lsq->gram_buf) cudaFree(h->lsq->gram_buf);
        delete h->lsq;
        h->lsq = nullptr;
    }
    auto* L = new (std::nothrow) cupso_swarm::Lsq();
    if (!L) return fail(CUPSO_ERR_OOM, "host allocation failed%s");
    h->lsq = L;
    L->A = A_dev;
    L->b = b_dev;
    L->M = M;
    L->precision = precision;
    const int nlists = lsq_cand_lists(h->Np);
    // FP64 rescoring in pieces of at most 8 row pairs of A^T A (one per warp of
    // a block), as many pieces as give every SM two of the 4 x pieces blocks
    {
        const int npairs = (h->D + 1) / 2;
        const int target = std::max(1, h->num_sms / 2);
        const int per = std::min(8, std::max(1, (npairs + target - 1) / target));
        L->chunks = std::max(32, (npairs + per - 1) / per);
    }
    // candidates: 16 per list, the merged 16, and the merging ticket; partial
    // sums: 16 per piece of the row-wise rescoring or tile of the float-float one
    const int npart = std::max(L->chunks, lsq_ff_tiles(h->D));
    const size_t bytes = align_up(sizeof(float) * h->Np, 256) + align_up(sizeof(unsigned long long) * (nlists * 16 + 17), 256) +
                         align_up(sizeof(double) * 16 * npart, 256) + align_up((size_t)h->Np, 256) + 256;
    const bool fp64_fit = precision == CUPSO_LSQ_FP64;
    cudaError_t e = lsq_approx(precision) ? cudaMalloc(&L->buf, bytes)
                                          : lsq_exact_alloc(&L->buf, bytes, h->N, h->D, M, fp64_fit, false, h->num_sms,
                                                            &L->exact_ws, &L->ws_most);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc (lsq)");
    char* p = static_cast<char*>(L->buf);
    L->f = reinterpret_cast<float*>(p); p += align_up(sizeof(float) * h->Np, 256);
    L->cand = reinterpret_cast<unsigned long long*>(p); p += align_up(sizeof(unsigned long long) * (nlists * 16 + 17), 256);
    L->partial = reinterpret_cast<double*>(p); p += align_up(sizeof(double) * 16 * npart, 256);
    L->flags = reinterpret_cast<unsigned int*>(p); p += align_up((size_t)h->Np, 256);
    L->g64 = reinterpret_cast<double*>(p); p += 256;
    const double inf = INFINITY;
    CUPSO_CUDA(cudaMemcpyAsync(L->g64, &inf, sizeof(double), cudaMemcpyHostToDevice, h->stream), "cudaMemcpyAsync");
    CUPSO_CUDA(cudaMemsetAsync(L->f, 0, sizeof(float) * h->Np, h->stream), "cudaMemsetAsync");
    CUPSO_CUDA(cudaMemsetAsync(L->cand + (size_t)nlists * 16 + 16, 0, sizeof(unsigned long long), h->stream),
               "cudaMemsetAsync");
    if (lsq_approx(precision)) {
        CUPSO_CUDA(cudaStreamCreateWithFlags(&L->side, cudaStreamNonBlocking), "cudaStreamCreate");
        CUPSO_CUDA(cudaEventCreateWithFlags(&L->fork, cudaEventDisableTiming), "cudaEventCreate");
        CUPSO_CUDA(cudaEventCreateWithFlags(&L->join, cudaEventDisableTiming), "cudaEventCreate");
        // FP8 scale of the operand: displacements between two points of the box
        // are at most max_pos - min_pos in magnitude
        const float span = h->dev.hi - h->dev.lo;
        const float sx = std::isfinite(span) && span > 0.0f ? 448.0f / span : 1.0f;
        rc = lsq_setup_tc(&L->tc, A_dev, b_dev, M, h->D, h->Np, precision == CUPSO_LSQ_FP8, sx, nullptr, 0,
                          h->stream);
        if (rc) return rc;
        if (!lsq_make_move_maps(L->tc.tmMove, h->dev.x, h->dev.v, h->dev.pb, h->Np, h->D))
            return fail(CUPSO_ERR_UNSUPPORTED, "tensor maps of the move could not be encoded%s");
        if (h->D <= M && h->D <= kGramMaxD) {
            // Gram data: A^T A, A^T b (device, FP64), A^T A again as binary32
            // pairs for the float-float rescoring, and b^T b (host, from b)
            const int ldf = (h->D + kFfTile - 1) / kFfTile * kFfTile;
            const size_t n64 = align_up(sizeof(double) * ((size_t)h->D * h->D + h->D), 256);
            CUPSO_CUDA(cudaMalloc(&L->gram_buf, n64 + sizeof(float2) * (size_t)ldf * ldf), "cudaMalloc (gram)");
            L->gram.Gm = static_cast<double*>(L->gram_buf);
            L->gram.cvec = L->gram.Gm + (size_t)h->D * h->D;
            L->gram.Gff = reinterpret_cast<float2*>(static_cast<char*>(L->gram_buf) + n64);
            L->gram.ldf = ldf;
            L->gram.ff = h->lsq_rescore == 0;
            CUPSO_CUDA(lsq_launch_gram(A_dev, b_dev, M, h->D, L->gram.Gm, L->gram.cvec, L->gram.Gff, ldf, h->stream),
                       "gram launch");
            std::vector<float> hb((size_t)M);
            CUPSO_CUDA(cudaMemcpyAsync(hb.data(), b_dev, sizeof(float) * M, cudaMemcpyDeviceToHost, h->stream),
                       "cudaMemcpyAsync");
            CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
            double bb = 0.0;
            for (float v : hb) bb = std::fma((double)v, (double)v, bb);
            L->gram.bb = bb;
        }
    }
    // Step 1 completes here: pbest_fit = f(pbest_pos), gbest from it.
    if (precision == CUPSO_LSQ_FP32 || precision == CUPSO_LSQ_FP64) {
        CUPSO_CUDA(lsq_exact_launch(h->dev.pb, h->Np, h->N, h->D, A_dev, b_dev, M, fp64_fit, L->f, L->exact_ws, L->ws_most,
                                    h->num_sms, h->stream),
                   "lsq fitness");
        CUPSO_CUDA(lsq_launch_set_pf(h->dev, L->f, h->stream), "lsq pbest");
        CUPSO_CUDA(launch_recompute(h->dev, h->t_host, 0, false, h->stream), "recompute launch");
    } else {
        // the positions' own fitness (reference point 0: offsets -b)
        rc = lsq_eval_tc(&L->tc, h->dev.pb, 1, (size_t)h->Np, h->N, L->f, h->stream);
        if (rc) return rc;
        CUPSO_CUDA(lsq_launch_set_pf(h->dev, L->f, h->stream), "lsq pbest");
        CUPSO_CUDA(lsq_reset_gbest(h, L->f, h->t_host, h->stream), "lsq gbest");
    }
    CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
    return CUPSO_OK;
}

int cupso_get_gbest_f64(cupso_handle h, double* fit_out) {
    if (!h || !fit_out) return fail(CUPSO_ERR_INVALID_ARG, "NULL argument%s");
    if (h->fid != CUPSO_LSQ || !h->lsq) return fail(CUPSO_ERR_INVALID_ARG, "not a least-squares swarm with A, b set%s");
    cupso_swarm::Lsq& L = *h->lsq;
    if (!lsq_approx(L.precision)) {
        // rescore the gbest particle's pbest_pos (== gbest_pos) in FP64
        const int rc = ensure_materialized(h);
        if (rc) return rc;
        const int cur = (int)(h->t_host & 1u);
        CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
        unsigned long long key = 0;
        CUPSO_CUDA(cudaMemcpy(&key, h->dev.gkey + cur, sizeof(key), cudaMemcpyDeviceToHost), "cudaMemcpy");
        const double inf = INFINITY;
        CUPSO_CUDA(cudaMemcpy(L.g64, &inf, sizeof(double), cudaMemcpyHostToDevice), "cudaMemcpy");
        CUPSO_CUDA(lsq_rescore_one(h->dev, L.A, L.b, L.M, key, L.cand, L.partial, L.chunks, L.g64, h->stream),
                   "lsq rescore");
    }
    CUPSO_CUDA(cudaMemcpyAsync(fit_out, L.g64, sizeof(double), cudaMemcpyDeviceToHost, h->stream), "cudaMemcpyAsync");
    CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
    return CUPSO_OK;
}

int cupso_create_fp64(int D, int N, const cupso_bounds_f64* bounds, double w, double c1, double c2, int fitness_id,
                      uint64_t seed, cupso_handle* out) {
    return create_swarm64(D, N, bounds, w, c1, c2, fitness_id, seed, out);
}

int cupso_get_gbest_fp64(cupso_handle h, double* fit_out, double* pos_out, int64_t* idx_out) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    if (!h->fp64) return fail(CUPSO_ERR_UNSUPPORTED, "not a double-precision swarm%s");
    const char* pos = nullptr;
    int rc = read_head(h, pos_out ? &pos : nullptr);
    if (rc) return rc;
    PKey key{};
    unsigned st = 0;
    std::memcpy(&key, h->head_copy.data() + sizeof(PKey) * (h->t_host & 1u), sizeof(PKey));
    std::memcpy(&st, h->head_copy.data() + kHeadStatus64, sizeof(st));
    if (pos_out) std::memcpy(pos_out, pos, sizeof(double) * (size_t)h->D);
    if (fit_out) *fit_out = key_to_fit64(key.k);
    if (idx_out) *idx_out = (int64_t)key.i;
    rc = status_code(st);
    if (rc) fail(rc, "device status set: %s", cupso_status_string(rc));
    return rc;
}

int cupso_get_state_fp64(cupso_handle h, double* pos, double* v, double* pbest_pos, double* pbest_fit,
                         uint32_t* t_out) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    if (!h->fp64) return fail(CUPSO_ERR_UNSUPPORTED, "not a double-precision swarm%s");
    double* const outs[3] = {pos, v, pbest_pos};
    const double* const planes[3] = {h->dev64.x, h->dev64.v, h->dev64.pb};
    const int rc = download_state(h, planes, static_cast<const double*>(h->dev64.pf), 0, outs, pbest_fit);
    if (rc) return rc;
    if (t_out) *t_out = h->t_host;
    return CUPSO_OK;
}

int cupso_set_state_fp64(cupso_handle h, const double* pos, const double* v, const double* pbest_pos,
                         const double* pbest_fit, uint32_t t) {
    if (!h) return fail(CUPSO_ERR_INVALID_ARG, "handle is NULL%s");
    if (!h->fp64) return fail(CUPSO_ERR_UNSUPPORTED, "not a double-precision swarm%s");
    if (!pos || !v || !pbest_pos || !pbest_fit) return fail(CUPSO_ERR_INVALID_ARG, "state array is NULL%s");
    const size_t N = (size_t)h->N;
    CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
    const double* const ins[3] = {pos, v, pbest_pos};
    double* const dsts[3] = {h->dev64.x, h->dev64.v, h->dev64.pb};
    const int rc = upload_state(h, ins, 0, dsts);
    if (rc) return rc;
    static const std::vector<double> inf((size_t)kPad, (double)INFINITY);   // pbest_fit of the padding
    CUPSO_CUDA(cudaMemcpyAsync(h->dev64.pf, pbest_fit, sizeof(double) * N, cudaMemcpyHostToDevice, h->stream), "cudaMemcpyAsync");
    CUPSO_CUDA(cudaMemcpyAsync(h->dev64.pf + N, inf.data(), sizeof(double) * (size_t)(h->Np - h->N), cudaMemcpyHostToDevice,
                               h->stream),
               "cudaMemcpyAsync");
    CUPSO_CUDA(cudaMemcpyAsync(h->dev64.t_dev, &t, sizeof(t), cudaMemcpyHostToDevice, h->stream), "cudaMemcpyAsync");
    CUPSO_CUDA(launch_recompute64(h->dev64, h->pbufs, h->stream), "recompute launch");
    CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
    h->t_host = t;
    return CUPSO_OK;
}

int cupso_get_info(cupso_handle h, cupso_info* info) {
    if (!h || !info) return fail(CUPSO_ERR_INVALID_ARG, "NULL argument%s");
    info->N = h->N;
    info->D = h->D;
    info->Np = h->Np;
    info->mode = resolved_mode(h);
    info->t = h->t_host;
    if (h->fp64) {
        info->sync_grid = paper_blocks(h->N);
        info->async_grid = 0;
        info->onchip_cluster = h->onchip_cluster;
        info->sync_stages = 0;
        info->sync_ppt = 0;
        info->sync_tile = 0;
        info->sync_panel = 0;
        info->sync_iters_per_launch = 1;
    } else {
        const int tile = sync_tile(h);
        info->sync_grid = tile ? std::min(tiled_grid(h, tile), (h->N + tile - 1) / tile) : sync_grid(h);
        info->async_grid = async_grid(h);
        info->onchip_cluster = h->onchip_cluster;
        const PanelCfg pc = panel_cfg(h);
        info->sync_stages = pc.width ? pc.stages : (tile ? 0 : sync_stages(h));
        info->sync_ppt = pc.width ? 1 : ((!tile && sync_stages(h)) ? sync_ppt(h) : 0);
        info->sync_tile = pc.width ? 0 : tile;
        info->sync_panel = pc.width;
        info->sync_iters_per_launch = pc.width ? panel_iters_per_launch(h) : 1;
    }
    info->one_launch_iters = h->fid == CUPSO_LSQ ? 0 : one_launch_from(h, info->mode);
    info->fitness_ms = 0.0f;
    info->fitness_timed = 0;
    if (h->lsq) {
        cupso_swarm::Lsq& L = *h->lsq;
        if (!L.ev.empty()) {
            CUPSO_CUDA(cudaStreamSynchronize(h->stream), "cudaStreamSynchronize");
            for (size_t k = 0; k + 1 < L.ev.size(); k += 2) {
                float ms = 0.0f;
                if (cudaEventElapsedTime(&ms, L.ev[k], L.ev[k + 1]) == cudaSuccess) {
                    L.fitness_ms_sum += ms;
                    ++L.fitness_timed;
                }
                cudaEventDestroy(L.ev[k]);
                cudaEventDestroy(L.ev[k + 1]);
            }
            L.ev.clear();
        }
        if (L.fitness_timed) {
            info->fitness_ms = (float)(L.fitness_ms_sum / L.fitness_timed);
            info->fitness_timed = L.fitness_timed;
        }
    }
    info->device_bytes = (uint64_t)h->arena_bytes;
    return CUPSO_OK;
}

int cupso_destroy(cupso_handle h) {
    if (!h) return CUPSO_OK;
    int rc = CUPSO_OK;
    if (h->stream) {
        cudaError_t e = cudaStreamSynchronize(h->stream);
        if (e != cudaSuccess) rc = cuda_fail(e, "cudaStreamSynchronize");
    }
    drop_graph(h);
    if (h->lsq) {
        for (cudaEvent_t ev : h->lsq->ev) cudaEventDestroy(ev);
        if (h->lsq->fork) cudaEventDestroy(h->lsq->fork);
        if (h->lsq->join) cudaEventDestroy(h->lsq->join);
        if (h->lsq->side) cudaStreamDestroy(h->lsq->side);
        lsq_free_tc(&h->lsq->tc);
        if (h->lsq->buf) cudaFree(h->lsq->buf);
        if (h->lsq->gram_buf) cudaFree(h->lsq->gram_buf);
        delete h->lsq;
        h->lsq = nullptr;
    }
    if (h->rec_stream) {
        cudaError_t e = cudaStreamSynchronize(h->rec_stream);
        if (e != cudaSuccess && rc == CUPSO_OK) rc = cuda_fail(e, "cudaStreamSynchronize");
        cudaStreamDestroy(h->rec_stream);
    }
    for (int k = 0; k < 2; ++k) {
        if (h->rec_ev[k]) cudaEventDestroy(h->rec_ev[k]);
        if (h->rec_done[k]) cudaEventDestroy(h->rec_done[k]);
    }
    if (h->rec_dev) cudaFree(h->rec_dev);
    if (h->rec_host) cudaFreeHost(h->rec_host);
    if (h->arena) cudaFree(h->arena);
    if (h->stage) cudaFree(h->stage);
    if (h->capture) cudaStreamDestroy(h->capture);
    if (h->own) cudaStreamDestroy(h->own);
    delete h;
    return rc;
}

const char* cupso_status_string(int status) {
    switch (status) {
        case CUPSO_OK: return "ok";
        case CUPSO_ERR_INVALID_ARG: return "invalid argument";
        case CUPSO_ERR_OOM: return "out of device memory";
        case CUPSO_ERR_CUDA: return "CUDA error";
        case CUPSO_ERR_DEVICE_TIMEOUT: return "device-side wait timed out";
        case CUPSO_ERR_NAN: return "fitness evaluated to NaN";
        case CUPSO_ERR_UNSUPPORTED: return "unsupported";
        default: return "unknown status";
    }
}

const char* cupso_last_error(void) { return g_last_error; }

}  // extern "C"
