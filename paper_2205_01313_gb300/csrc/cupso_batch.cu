// cupso_batch.cu -- cupso_solve_batch: many independent swarms at once.
//
// All swarms of a batch live in one device arena. Swarms of kBatchPanelMinD
// dimensions or more are kept in panels (but for those that padding to whole panels
// would slow, or where it would not fit the device) and advance together, one launch per
// iteration (kernels_batch_panel.cu). The others have a launch of their own: one
// runs Step 1 of every swarm (batch_init_kernel), then every iteration is ONE launch
// of batch_step_kernel covering the units of all of them (kernels_batch.cu). The
// `iters` launches are replayed from captured CUDA graphs. Two kernels can
// run the step of the swarms that are not in panels: the streaming one (kernels_batch.cu: 128-particle units per
// warp, rows staged through a cp.async ring) and the tiled one
// (kernels_tiled.cu: tiles of P particles with all their dimensions per CTA,
// P chosen per swarm so that tiles cost about the same). The launch shape
// (kernel, ring depth, CTAs per SM) is chosen online: the first iterations of
// the real run are timed under each candidate shape and the fastest one runs
// the rest -- every shape computes the same bits, so tuning costs no extra
// work. Choices are remembered per batch shape for the life of the process.
//
// Swarms with fewer than three dimensions (too few dimension pairs for the
// ring's look-ahead) are solved one by one through their own handles.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "../../include/cupso.h"
#include "cupso_device.cuh"
#include "cupso_internal.h"
#include "tiled_kernels.h"

using namespace cupso;

namespace {

size_t up(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct Shape {
    int stages;          // ring depth of the streaming kernel; 0: the tiled kernel; -1: the panels'
    int minb;            // register budget: CTAs per SM (the panels' kernel: its deep ring)
    int blocks_per_sm;   // CTAs per SM launched (the panels' kernel: CTAs in all)
};

// Launch shapes remembered per batch signature.
std::mutex g_tune_mutex;
std::map<std::tuple<int, long long, int, int>, Shape> g_tuned;

// BatchSwarm::cst from the other fields.
void set_constants(BatchSwarm& w) {
    uint32_t rk0[10], rk1[10];
    philox_round_keys(w.key0, w.key1, rk0, rk1);
    for (int k = 0; k < 5; ++k) w.cst[k] = make_uint4(rk0[2 * k], rk1[2 * k], rk0[2 * k + 1], rk1[2 * k + 1]);
    const float m[6] = {w.w, w.fast ? w.c1s : w.c1, w.fast ? w.c2s : w.c2, w.vmax, w.lo, w.hi};
    uint32_t u[6];
    std::memcpy(u, m, sizeof u);
    w.cst[5] = make_uint4(u[0], u[1], u[2], u[3]);
    w.cst[6] = make_uint4(u[4], u[5], w.swarm, 0u);
    w.cst[7] = make_uint4(0u, 0u, 0u, 0u);
}

// The swarms that advance in one launch.
struct BatchRun {
    cudaStream_t st = nullptr;
    BatchDev dev{};
    BatchTiles tiles{};
    int num_sms = 1;
    cudaGraphExec_t graph = nullptr;
    Shape graph_shape{0, 0, 0};
    int graph_len = 0;

    ~BatchRun() {
        if (graph) cudaGraphExecDestroy(graph);
    }

    cudaError_t launch(const Shape& sh) { return launch_on(sh, st); }

    cudaError_t launch_on(const Shape& sh, cudaStream_t s) {
        if (sh.stages < 0) return launch_batch_panel(dev, sh.minb != 0, sh.blocks_per_sm, s);
        if (sh.stages == 0) return launch_batch_tiled(dev, tiles, num_sms * sh.blocks_per_sm, s);
        return launch_batch_step(dev, sh.stages, sh.minb, num_sms * sh.blocks_per_sm, s);
    }

    // `n` iterations with shape `sh`, through a captured graph of up to 32 launches.
    int run(const Shape& sh, int n) {
        const int L = std::min(n, 32);
        if (L >= 4 && (!graph || graph_len != L || graph_shape.stages != sh.stages || graph_shape.minb != sh.minb ||
                       graph_shape.blocks_per_sm != sh.blocks_per_sm)) {
            if (graph) cudaGraphExecDestroy(graph);
            graph = nullptr;
            cudaStream_t cap = nullptr;
            cudaError_t e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
            if (e != cudaSuccess) return set_cuda_error(e, "cudaStreamCreate"), CUPSO_ERR_CUDA;
            e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
            cudaError_t le = cudaSuccess;
            for (int k = 0; k < L && e == cudaSuccess && le == cudaSuccess; ++k)
                le = launch_on(sh, cap);
            cudaGraph_t g = nullptr;
            cudaError_t ee = e == cudaSuccess ? cudaStreamEndCapture(cap, &g) : e;
            cudaStreamDestroy(cap);
            if (le != cudaSuccess || ee != cudaSuccess) {
                if (g) cudaGraphDestroy(g);
                set_cuda_error(le != cudaSuccess ? le : ee, "batch graph capture");
                return CUPSO_ERR_CUDA;
            }
            e = cudaGraphInstantiate(&graph, g, 0);
            cudaGraphDestroy(g);
            if (e != cudaSuccess) {
                graph = nullptr;
                set_cuda_error(e, "cudaGraphInstantiate");
                return CUPSO_ERR_CUDA;
            }
            graph_len = L;
            graph_shape = sh;
        }
        int left = n;
        while (graph && left >= graph_len) {
            cudaError_t e = cudaGraphLaunch(graph, st);
            if (e != cudaSuccess) return set_cuda_error(e, "cudaGraphLaunch"), CUPSO_ERR_CUDA;
            left -= graph_len;
        }
        for (; left > 0; --left) {
            cudaError_t e = launch(sh);
            if (e != cudaSuccess) return set_cuda_error(e, "batch launch"), CUPSO_ERR_CUDA;
        }
        return CUPSO_OK;
    }
};

float key_fit(unsigned long long key) {
    const uint32_t k = (uint32_t)(key >> 32);
    if (k == 0xFFFFFFFFu) return NAN;
    const uint32_t bits = (k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k;
    float f;
    std::memcpy(&f, &bits, 4);
    return f;
}

}  // namespace

extern "C" int cupso_solve_batch(int n_swarms, const cupso_problem* problems, int iters, cupso_result* results,
                                 void* cuda_stream) {
    if (n_swarms < 0 || iters < 0) {
        set_last_error("n_swarms and iters must be >= 0");
        return CUPSO_ERR_INVALID_ARG;
    }
    if (n_swarms > 0 && (!problems || !results)) {
        set_last_error("NULL problems/results");
        return CUPSO_ERR_INVALID_ARG;
    }
    for (int k = 0; k < n_swarms; ++k) {
        const cupso_problem& p = problems[k];
        const int rc = check_problem_args(p.D, p.N, &p.bounds, p.w, p.c1, p.c2, p.fitness_id);
        if (rc) return rc;
        if (p.fitness_id == CUPSO_LSQ) {
            // the least-squares fitness needs A and b (cupso_set_lsq); a problem record has neither
            set_last_error("the least-squares fitness is not available in a batch");
            return CUPSO_ERR_INVALID_ARG;
        }
    }
    if (n_swarms == 0) return CUPSO_OK;

    BatchRun run, prun;   // the swarms with a launch of their own, those in panels
    cudaStream_t own = nullptr, side = nullptr;
    cudaEvent_t handover = nullptr;
    if (cuda_stream) {
        run.st = static_cast<cudaStream_t>(cuda_stream);
    } else {
        cudaError_t e = cudaStreamCreateWithFlags(&own, cudaStreamNonBlocking);
        if (e != cudaSuccess) return set_cuda_error(e, "cudaStreamCreate"), CUPSO_ERR_CUDA;
        run.st = own;
    }
    int first = CUPSO_OK;
    auto note = [&](int rc) {
        if (rc != CUPSO_OK && first == CUPSO_OK) first = rc;
    };

    std::vector<int> batched;
    for (int k = 0; k < n_swarms; ++k) {
        if (problems[k].D >= 3) {
            batched.push_back(k);
        } else {
            note(solve_one_plain(problems[k], iters, results[k], run.st));
        }
    }
    const int nb = (int)batched.size();
    void* arena = nullptr;
    int rc = CUPSO_OK;
    do {
        if (nb == 0) break;
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&run.num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = prepare_batch();
        if (e == cudaSuccess) e = prepare_batch_panel();
        if (e != cudaSuccess) { set_cuda_error(e, "batch setup"); rc = CUPSO_ERR_CUDA; break; }

        // Arena: per-swarm planes, then gbest positions, keys, words, flags, descriptors, units, counters.
        // CUPSO_BATCH_KERNEL=tiled|streaming keeps every swarm out of the panels and fixes
        // the kernel (for tests and measurements; all kernels give the same bits).
        const char* force = std::getenv("CUPSO_BATCH_KERNEL");
        const bool want_tiled = force && std::strcmp(force, "tiled") == 0;
        const bool want_stream = force && std::strcmp(force, "streaming") == 0;
        const size_t A = 256;
        // Panels from kBatchPanelMinD dimensions (the ring's look-ahead) to 65,536
        // particles: 16 swarms of 50,000 x 128 take 378 us an iteration there and 413 out of
        // them, 8 of 100,000 x 96 317 and 311 (with the limit on D
        // it also keeps offsets of 16 bytes in 32 bits). And not where particles are too few to fill the chip and the dimensions
        // many: a particle's panels follow one another, about 0.9 us each, where the tiled
        // kernel spreads them over a CTA -- 256 dimensions, 4,000 particles in all: 26.5 us
        // and 20.9; 8,000: 28.3 and 34.4; 64 dimensions: 11.4 and 17.7.
        std::vector<char> panel(nb);
        long long rest = 0, padded = 0;   // units of 128 particles out of the panels, and of swarms that padding slows
        std::vector<char> pad(nb);
        for (int j = 0; j < nb; ++j) {
            const cupso_problem& p = problems[batched[j]];
            panel[j] = !want_tiled && !want_stream && p.D >= kBatchPanelMinD && p.D <= 65536 &&
                       p.N <= 65536;
            const int past = (p.D + 7) / 8 * 8 - p.D;
            pad[j] = panel[j] && past * 100ll > (p.N <= 8192 ? 5ll : 1ll) * p.D;
            (panel[j] ? padded : rest) += !panel[j] || pad[j] ? (p.N + 127) / 128 : 0;
        }
        // A panel partly used moves its unused dimensions too. Where memory bounds the batch
        // either way, swarms that it adds more than 5 % to (1 % of long rows, which the
        // streaming kernel moves best) stay out: when with those that stay out anyway there
        // are units of 128 particles for five quarters of the streaming kernel's warps (16 an SM). 500
        // swarms of up to 20000 x 25 to 32: 618 us an iteration out of the panels, 700 in
        // them; 100 of up to 60000 x 30 to 60 528 and 600. With fewer units the
        // panels' shorter ones win all the same: 200 of up to 4000 x 3 to 256 317 and 231.
        if (rest + padded >= 20ll * run.num_sms)
            for (int j = 0; j < nb; ++j)
                if (pad[j]) panel[j] = 0;
        long long panel_pd = 0, shallow_pd = 0;
        int panel_maxD = 0;
        for (int j = 0; j < nb; ++j) {
            const cupso_problem& p = problems[batched[j]];
            if (!panel[j]) continue;
            panel_pd += (long long)p.N * p.D;
            if (p.D < kBatchPanelDeepD) shallow_pd += (long long)p.N * p.D;
            panel_maxD = std::max(panel_maxD, p.D);
        }
        // the deep ring from about 300 swarms of 4000 x 130 on, where few are too narrow for it
        const bool deep = panel_pd >= (160ll << 20) && shallow_pd * 16 <= panel_pd;
        if (deep)
            for (int j = 0; j < nb; ++j)
                if (problems[batched[j]].D < kBatchPanelDeepD) panel[j] = 0;
        if (panel_maxD > 64 && panel_pd < 6144ll * panel_maxD) panel.assign(nb, 0);
        std::vector<int> rows(nb);   // dimensions the state has room for
        std::vector<size_t> o_state(nb), o_G(nb), o_flag(nb);
        std::vector<int> Np(nb), tileP(nb);
        std::vector<unsigned> ntiles(nb);
        size_t off, total_units, panel_units, sumG, sumFlag, total_tiles;
        int nlegacy, minD, maxD;
        long long total_pd;
        size_t o_Gall, o_keys, o_words, o_flags, o_desc, o_units, o_punits, o_tunits, o_tileP, o_ntiles, o_ctr;
        auto place = [&](size_t bytes) {
            const size_t o = off;
            off = up(off + bytes, A);
            return o;
        };
        auto layout = [&] {
            off = total_units = panel_units = sumG = sumFlag = total_tiles = 0;
            nlegacy = maxD = 0;
            minD = 1 << 30;
            total_pd = 0;
            for (int j = 0; j < nb; ++j) {
                const cupso_problem& p = problems[batched[j]];
                Np[j] = (p.N + kPad - 1) / kPad * kPad;
                rows[j] = panel[j] ? (p.D + 7) / 8 * 8 : p.D;
                o_state[j] = place(sizeof(float) * ((size_t)3 * rows[j] * Np[j] + Np[j]));
                o_G[j] = sumG = up(sumG, 4);   // 16-byte rows
                sumG += 2 * (size_t)rows[j];
                o_flag[j] = sumFlag;
                sumFlag += (size_t)Np[j];
                if (panel[j]) {
                    panel_units += (size_t)Np[j] / 16;
                    continue;
                }
                ++nlegacy;
                total_units += (size_t)Np[j] / 128;
                tileP[j] = batch_tile_particles(p.D);
                ntiles[j] = tileP[j] > 0 ? (unsigned)((p.N + tileP[j] - 1) / tileP[j]) : 0u;
                total_tiles += ntiles[j];
                minD = std::min(minD, p.D);
                maxD = std::max(maxD, p.D);
                total_pd += (long long)p.N * p.D;
            }
            o_Gall = place(sizeof(float) * sumG);
            o_keys = place(sizeof(unsigned long long) * 2 * nb);
            o_words = place(sizeof(unsigned int) * 4 * nb);
            o_flags = place(sumFlag);
            o_desc = place(sizeof(BatchSwarm) * nb);
            o_units = place(sizeof(uint2) * total_units);
            o_punits = place(sizeof(uint2) * panel_units);
            o_tunits = place(sizeof(uint2) * std::max<size_t>(total_tiles, 1));
            o_tileP = place(sizeof(int) * nb);
            o_ntiles = place(sizeof(unsigned) * nb);
            o_ctr = place(128);
        };
        layout();
        e = cudaMalloc(&arena, off);
        if (e == cudaErrorMemoryAllocation && nlegacy < nb) {
            // without the room that whole panels take
            cudaGetLastError();
            panel.assign(nb, 0);
            layout();
            e = cudaMalloc(&arena, off);
        }
        if (e != cudaSuccess) { set_cuda_error(e, "cudaMalloc (batch arena)"); rc = e == cudaErrorMemoryAllocation ? CUPSO_ERR_OOM : CUPSO_ERR_CUDA; break; }
        char* base = static_cast<char*>(arena);
        float* Gall = reinterpret_cast<float*>(base + o_Gall);
        unsigned long long* keys = reinterpret_cast<unsigned long long*>(base + o_keys);
        unsigned int* words = reinterpret_cast<unsigned int*>(base + o_words);   // done, status, 2 spare
        unsigned char* flags = reinterpret_cast<unsigned char*>(base + o_flags);
        unsigned int* ctr = reinterpret_cast<unsigned int*>(base + o_ctr);       // work[2], ticket, t; the panels' from 16
        e = cudaMemsetAsync(keys, 0xFF, sizeof(unsigned long long) * 2 * nb, run.st);
        if (e == cudaSuccess) e = cudaMemsetAsync(base + o_words, 0, o_desc - o_words, run.st);
        if (e == cudaSuccess) e = cudaMemsetAsync(ctr, 0, 128, run.st);
        if (e == cudaSuccess) e = cudaMemsetAsync(Gall, 0, sizeof(float) * sumG, run.st);
        if (e != cudaSuccess) { set_cuda_error(e, "cudaMemsetAsync"); rc = CUPSO_ERR_CUDA; break; }

        // The descriptor of every swarm.
        std::vector<BatchSwarm> desc(nb);
        for (int j = 0; j < nb; ++j) {
            const cupso_problem& p = problems[batched[j]];
            float* st = reinterpret_cast<float*>(base + o_state[j]);
            const size_t plane = (size_t)rows[j] * Np[j];
            BatchSwarm& w = desc[j];
            w.x = st;
            w.v = st + plane;
            w.pb = st + 2 * plane;
            w.pf = st + 3 * plane;
            w.pflag = flags + o_flag[j];
            w.G = Gall + o_G[j];
            w.g16 = (uint32_t)(o_G[j] / 4);
            w.gkey = keys + 2 * j;
            w.done = words + 4 * j + 0;
            w.status = words + 4 * j + 1;
            w.N = p.N; w.D = p.D; w.Np = Np[j]; w.fid = p.fitness_id;
            w.Gs = rows[j];
            w.nunits = (unsigned)(Np[j] / (panel[j] ? 16 : 128));
            w.lo = p.bounds.min_pos; w.hi = p.bounds.max_pos; w.vmax = p.bounds.max_v;
            w.w = p.w; w.c1 = p.c1; w.c2 = p.c2;
            w.c1s = std::ldexp(p.c1, -24);
            w.c2s = std::ldexp(p.c2, -24);
            const bool fast_cr = std::ldexp(w.c1s, 24) == p.c1 && std::ldexp(w.c2s, 24) == p.c2 &&
                                 (p.c1 == 0.0f || std::fabs(w.c1s) >= FLT_MIN) &&
                                 (p.c2 == 0.0f || std::fabs(w.c2s) >= FLT_MIN);
            const bool has_cos = p.fitness_id == CUPSO_RASTRIGIN || p.fitness_id == CUPSO_ACKLEY;
            const bool small = std::fabs(p.bounds.min_pos) <= kSmallX && std::fabs(p.bounds.max_pos) <= kSmallX;
            w.fast = (!panel[j] || !has_cos || small) && fast_cr && p.bounds.min_pos != 0.0f && p.bounds.max_pos != 0.0f;
            w.key0 = (uint32_t)(p.seed & 0xFFFFFFFFull);
            w.key1 = (uint32_t)(p.seed >> 32);
            w.swarm = p.swarm_id;
            set_constants(w);
        }

        // Hand-out order: swarms that run the same code (fitness function and
        // arithmetic path) together, so that the warps of an SM share their
        // instructions; within such a class the units with the most dimensions
        // first, swarms of equal D interleaved. The smallest units come last
        // and fill the tail.
        std::vector<int> order(nb);
        for (int j = 0; j < nb; ++j) order[j] = j;
        auto code_of = [&](int j) { return desc[j].fid * 2 + desc[j].fast; };
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
            if (panel[a] != panel[b]) return panel[a] > panel[b];
            if (code_of(a) != code_of(b)) return code_of(a) < code_of(b);
            return desc[a].D > desc[b].D;
        });
        auto same_group = [&](int a, int b) {
            return panel[a] == panel[b] && code_of(a) == code_of(b) && desc[a].D == desc[b].D;
        };
        // (swarm, unit) pairs of the swarms in panels or of the others, `count(j)` of each
        auto hand_out = [&](bool panels, size_t total, auto count) {
            std::vector<uint2> out;
            out.reserve(total);
            for (size_t pos = 0; pos < (size_t)nb;) {
                size_t endg = pos;
                while (endg < (size_t)nb && same_group(order[endg], order[pos])) ++endg;
                if ((panel[order[pos]] != 0) == panels) {
                    unsigned most = 0;
                    for (size_t q = pos; q < endg; ++q) most = std::max(most, count(order[q]));
                    for (unsigned u = 0; u < most; ++u)
                        for (size_t q = pos; q < endg; ++q)
                            if (u < count(order[q])) out.push_back(make_uint2((unsigned)order[q], u));
                }
                pos = endg;
            }
            return out;
        };
        auto units_of = [&](int j) { return desc[j].nunits; };
        const std::vector<uint2> units = hand_out(false, total_units, units_of);
        const std::vector<uint2> punits = hand_out(true, panel_units, units_of);
        e = cudaMemcpyAsync(base + o_desc, desc.data(), sizeof(BatchSwarm) * nb, cudaMemcpyHostToDevice, run.st);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(base + o_units, units.data(), sizeof(uint2) * units.size(), cudaMemcpyHostToDevice,
                                run.st);
        if (e == cudaSuccess && !punits.empty())
            e = cudaMemcpyAsync(base + o_punits, punits.data(), sizeof(uint2) * punits.size(), cudaMemcpyHostToDevice,
                                run.st);
        if (e != cudaSuccess) { set_cuda_error(e, "cudaMemcpyAsync"); rc = CUPSO_ERR_CUDA; break; }
        run.dev.G = Gall;
        run.dev.swarms = reinterpret_cast<const BatchSwarm*>(base + o_desc);
        run.dev.units = reinterpret_cast<const uint2*>(base + o_units);
        run.dev.nunits = (unsigned)units.size();
        run.dev.work = ctr;
        run.dev.ticket = ctr + 2;
        run.dev.t_dev = ctr + 3;

        prun.num_sms = run.num_sms;
        prun.dev = run.dev;
        prun.dev.units = reinterpret_cast<const uint2*>(base + o_punits);
        prun.dev.nunits = (unsigned)punits.size();
        prun.dev.work = ctr + 16;
        prun.dev.ticket = ctr + 18;
        prun.dev.t_dev = ctr + 19;
        const Shape pshape{-1, deep ? 1 : 0,
                           prun.dev.nunits ? batch_panel_grid(prun.dev.nunits, deep, run.num_sms) : 0};

        // Step 1 of every swarm, one launch for each kind.
        e = cudaSuccess;
        if (prun.dev.nunits) e = launch_batch_panel_init(prun.dev, run.num_sms, run.st);
        if (e == cudaSuccess && run.dev.nunits) e = launch_batch_init(run.dev, run.num_sms * 4, run.st);
        if (e != cudaSuccess) { set_cuda_error(e, "batch init launch"); rc = CUPSO_ERR_CUDA; break; }

        // The tiled kernel's units in the same order.
        const bool tiled_ok = nlegacy > 0 && maxD <= kTiledItems;
        std::vector<uint2> tunits;
        if (tiled_ok) {
            tunits = hand_out(false, total_tiles, [&](int j) { return ntiles[j]; });
            e = cudaMemcpyAsync(base + o_tunits, tunits.data(), sizeof(uint2) * tunits.size(), cudaMemcpyHostToDevice,
                                run.st);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(base + o_tileP, tileP.data(), sizeof(int) * nb, cudaMemcpyHostToDevice, run.st);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(base + o_ntiles, ntiles.data(), sizeof(unsigned) * nb, cudaMemcpyHostToDevice,
                                    run.st);
            if (e != cudaSuccess) { set_cuda_error(e, "cudaMemcpyAsync"); rc = CUPSO_ERR_CUDA; break; }
            run.tiles.units = reinterpret_cast<const uint2*>(base + o_tunits);
            run.tiles.nunits = (unsigned)tunits.size();
            run.tiles.P = reinterpret_cast<const int*>(base + o_tileP);
            run.tiles.ntiles = reinterpret_cast<const unsigned*>(base + o_ntiles);
        }

        // Launch shapes to try: ring depth 4 needs three dimension pairs everywhere.
        std::vector<Shape> cand;
        if ((minD + 1) / 2 >= 3) cand.push_back(Shape{4, 2, batch_blocks_per_sm(4, 2)});
        cand.push_back(Shape{3, 2, batch_blocks_per_sm(3, 2)});
        cand.push_back(Shape{3, 3, batch_blocks_per_sm(3, 3)});
        if (tiled_ok) cand.push_back(Shape{0, 0, batch_tiled_blocks_per_sm()});
        const auto key = std::make_tuple(nlegacy, total_pd, minD, maxD);
        Shape best = cand[0];
        bool known = nlegacy == 0;
        if (!known) {
            std::lock_guard<std::mutex> lk(g_tune_mutex);
            auto it = g_tuned.find(key);
            if (it != g_tuned.end()) { best = it->second; known = true; }
        }
        if (want_tiled && !tiled_ok) { set_last_error("CUPSO_BATCH_KERNEL=tiled: D too large"); rc = CUPSO_ERR_UNSUPPORTED; break; }
        if (want_tiled || want_stream) {
            for (const Shape& sh : cand)
                if ((sh.stages == 0) == want_tiled) { best = sh; break; }
            known = true;
        }
        int done_iters = 0;
        const int probe = 2;
        if (!known && iters >= (int)cand.size() * probe * 2) {
            float best_ms = 1e30f;
            cudaEvent_t ev0, ev1;
            cudaEventCreate(&ev0);
            cudaEventCreate(&ev1);
            for (const Shape& sh : cand) {
                cudaEventRecord(ev0, run.st);
                for (int k = 0; k < probe && rc == CUPSO_OK; ++k) {
                    e = run.launch(sh);
                    if (e != cudaSuccess) { set_cuda_error(e, "batch launch"); rc = CUPSO_ERR_CUDA; }
                }
                cudaEventRecord(ev1, run.st);
                cudaEventSynchronize(ev1);
                float ms = 0.f;
                cudaEventElapsedTime(&ms, ev0, ev1);
                if (rc == CUPSO_OK && ms < best_ms) { best_ms = ms; best = sh; }
                done_iters += probe;
            }
            cudaEventDestroy(ev0);
            cudaEventDestroy(ev1);
            if (rc == CUPSO_OK) {
                std::lock_guard<std::mutex> lk(g_tune_mutex);
                g_tuned[key] = best;
            }
        }
        if (rc != CUPSO_OK) break;
        // Neither kind waits for the other: with both, the panels advance on a stream
        // of their own, from here until the results are read.
        prun.st = run.st;
        if (prun.dev.nunits && run.dev.nunits) {
            e = cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&handover, cudaEventDisableTiming);
            if (e == cudaSuccess) e = cudaEventRecord(handover, run.st);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(side, handover, 0);
            if (e != cudaSuccess) { set_cuda_error(e, "batch streams"); rc = CUPSO_ERR_CUDA; break; }
            prun.st = side;
        }
        if (prun.dev.nunits) rc = prun.run(pshape, iters);
        if (rc == CUPSO_OK && run.dev.nunits) rc = run.run(best, iters - done_iters);
        if (rc != CUPSO_OK) break;
        if (side) {
            e = cudaEventRecord(handover, side);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(run.st, handover, 0);
            if (e != cudaSuccess) { set_cuda_error(e, "batch streams"); rc = CUPSO_ERR_CUDA; break; }
        }

        // Results: gbest key, position and status of every swarm.
        std::vector<unsigned long long> hkeys(2 * (size_t)nb);
        std::vector<float> hG(sumG);
        std::vector<unsigned int> hw(4 * (size_t)nb);
        e = cudaMemcpyAsync(hkeys.data(), keys, sizeof(unsigned long long) * 2 * nb, cudaMemcpyDeviceToHost, run.st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(hG.data(), Gall, sizeof(float) * sumG, cudaMemcpyDeviceToHost, run.st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(hw.data(), words, sizeof(unsigned) * 4 * nb, cudaMemcpyDeviceToHost, run.st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(run.st);
        if (e != cudaSuccess) { set_cuda_error(e, "batch results"); rc = CUPSO_ERR_CUDA; break; }
        const int cur = iters & 1;
        for (int j = 0; j < nb; ++j) {
            cupso_result& r = results[batched[j]];
            const unsigned long long k = hkeys[2 * j + cur];
            r.fit = key_fit(k);
            r.idx = (int64_t)(k & 0xFFFFFFFFull);
            if (r.pos) std::memcpy(r.pos, hG.data() + o_G[j] + (size_t)cur * desc[j].Gs, sizeof(float) * desc[j].D);
            r.status = (hw[4 * j + 1] & kStatusTimeout) ? CUPSO_ERR_DEVICE_TIMEOUT
                       : (hw[4 * j + 1] & kStatusNaN)   ? CUPSO_ERR_NAN
                                                        : CUPSO_OK;
            note(r.status);
        }
    } while (false);
    if (rc != CUPSO_OK) {
        for (int j = 0; j < nb; ++j) results[batched[j]].status = rc;
        note(rc);
    }
    if (side) cudaStreamSynchronize(side);
    if (arena) {
        cudaStreamSynchronize(run.st);
        cudaFree(arena);
    }
    if (handover) cudaEventDestroy(handover);
    if (side) cudaStreamDestroy(side);
    if (own) cudaStreamDestroy(own);
    return first;
}
