// Batched stepping and the autotuners (include/lbm_axi_batch.h).
#include <string.h>

#include <algorithm>
#include <new>
#include <utility>
#include <vector>

#include "lbm_axi_batch.h"
#include "lbm_handle.h"
#include "lbm_launch.h"

using lbm::BatchSolve;
using lbm::Ops;

// How a batch steps: one or three launches over node tiles (lbm_tile.cuh, lbm_phase.cuh), one warp per tile (lbm_march.cuh) or
// the marching kernel of the chosen strip width and CTA slots (lbm_step.cuh).
enum BatchForm { FORM_TILES, FORM_PHASES, FORM_WARPS, FORM_MARCH };

// The form of one (strip, grid) and the work lists it launches over.
struct StepPlan {
    int strip = lbm::kStripWide, grid = 0;
    BatchForm form = FORM_MARCH;
    lbm::TileForm tile = lbm::TILE_NONE;
    lbm::PhaseTile* d_ptiles = nullptr;
    int nptiles = 0, nghost = 0, prows = 0;
    lbm::Tile* d_tiles = nullptr;  // tile plan for (strip, grid)
    int* d_first = nullptr;        // [ncta + 1]
    int ncta = 0, ntiles = 0;
    int kind = 0;  // of the warp march
};

struct lbm_axi_batch {
    int n;
    int precision;
    bool mp, ax;
    int device;
    std::vector<lbm_axi*> solves;
    std::vector<int> cur0;  // each solve's current buffer when the batch was made
    void* d_solves;         // BatchSolve<R>[n]
    lbm::BatchTable<float>* h_table;  // FP32, n <= BatchTable::N: the descriptors as one kernel argument
    StepPlan plan;          // replaced whole (replan), so it is always complete
    int* d_err;             // [n]
    int* h_err;             // pinned [n]
    cudaStream_t stream;
    bool own_stream;
    long long steps;  // batch steps taken; parity = steps & 1
    cudaGraphExec_t graph;  // an even number of steps from parity 0 of the plan
    int graph_steps;
    int pending;
};

namespace {

struct DevGuard {
    int prev = -1;
    explicit DevGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DevGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

template <typename R>
const Params<R>& params_of(const lbm_axi* h);
template <>
const Params<float>& params_of<float>(const lbm_axi* h) {
    return h->pf;
}
template <>
const Params<double>& params_of<double>(const lbm_axi* h) {
    return h->pdd;
}

// FP64 steps by phases at every tuning; FP32 at the default one (wide strips, grid
// 0) by tiles or phases while the batch is small and by warps beyond, at the others by march2.
BatchForm form_of(const lbm_axi_batch* b, const StepPlan& p, long long phase_nodes) {
    if (b->precision == 64) return FORM_PHASES;
    if (p.strip != lbm::kStripWide || p.grid != 0) return FORM_MARCH;
    if (p.tile != lbm::TILE_NONE) return FORM_TILES;
    return lbm_by_phases(32, phase_nodes) ? FORM_PHASES : FORM_WARPS;
}

void release(StepPlan& p) {
    if (p.d_tiles) cudaFree(p.d_tiles);
    if (p.d_first) cudaFree(p.d_first);
    if (p.d_ptiles) cudaFree(p.d_ptiles);
    p = StepPlan();
}

// The device's table of descriptors and the kernel argument that holds it when it fits (may throw).
template <typename R>
cudaError_t upload_solves(lbm_axi_batch* b) {
    std::vector<BatchSolve<R>> hs(b->n);
    for (int i = 0; i < b->n; i++) hs[i] = lbm_handle_solve<R>(b->solves[i], params_of<R>(b->solves[i]), b->cur0[i]);
    if constexpr (sizeof(R) == 4) {
        if (b->h_table)
            for (int i = 0; i < b->n; i++) b->h_table->s[i] = hs[i];
    }
    const cudaError_t e = cudaMemcpyAsync(b->d_solves, hs.data(), sizeof(BatchSolve<R>) * b->n, cudaMemcpyHostToDevice,
                                          b->stream);
    return e == cudaSuccess ? cudaStreamSynchronize(b->stream) : e;
}

// Fill in the plan of p.strip and p.grid (may throw, device lists allocated so far in p).
template <typename R>
cudaError_t make_plan(const lbm_axi_batch* b, StepPlan& p) {
    std::vector<int> nz(b->n), nr(b->n);
    long long nodes = 0, phase_nodes = 0;
    for (int i = 0; i < b->n; i++) {
        nz[i] = b->solves[i]->nz;
        nr[i] = b->solves[i]->nr;
        nodes += (long long)nz[i] * nr[i];
        phase_nodes += lbm::phase_nodes(nz[i], nr[i]);
    }
    p.tile = b->precision == 32 ? lbm::tile_form(nz.data(), nr.data(), b->n, b->mp, b->ax, 0) : lbm::TILE_NONE;
    p.form = form_of(b, p, phase_nodes);
    std::vector<lbm::Tile> tiles;
    std::vector<lbm::PhaseTile> ptiles;
    size_t inner = 0;  // tiles before the ghost rows'
    std::vector<int> first;
    const bool node_tiles = p.form == FORM_PHASES || p.form == FORM_TILES;
    if (node_tiles) {
        int tz = Ops<R>::phase_tile_z();
        p.prows = Ops<R>::phase_rows(nodes);
        if (p.form == FORM_TILES) lbm::tile_size(p.tile, &tz, &p.prows);
        for (int i = 0; i < b->n; i++)
            for (int j = 0; j < nr[i]; j += p.prows)
                for (int k = 0; k < nz[i]; k += tz) ptiles.push_back(lbm::PhaseTile{i, k, j});
        inner = ptiles.size();
        for (int i = 0; i < b->n && b->ax && p.form == FORM_PHASES; i++)
            for (int k = 0; k < nz[i] && b->solves[i]->opts.top_bc != LBM_TOP_PERIODIC; k += tz)
                ptiles.push_back(lbm::PhaseTile{i, k, -2});
    } else if (p.form == FORM_WARPS) {
        const int slots = Ops<float>::warp_slots();
        if (slots <= 0) return cudaErrorInvalidConfiguration;
        if (lbm::plan_warp_tiles(nz.data(), nr.data(), b->n, slots, tiles) != LBM_OK) return cudaErrorMemoryAllocation;
        p.kind = Ops<float>::warp_kind(b->solves[0]->pf);
        for (int i = 1; i < b->n; i++) p.kind = Ops<float>::warp_kind(p.kind, Ops<float>::warp_kind(b->solves[i]->pf));
    } else {
        const int slots = p.grid > 0 ? p.grid : Ops<R>::batch_resident_ctas(p.strip);
        if (slots <= 0) return cudaErrorInvalidConfiguration;
        if (lbm::plan_tiles(nz.data(), nr.data(), b->n, p.strip, slots, tiles, first, nullptr) != LBM_OK)
            return cudaErrorMemoryAllocation;
    }
    cudaError_t e = cudaSuccess;
    auto put = [&](void** d, const void* from, size_t bytes) {
        if (bytes == 0) return;
        if (e == cudaSuccess) e = cudaMalloc(d, bytes);
        if (e == cudaSuccess) e = cudaMemcpyAsync(*d, from, bytes, cudaMemcpyHostToDevice, b->stream);
    };
    put((void**)&p.d_ptiles, ptiles.data(), ptiles.size() * sizeof(lbm::PhaseTile));
    put((void**)&p.d_tiles, tiles.data(), tiles.size() * sizeof(lbm::Tile));
    put((void**)&p.d_first, first.data(), first.size() * sizeof(int));
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return e;
    p.nptiles = (int)inner;
    p.nghost = (int)(ptiles.size() - inner);
    p.ncta = first.empty() ? 0 : (int)first.size() - 1;
    p.ntiles = (int)tiles.size();
    return cudaSuccess;
}

// The plan of (strip, grid) in place of the present one, which stays if anything fails.
cudaError_t replan(lbm_axi_batch* b, int strip, int grid) {
    StepPlan p;
    p.strip = strip;
    p.grid = grid;
    cudaError_t e;
    try {
        e = b->precision == 32 ? make_plan<float>(b, p) : make_plan<double>(b, p);
    } catch (...) {
        cudaStreamSynchronize(b->stream);  // copies from the lists that went away
        e = cudaErrorMemoryAllocation;
    }
    if (e == cudaSuccess) {
        if (b->graph) cudaGraphExecDestroy(b->graph);  // holds the old plan's pointers
        b->graph = nullptr;
        std::swap(b->plan, p);
    }
    release(p);
    if (e != cudaSuccess) cudaGetLastError();  // not the next launch's error
    return e;
}

cudaError_t launch(lbm_axi_batch* b, int parity) {
    const StepPlan& p = b->plan;
    if (!p.d_ptiles && !p.d_tiles) return cudaErrorInvalidConfiguration;
    if (b->precision == 64)
        return Ops<double>::phase_step_many(static_cast<const BatchSolve<double>*>(b->d_solves), p.d_ptiles, p.nptiles,
                                            p.nghost, p.prows, b->mp, b->ax, parity, b->d_err, b->stream);
    const BatchSolve<float>* solves = static_cast<const BatchSolve<float>*>(b->d_solves);
    if (p.form == FORM_WARPS)
        return Ops<float>::step_warp_many(solves, p.kind, p.d_tiles, p.ntiles, b->mp, b->ax, parity, b->d_err, b->stream);
    if (p.form == FORM_TILES)
        return Ops<float>::tile_step_many(p.tile, solves, p.d_ptiles, p.nptiles, b->ax, parity, b->d_err, b->stream);
    if (p.form == FORM_PHASES)
        return Ops<float>::phase_step_many(solves, p.d_ptiles, p.nptiles, p.nghost, p.prows, b->mp, b->ax, parity, b->d_err,
                                           b->stream);
    if (b->h_table)  // n <= BatchTable::N: parameters through the constant bank
        return Ops<float>::step_table(*b->h_table, p.d_tiles, p.d_first, p.ncta, b->mp, b->ax, parity, p.strip,
                                      b->d_err, b->stream);
    return Ops<float>::step_batch(solves, p.d_tiles, p.d_first, p.ncta, b->mp, b->ax, parity, p.strip, b->d_err,
                                  b->stream);
}

// Steps per graph replay: small batches take a few us per step, which a replay would otherwise spend on itself.
int graph_steps_of(const lbm_axi_batch* b) { return b->plan.form == FORM_TILES || b->plan.form == FORM_PHASES ? 16 : 2; }

int build_graph(lbm_axi_batch* b) {
    if (b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return LBM_ERR_CUDA;
    b->graph_steps = graph_steps_of(b);
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < b->graph_steps && e == cudaSuccess; i++) e = launch(b, i & 1);
    cudaError_t e2 = cudaStreamEndCapture(b->stream, &g);
    if (e != cudaSuccess || e2 != cudaSuccess || !g) {
        if (g) cudaGraphDestroy(g);
        cudaGetLastError();
        return LBM_ERR_CUDA;
    }
    cudaError_t e3 = cudaGraphInstantiate(&b->graph, g, 0);
    cudaGraphDestroy(g);
    if (e3 != cudaSuccess) {
        b->graph = nullptr;
        return LBM_ERR_CUDA;
    }
    return LBM_OK;
}

// Point every handle at the buffer holding its latest state.
void sync_handles(lbm_axi_batch* b) {
    for (int i = 0; i < b->n; i++) b->solves[i]->cur = b->cur0[i] ^ (int)(b->steps & 1);
}

void release(lbm_axi_batch* b) {
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->d_solves) cudaFree(b->d_solves);
    release(b->plan);
    if (b->d_err) cudaFree(b->d_err);
    if (b->h_err) cudaFreeHost(b->h_err);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    delete b->h_table;
}

// Time `trials` launches of fn on stream s (ms per launch), non-destructively.
template <typename F>
float time_launches(cudaStream_t s, int trials, F&& fn) {
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return -1.f;
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return -1.f;
    }
    bool ok = fn() == cudaSuccess;  // warm-up launch
    ok = ok && cudaEventRecord(e0, s) == cudaSuccess;
    for (int t = 0; t < trials && ok; t++) ok = fn() == cudaSuccess;
    ok = ok && cudaEventRecord(e1, s) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess;
    float ms = -1.f;
    if (ok) cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return ok ? ms / trials : -1.f;
}

}  // namespace

extern "C" {

int lbm_axi_batch_create(lbm_axi* const* solves, int n, void* stream, lbm_axi_batch** out) {
    if (!out || !solves || n < 1) return LBM_ERR_INVALID_ARG;
    *out = nullptr;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LBM_ERR_CUDA;
    const lbm_axi* h0 = solves[0];
    if (!h0) return LBM_ERR_INVALID_ARG;
    for (int i = 0; i < n; i++) {
        const lbm_axi* h = solves[i];
        if (!h || !h->initialized || h->device != dev || h->precision != h0->precision ||
            h->nr < lbm::kStepMinRows || h->opts.multiphase != h0->opts.multiphase ||
            h->opts.axis_terms != h0->opts.axis_terms || unbatchable(h))
            return LBM_ERR_INVALID_ARG;
        for (int k = 0; k < i; k++)
            if (solves[k] == h) return LBM_ERR_INVALID_ARG;
    }
    lbm_axi_batch* b = new (std::nothrow) lbm_axi_batch;
    if (!b) return LBM_ERR_OOM;
    b->n = n;
    b->precision = h0->precision;
    b->mp = h0->opts.multiphase != 0;
    b->ax = h0->opts.axis_terms != 0;
    b->device = dev;
    b->d_solves = nullptr;
    b->h_table = nullptr;
    b->d_err = nullptr;
    b->h_err = nullptr;
    b->stream = nullptr;
    b->own_stream = false;
    b->steps = 0;
    b->graph = nullptr;
    b->graph_steps = 0;
    b->pending = LBM_OK;
    try {
        b->solves.assign(solves, solves + n);
        b->cur0.resize(n);
    } catch (...) {
        delete b;
        return LBM_ERR_OOM;
    }
    for (int i = 0; i < n; i++) {
        // finish whatever the solve's own stream was doing before the batch takes over
        if (cudaStreamSynchronize(solves[i]->stream) != cudaSuccess) {
            delete b;
            return LBM_ERR_CUDA;
        }
        b->cur0[i] = solves[i]->cur;
    }
    if (b->precision == 32 && n <= lbm::BatchTable<float>::N) {
        b->h_table = new (std::nothrow) lbm::BatchTable<float>();
        if (!b->h_table) {
            delete b;
            return LBM_ERR_OOM;
        }
    }
    const size_t ssz = b->precision == 32 ? sizeof(BatchSolve<float>) : sizeof(BatchSolve<double>);
    bool ok = cudaMalloc(&b->d_solves, ssz * n) == cudaSuccess &&
              cudaMalloc(&b->d_err, sizeof(int) * n) == cudaSuccess &&
              cudaMallocHost(&b->h_err, sizeof(int) * n) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        release(b);
        delete b;
        return LBM_ERR_OOM;
    }
    if (stream) {
        b->stream = static_cast<cudaStream_t>(stream);
    } else {
        if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) {
            release(b);
            delete b;
            return LBM_ERR_CUDA;
        }
        b->own_stream = true;
    }
    cudaError_t e = cudaMemsetAsync(b->d_err, 0, sizeof(int) * n, b->stream);
    try {
        if (e == cudaSuccess) e = b->precision == 32 ? upload_solves<float>(b) : upload_solves<double>(b);
    } catch (...) {
        e = cudaErrorMemoryAllocation;
    }
    if (e == cudaSuccess) e = replan(b, lbm::kStripWide, 0);
    if (e != cudaSuccess) {
        release(b);
        delete b;
        return LBM_ERR_CUDA;
    }
    *out = b;
    return LBM_OK;
}

int lbm_axi_batch_step_async(lbm_axi_batch* b, long long nsteps) {
    if (!b || nsteps < 0) return LBM_ERR_INVALID_ARG;
    DevGuard g(b->device);
    cudaError_t e = cudaSuccess;
    if (nsteps > 0 && (b->steps & 1)) {
        e = launch(b, 1);
        b->steps++;
        nsteps--;
    }
    if (e == cudaSuccess && nsteps >= graph_steps_of(b)) {
        if (!b->graph) {
            int rc = build_graph(b);
            if (rc != LBM_OK) return rc;
        }
        while (nsteps >= b->graph_steps && e == cudaSuccess) {
            e = cudaGraphLaunch(b->graph, b->stream);
            b->steps += b->graph_steps;
            nsteps -= b->graph_steps;
        }
    }
    while (e == cudaSuccess && nsteps > 0) {
        e = launch(b, (int)(b->steps & 1));
        b->steps++;
        nsteps--;
    }
    sync_handles(b);
    if (e != cudaSuccess) {
        b->pending = LBM_ERR_CUDA;
        return LBM_ERR_CUDA;
    }
    return LBM_OK;
}

int lbm_axi_batch_status(lbm_axi_batch* b, int* status) {
    if (!b) return LBM_ERR_INVALID_ARG;
    DevGuard g(b->device);
    if (cudaMemcpyAsync(b->h_err, b->d_err, sizeof(int) * b->n, cudaMemcpyDeviceToHost, b->stream) != cudaSuccess ||
        cudaStreamSynchronize(b->stream) != cudaSuccess)
        return LBM_ERR_CUDA;
    int any = LBM_OK;
    for (int i = 0; i < b->n; i++) {
        const int s = b->h_err[i] ? LBM_ERR_UNPHYSICAL : LBM_OK;
        if (status) status[i] = s;
        if (s != LBM_OK) any = s;
    }
    return any;
}

int lbm_axi_batch_sync(lbm_axi_batch* b) {
    if (!b) return LBM_ERR_INVALID_ARG;
    int rc = lbm_axi_batch_status(b, nullptr);
    if (b->pending != LBM_OK) rc = b->pending;
    b->pending = LBM_OK;
    return rc;
}

int lbm_axi_batch_step(lbm_axi_batch* b, long long nsteps) {
    int rc = lbm_axi_batch_step_async(b, nsteps);
    if (rc != LBM_OK) {
        if (b && rc != LBM_ERR_INVALID_ARG) lbm_axi_batch_sync(b);
        return rc;
    }
    return lbm_axi_batch_sync(b);
}

int lbm_axi_batch_steps(const lbm_axi_batch* b, long long* steps) {
    if (!b || !steps) return LBM_ERR_INVALID_ARG;
    *steps = b->steps;
    return LBM_OK;
}

int lbm_axi_batch_get_tuning(const lbm_axi_batch* b, lbm_axi_batch_tuning* t) {
    if (!b || !t) return LBM_ERR_INVALID_ARG;
    t->strip = b->plan.strip;
    t->grid = b->plan.grid;
    return LBM_OK;
}

int lbm_axi_batch_set_tuning(lbm_axi_batch* b, const lbm_axi_batch_tuning* t) {
    if (!b || !t || (t->strip != lbm::kStripNarrow && t->strip != lbm::kStripWide) || t->grid < 0) return LBM_ERR_INVALID_ARG;
    DevGuard g(b->device);
    if (cudaStreamSynchronize(b->stream) != cudaSuccess) return LBM_ERR_CUDA;
    if ((t->strip != b->plan.strip || t->grid != b->plan.grid) && replan(b, t->strip, t->grid) != cudaSuccess)
        return LBM_ERR_CUDA;
    return LBM_OK;
}

int lbm_axi_batch_autotune(lbm_axi_batch* b, int trials, lbm_axi_batch_tuning* chosen) {
    if (!b || trials < 1) return LBM_ERR_INVALID_ARG;
    DevGuard g(b->device);
    const int parity = (int)(b->steps & 1);
    float best = -1.f;
    lbm_axi_batch_tuning bt = {b->plan.strip, b->plan.grid};
    const int strips[2] = {lbm::kStripNarrow, lbm::kStripWide};
    // the solves' error words before the trials (trial results are discarded; a
    // solve that had already failed stays failed, and skipped, afterwards)
    if (cudaMemcpyAsync(b->h_err, b->d_err, sizeof(int) * b->n, cudaMemcpyDeviceToHost, b->stream) != cudaSuccess ||
        cudaStreamSynchronize(b->stream) != cudaSuccess)
        return LBM_ERR_CUDA;
    std::vector<int> err0;
    try {
        err0.assign(b->h_err, b->h_err + b->n);
    } catch (...) {
        return LBM_ERR_OOM;
    }
    for (int si = 0; si < 2; si++) {
        const int strip = strips[si];
        // FP64 has one form, whatever the strip and the slots
        const int resident = b->precision == 32 ? Ops<float>::batch_resident_ctas(strip) : 0;
        if (b->precision == 32 ? resident <= 0 : strip != lbm::kStripWide) continue;
        const int grids[2] = {0, 2 * resident};
        for (int gi = 0; gi < (resident > 0 ? 2 : 1); gi++) {
            lbm_axi_batch_tuning t = {strip, grids[gi]};
            if (lbm_axi_batch_set_tuning(b, &t) != LBM_OK) return LBM_ERR_CUDA;
            const float ms = time_launches(b->stream, trials, [&] { return launch(b, parity); });
            if (ms > 0 && (best < 0 || ms < best)) {
                best = ms;
                bt.strip = strip;
                bt.grid = grids[gi];
            }
        }
    }
    if (best < 0) return LBM_ERR_CUDA;
    if (lbm_axi_batch_set_tuning(b, &bt) != LBM_OK) return LBM_ERR_CUDA;
    if (cudaMemcpyAsync(b->d_err, err0.data(), sizeof(int) * b->n, cudaMemcpyHostToDevice, b->stream) !=
            cudaSuccess ||
        cudaStreamSynchronize(b->stream) != cudaSuccess)
        return LBM_ERR_CUDA;
    if (chosen) *chosen = bt;
    return LBM_OK;
}

int lbm_axi_autotune(lbm_axi* h, int trials, lbm_axi_tuning* chosen) {
    if (!h || trials < 1) return LBM_ERR_INVALID_ARG;
    if (!h->initialized) return LBM_ERR_STATE;
    DevGuard g(h->device);
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return LBM_ERR_CUDA;
    const int c = h->cur;
    float best = -1.f;
    lbm_axi_tuning bt = {h->path, h->rows_per_cta};
    auto fused = [&](int rows) {
        return h->precision == 32
                   ? Ops<float>::step(h->pf, (const float*)h->f[c], (float*)h->f[c ^ 1], rows, h->derr, h->stream)
                   : Ops<double>::step(h->pdd, (const double*)h->f[c], (double*)h->f[c ^ 1], rows, h->derr,
                                       h->stream);
    };
    auto split = [&]() {
        cudaError_t e;
        if (h->precision == 32) {
            const lbm::LinkPlanes<float> lk = link_planes<float>(h, c);
            e = Ops<float>::density(h->pf, (const float*)h->f[c], (float*)h->aux, h->derr, h->stream, lk);
            if (e == cudaSuccess)
                e = Ops<float>::update(h->pf, (const float*)h->f[c], (float*)h->f[c ^ 1],
                                       (const float*)h->aux, h->stream, lk, guo_of(h));
        } else {
            const lbm::LinkPlanes<double> lk = link_planes<double>(h, c);
            e = Ops<double>::density(h->pdd, (const double*)h->f[c], (double*)h->aux, h->derr, h->stream, lk);
            if (e == cudaSuccess)
                e = Ops<double>::update(h->pdd, (const double*)h->f[c], (double*)h->f[c ^ 1],
                                        (const double*)h->aux, h->stream, lk, guo_of(h));
        }
        return e;
    };
    if (fused_ok(h)) {
        // rows 0: the form the size chooses (every collision variant has it)
        const int rows_list[5] = {0, 32, 64, 144, 256};
        const int nrows = fv_of(h) ? 1 : 5;
        for (int q = 0; q < nrows; q++) {
            const float ms = time_launches(h->stream, trials, [&] {
                return rows_list[q] == 0 ? lbm_handle_step_fused(h, c) : fused(rows_list[q]);
            });
            if (ms > 0 && (best < 0 || ms < best)) {
                best = ms;
                bt.path = LBM_PATH_FUSED;
                bt.rows_per_cta = rows_list[q];
            }
        }
    }
    const float ms = time_launches(h->stream, trials, split);
    if (ms > 0 && (best < 0 || ms < best)) {
        best = ms;
        bt.path = LBM_PATH_SPLIT;
        bt.rows_per_cta = h->rows_per_cta;
    }
    if (best < 0) return LBM_ERR_CUDA;
    if (cudaMemsetAsync(h->derr, 0, sizeof(int), h->stream) != cudaSuccess ||
        cudaStreamSynchronize(h->stream) != cudaSuccess)
        return LBM_ERR_CUDA;
    const int rc = lbm_axi_set_tuning(h, &bt);
    if (rc == LBM_OK && chosen) *chosen = bt;
    return rc;
}

void lbm_axi_batch_destroy(lbm_axi_batch* b) {
    if (!b) return;
    DevGuard g(b->device);
    cudaStreamSynchronize(b->stream);
    sync_handles(b);
    release(b);
    delete b;
}

}  // extern "C"
