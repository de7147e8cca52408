// C ABI of the engine (include/lbm_axi.h): handle lifetime, device memory,
// the step loop (replayed as CUDA-graph chunks), moments and FP64 reductions.
#include <cuda.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <new>
#include <vector>

#include "lbm_axi.h"
#include "lbm_eos_host.h"
#include "lbm_launch.h"

using lbm::Ops;
using lbm::Params;

namespace {

void* (*g_alloc)(size_t, void*) = nullptr;
void (*g_release)(void*, void*) = nullptr;
void* g_alloc_ctx = nullptr;

void* dev_alloc(size_t bytes) {
    if (bytes == 0) bytes = 256;
    if (g_alloc) return g_alloc(bytes, g_alloc_ctx);
    void* p = nullptr;
    return cudaMalloc(&p, bytes) == cudaSuccess ? p : nullptr;
}

void dev_free(void* p, bool via_hook, void* ctx, void (*release)(void*, void*)) {
    if (!p) return;
    if (via_hook) release(p, ctx);
    else cudaFree(p);
}

int pitch_of(int nz) { return (nz + 31) / 32 * 32; }

}  // namespace

#include "lbm_handle.h"

template <typename R>
static cudaError_t step_fused(lbm_axi* h, const Params<R>& p, int c) {
    const bool mp = h->opts.multiphase != 0, ax = h->opts.axis_terms != 0;
    const lbm::BatchSolve<R> s = lbm_handle_solve<R>(h, p, 0);
    const lbm::LinkSets<R> hs{static_cast<const R*>(h->hb[0]), static_cast<R*>(h->hb[1])};
    if constexpr (sizeof(R) == 4)
        if (h->tile != lbm::TILE_NONE) return Ops<R>::tile_step(h->tile, s, ax, c, h->derr, h->stream);
    if (lbm_by_phases(h->precision, lbm::phase_nodes(h->nz, h->nr)))
        return Ops<R>::phase_step(s, hs, mp, ax, c, h->derr, h->stream, fv_of(h));
    if constexpr (sizeof(R) == 4)
        if (fv_of(h) == 0) return Ops<R>::step_warp(s, h->d_tiles, h->ncta, mp, ax, c, h->derr, h->stream);
    return Ops<R>::step_single(s, hs, h->d_tiles, h->d_first, h->ncta, mp, ax, c, h->derr, h->stream, fv_of(h));
}
cudaError_t lbm_handle_step_fused(lbm_axi* h, int c) {
    return h->precision == 32 ? step_fused<float>(h, h->pf, c) : step_fused<double>(h, h->pdd, c);
}

namespace {

template <typename R>
Params<R> make_params(const lbm_axi* h) {
    Params<R> p;
    p.nz = h->nz;
    p.nr = h->nr;
    p.pitch = h->pitch;
    p.axis_a = (R)(h->opts.axis_a_term == LBM_AXIS_A_EXPANSION ? 2.0 : 6.0);
    p.plane = h->plane;
    p.tau_inv = (R)(1.0 / h->tau);
    p.nu = (R)((h->tau - 0.5) / 3.0);
    p.A = (R)h->A;
    p.rho_ref = (R)h->opts.rho_ref;
    p.gz = (R)h->opts.g_z;
    p.eos = h->eos.kind;
    p.T = (R)h->T;
    p.a = (R)h->eos.a;
    p.b = (R)h->eos.b;
    p.Rg = (R)h->eos.R;
    p.lambda = (R)h->eos.lambda;
    p.top = h->opts.top_bc;
    p.axis = h->opts.axis_terms;
    p.multiphase = h->opts.multiphase;
    p.kappa = h->opts.kappa_mode;
    p.hr_sign = h->opts.hr_sign;
    return p;
}

// The FP64 copy used for outputs (moments' P_k, pressure jump) carries the
// reference density as stored in the arithmetic type of the populations.
Params<double> make_params_out(const lbm_axi* h) {
    Params<double> pd = make_params<double>(h);
    if (h->precision == 32) pd.rho_ref = (double)(float)h->opts.rho_ref;
    return pd;
}

double stored_rho_ref(const lbm_axi* h) {
    return h->precision == 32 ? (double)(float)h->opts.rho_ref : h->opts.rho_ref;
}

// One step.  Fused path: kernel (b') reads f[cur] and writes f[cur^1].  Split
// path: kernel (a) on the current populations, kernel (b) into the other buffer.
cudaError_t enqueue_step(lbm_axi* h) {
    const int c = h->cur;
    cudaError_t e;
    if (h->path == LBM_PATH_FUSED && h->rows_per_cta == 0) {
        e = lbm_handle_step_fused(h, c);
        h->cur = c ^ 1;
        return e;
    }
    if (h->path == LBM_PATH_FUSED) {
        if (h->precision == 32)
            e = Ops<float>::step(h->pf, (const float*)h->f[c], (float*)h->f[c ^ 1], h->rows_per_cta, h->derr,
                                 h->stream);
        else
            e = Ops<double>::step(h->pdd, (const double*)h->f[c], (double*)h->f[c ^ 1], h->rows_per_cta, h->derr,
                                  h->stream);
        h->cur = c ^ 1;
        return e;
    }
    if (h->precision == 32) {
        const lbm::LinkPlanes<float> lk = link_planes<float>(h, c);
        e = Ops<float>::density(h->pf, (const float*)h->f[c], (float*)h->aux, h->derr, h->stream, lk);
        if (e == cudaSuccess)
            e = Ops<float>::update(h->pf, (const float*)h->f[c], (float*)h->f[c ^ 1], (const float*)h->aux,
                                   h->stream, lk, guo_of(h));
    } else {
        const lbm::LinkPlanes<double> lk = link_planes<double>(h, c);
        e = Ops<double>::density(h->pdd, (const double*)h->f[c], (double*)h->aux, h->derr, h->stream, lk);
        if (e == cudaSuccess)
            e = Ops<double>::update(h->pdd, (const double*)h->f[c], (double*)h->f[c ^ 1],
                                    (const double*)h->aux, h->stream, lk, guo_of(h));
    }
    h->cur = c ^ 1;
    return e;
}

cudaError_t enqueue_density(lbm_axi* h) {
    if (h->precision == 32)
        return Ops<float>::density(h->pf, (const float*)h->f[h->cur], (float*)h->aux, h->derr, h->stream,
                                   link_planes<float>(h, h->cur));
    return Ops<double>::density(h->pdd, (const double*)h->f[h->cur], (double*)h->aux, h->derr, h->stream,
                                link_planes<double>(h, h->cur));
}

// Graph of an even number of steps starting and ending in buffer 0.
int build_graph(lbm_axi* h, int steps) {
    if (h->graph) {
        cudaGraphExecDestroy(h->graph);
        h->graph = nullptr;
    }
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return LBM_ERR_CUDA;
    const int saved = h->cur;
    h->cur = 0;
    cudaError_t e = cudaSuccess;
    for (int s = 0; s < steps && e == cudaSuccess; s++) e = enqueue_step(h);
    cudaError_t e2 = cudaStreamEndCapture(h->stream, &g);
    h->cur = saved;
    if (e != cudaSuccess || e2 != cudaSuccess || !g) {
        if (g) cudaGraphDestroy(g);
        cudaGetLastError();
        return LBM_ERR_CUDA;
    }
    cudaError_t e3 = cudaGraphInstantiate(&h->graph, g, 0);
    cudaGraphDestroy(g);
    if (e3 != cudaSuccess) {
        h->graph = nullptr;
        return LBM_ERR_CUDA;
    }
    h->graph_steps = steps;
    return LBM_OK;
}

// Steps per graph replay: enough work per launch for tiny grids, at least 2.
int chunk_steps(const lbm_axi* h) {
    const long long cells = (long long)h->nz * h->nr;
    long long c = (4LL << 20) / (cells > 0 ? cells : 1);
    if (c < 2) c = 2;
    if (c > 32) c = 32;
    return (int)(c & ~1LL);
}

// Steps go to the stream one by one where no graph of them can be made or launched: the legacy stream, which
// cannot be captured, and a stream that the caller is capturing.
bool one_by_one(cudaStream_t s) {
    if (s == cudaStreamLegacy) return true;
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) == cudaSuccess) return st != cudaStreamCaptureStatusNone;
    cudaGetLastError();  // not the next launch's error
    return false;
}

int read_error(lbm_axi* h) {
    // one launch that writes the pinned word and clears the device's (a copy and a memset take twice as long)
    if (Ops<float>::take_error(h->derr, h->herr, h->stream) != cudaSuccess) return LBM_ERR_CUDA;
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return LBM_ERR_CUDA;
    return *h->herr ? LBM_ERR_UNPHYSICAL : LBM_OK;
}

// Fields of the current state into device arrays (each may be null) and u into pitched planes (or null).
cudaError_t enqueue_fields(lbm_axi* h, double* rho, double* uz, double* ur, double* p, void* u) {
    if (h->precision == 32)
        return Ops<float>::fields(lbm_handle_solve<float>(h, h->pf, 0), link_planes<float>(h, h->cur), h->pdd, h->cur,
                                  rho, uz, ur, p, static_cast<float*>(u), h->derr, h->stream);
    return Ops<double>::fields(lbm_handle_solve<double>(h, h->pdd, 0), link_planes<double>(h, h->cur), h->pdd, h->cur,
                               rho, uz, ur, p, static_cast<double*>(u), h->derr, h->stream);
}

cudaError_t enqueue_init(lbm_axi* h, const double* rho, const double* uz, const double* ur, const void* phys) {
    if (h->precision == 32)
        return Ops<float>::init(h->pf, stored_rho_ref(h), rho, uz, ur, (float*)h->f[0], h->stream,
                                static_cast<const float*>(phys), h->derr);
    return Ops<double>::init(h->pdd, stored_rho_ref(h), rho, uz, ur, (double*)h->f[0], h->stream,
                             static_cast<const double*>(phys), h->derr);
}

// Memory of this device, [base, base + size).
struct DeviceRange {
    uintptr_t base = 0;
    size_t size = 0;
    // n doubles at p that a kernel may write: all of them in the range, as a copy would check (and a copy takes any
    // address)
    bool holds(const void* p, size_t n) const {
        const uintptr_t at = reinterpret_cast<uintptr_t>(p);
        return at % sizeof(double) == 0 && at >= base && at - base <= size && size - (at - base) >= n * sizeof(double);
    }
};

// The allocation of this device that p lies in (size 0: none, or not known).
DeviceRange allocation_of(const void* p, int device) {
    using F = CUresult (*)(CUdeviceptr*, size_t*, CUdeviceptr);
    static const F range = [] {  // from the driver: the runtime has no call for it
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        const bool ok = cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &q) ==
                            cudaSuccess &&
                        q == cudaDriverEntryPointSuccess;
        if (!ok) cudaGetLastError();
        return ok ? reinterpret_cast<F>(f) : nullptr;
    }();
    DeviceRange r;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return r;
    }
    CUdeviceptr base = 0;
    size_t size = 0;
    if (a.type != cudaMemoryTypeDevice || a.device != device || !range ||
        range(&base, &size, reinterpret_cast<CUdeviceptr>(p)) != CUDA_SUCCESS)
        return r;
    r.base = static_cast<uintptr_t>(base);
    r.size = size;
    return r;
}

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

void release_all(lbm_axi* h) {
    if (h->graph) cudaGraphExecDestroy(h->graph);
    dev_free(h->f[0], h->via_hook, h->hook_ctx, h->hook_release);
    dev_free(h->f[1], h->via_hook, h->hook_ctx, h->hook_release);
    dev_free(h->aux, h->via_hook, h->hook_ctx, h->hook_release);
    dev_free(h->mout, h->via_hook, h->hook_ctx, h->hook_release);
    dev_free(h->partial, h->via_hook, h->hook_ctx, h->hook_release);
    dev_free(h->derr, h->via_hook, h->hook_ctx, h->hook_release);
    dev_free(h->d_tiles, h->via_hook, h->hook_ctx, h->hook_release);
    dev_free(h->d_first, h->via_hook, h->hook_ctx, h->hook_release);
    dev_free(h->hb[0], h->via_hook, h->hook_ctx, h->hook_release);
    dev_free(h->hb[1], h->via_hook, h->hook_ctx, h->hook_release);
    if (h->herr) cudaFreeHost(h->herr);
    if (h->hred) cudaFreeHost(h->hred);
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
}

}  // namespace

extern "C" {

void lbm_axi_default_opts(lbm_axi_opts* o) {
    if (!o) return;
    memset(o, 0, sizeof(*o));
    o->precision = 64;
    o->top_bc = LBM_TOP_FREESLIP;
    o->axis_terms = 1;
    o->multiphase = 1;
    o->kappa_mode = LBM_KAPPA_THERMO;
    o->hr_sign = -1;
    o->rho_ref = 0.0;
    o->g_z = 0.0;
    o->stream = nullptr;
    o->h_eval = LBM_H_LOCAL;
    o->forcing = LBM_FORCING_EDM;
    o->axis_a_term = LBM_AXIS_A_PRINTED;
}

size_t lbm_axi_footprint(int nz, int nr, int precision) {
    if (nz < 1 || nr < 1) return 0;
    const size_t s = precision == 32 ? 4 : 8;
    const size_t plane = (size_t)pitch_of(nz) * nr;
    const size_t n = (size_t)nz * nr;
    return 2 * 9 * plane * s + 4 * plane * s + 4 * n * 8 + 4 * (size_t)lbm::reduce_blocks((long long)n) * 8 + 64;
}

int lbm_axi_create(int nz, int nr, double tau, const lbm_eos* eos, double A, const lbm_axi_opts* opts,
                   lbm_axi** out) {
    if (!out) return LBM_ERR_INVALID_ARG;
    *out = nullptr;
    lbm_axi_opts o;
    if (opts) o = *opts;
    else lbm_axi_default_opts(&o);
    if (nz < 1 || nr < 1 || (long long)nz * nr > (1LL << 31) / 16) return LBM_ERR_INVALID_ARG;
    // the step kernels index a population buffer (9 planes of pitch x nr) with 32-bit offsets
    if (9LL * pitch_of(nz) * nr >= (1LL << 31)) return LBM_ERR_INVALID_ARG;
    if (!(tau > 0.5) || !(tau < 1e6)) return LBM_ERR_INVALID_ARG;
    if (o.precision != 32 && o.precision != 64) return LBM_ERR_INVALID_ARG;
    if (o.top_bc < 0 || o.top_bc > 2 || o.kappa_mode < 0 || o.kappa_mode > 2) return LBM_ERR_INVALID_ARG;
    if (o.hr_sign != 1 && o.hr_sign != -1) return LBM_ERR_INVALID_ARG;
    if (o.h_eval != LBM_H_LOCAL && o.h_eval != LBM_H_LINK_AVG) return LBM_ERR_INVALID_ARG;
    if (o.forcing != LBM_FORCING_EDM && o.forcing != LBM_FORCING_GUO) return LBM_ERR_INVALID_ARG;
    if (o.axis_a_term != LBM_AXIS_A_PRINTED && o.axis_a_term != LBM_AXIS_A_EXPANSION) return LBM_ERR_INVALID_ARG;
    lbm_eos e;
    memset(&e, 0, sizeof(e));
    double T = 0.0, Tc = 0.0;
    if (o.multiphase) {
        if (!eos || (eos->kind != LBM_EOS_VDW && eos->kind != LBM_EOS_CS)) return LBM_ERR_INVALID_ARG;
        e = *eos;
        if (e.kind == LBM_EOS_VDW && !(e.lambda > 0)) return LBM_ERR_INVALID_ARG;
        double rc;
        if (!(e.T_over_Tc > 0) || !lbm::critical_point(e, &Tc, &rc)) return LBM_ERR_INVALID_ARG;
        T = e.T_over_Tc * Tc;
    } else if (eos) {
        e = *eos;
    }
    lbm_axi* h = new (std::nothrow) lbm_axi;
    if (!h) return LBM_ERR_OOM;
    memset(h, 0, sizeof(*h));
    h->nz = nz;
    h->nr = nr;
    h->pitch = pitch_of(nz);
    h->plane = (long long)h->pitch * nr;
    h->precision = o.precision;
    h->tau = tau;
    h->A = A;
    h->eos = e;
    h->T = T;
    h->Tc = Tc;
    h->opts = o;
    h->via_hook = g_alloc != nullptr;
    h->hook_ctx = g_alloc_ctx;
    h->hook_release = g_release;
    if (cudaGetDevice(&h->device) != cudaSuccess ||
        (o.precision == 32 ? Ops<float>::prepare() : Ops<double>::prepare()) != cudaSuccess) {
        cudaGetLastError();
        delete h;
        return LBM_ERR_CUDA;
    }
    const size_t s = o.precision == 32 ? 4 : 8;
    const size_t plane_bytes = (size_t)h->plane * s;
    h->f[0] = dev_alloc(9 * plane_bytes);
    h->f[1] = dev_alloc(9 * plane_bytes);
    h->aux = dev_alloc(4 * plane_bytes);
    h->mout = (double*)dev_alloc(4 * (size_t)nz * nr * sizeof(double));
    h->partial = (double*)dev_alloc(4 * (size_t)lbm::reduce_blocks((long long)nz * nr) * sizeof(double));
    h->derr = (int*)dev_alloc(sizeof(int));
    // tile plan of the marching step: warps, or CTAs on wide strips with the link source or Guo forcing
    // (4096 x 2048 Guo: 210 us per step by CTAs, 155 by warps, whose sums round differently)
    const bool link = o.h_eval == LBM_H_LINK_AVG && o.axis_terms, ctas = link || guo_of(h);
    std::vector<lbm::Tile> tiles;
    std::vector<int> first;
    if (!lbm_by_phases(o.precision, lbm::phase_nodes(nz, nr))) {
        const int slots = ctas ? Ops<float>::batch_resident_ctas(lbm::kStripWide) : Ops<float>::warp_slots();
        int rc = LBM_ERR_CUDA;
        try {
            if (ctas)
                rc = slots > 0 ? lbm::plan_tiles(&nz, &nr, 1, lbm::kStripWide, slots, tiles, first, nullptr) : rc;
            else
                rc = slots > 0 ? lbm::plan_warp_tiles(&nz, &nr, 1, slots, tiles) : rc;
        } catch (...) {
            rc = LBM_ERR_OOM;
        }
        if (rc != LBM_OK) {
            release_all(h);
            delete h;
            return rc;
        }
    }
    h->ncta = first.empty() ? (int)tiles.size() : (int)first.size() - 1;
    h->d_tiles = (lbm::Tile*)dev_alloc(tiles.size() * sizeof(lbm::Tile));
    h->d_first = (int*)dev_alloc(first.size() * sizeof(int));
    h->bytes = lbm_axi_footprint(nz, nr, o.precision);
    if (link) {
        h->hb[0] = dev_alloc(3 * plane_bytes);
        h->hb[1] = dev_alloc(3 * plane_bytes);
        h->bytes += 6 * plane_bytes;
    }
    bool ok = h->f[0] && h->f[1] && h->aux && h->mout && h->partial && h->derr &&
              h->d_tiles && h->d_first && (!link || (h->hb[0] && h->hb[1]));
    ok = ok && cudaMallocHost(&h->herr, sizeof(int)) == cudaSuccess;
    ok = ok && cudaMallocHost(&h->hred, 4 * sizeof(double)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        release_all(h);
        delete h;
        return LBM_ERR_OOM;
    }
    if (o.stream) {
        h->stream = (cudaStream_t)o.stream;
        h->own_stream = false;
    } else {
        if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) {
            release_all(h);
            delete h;
            return LBM_ERR_CUDA;
        }
        h->own_stream = true;
    }
    h->pf = make_params<float>(h);
    h->pdd = make_params<double>(h);
    h->path = fused_ok(h) ? LBM_PATH_FUSED : LBM_PATH_SPLIT;
    h->tile = o.precision == 32 ? lbm::tile_form(&nz, &nr, 1, o.multiphase != 0, o.axis_terms != 0, fv_of(h))
                                : lbm::TILE_NONE;
    h->rows_per_cta = 0;  // the form the size chooses (step_fused)
    if (h->precision == 32) h->pdd = make_params_out(h);
    *h->herr = 0;
    cudaError_t err = cudaSuccess;
    if (!tiles.empty()) {
        err = cudaMemcpy(h->d_tiles, tiles.data(), tiles.size() * sizeof(lbm::Tile), cudaMemcpyHostToDevice);
        if (err == cudaSuccess && !first.empty())
            err = cudaMemcpy(h->d_first, first.data(), first.size() * sizeof(int), cudaMemcpyHostToDevice);
    }
    if (err == cudaSuccess) err = cudaMemsetAsync(h->derr, 0, sizeof(int), h->stream);
    if (err == cudaSuccess) err = cudaMemsetAsync(h->aux, 0, 4 * plane_bytes, h->stream);
    if (err == cudaSuccess) err = cudaStreamSynchronize(h->stream);
    if (err != cudaSuccess) {
        release_all(h);
        delete h;
        return LBM_ERR_CUDA;
    }
    *out = h;
    return LBM_OK;
}

// f^eq(rho, u) into buffer 0, no error and no arrival halves pending.
static cudaError_t begin_init(lbm_axi* h, const double* rho, const double* uz, const double* ur) {
    cudaError_t e = enqueue_init(h, rho, uz, ur, nullptr);
    h->cur = 0;
    // a fresh state: clear the sticky error word (a step skips a solve whose word is set)
    if (e == cudaSuccess) e = cudaMemsetAsync(h->derr, 0, sizeof(int), h->stream);
    for (int q = 0; q < 2 && e == cudaSuccess && h->hb[0]; q++)
        e = cudaMemsetAsync(h->hb[q], 0, 3 * (size_t)h->plane * (h->precision == 32 ? 4 : 8), h->stream);
    return e;
}

int lbm_axi_init_device(lbm_axi* h, const double* rho, const double* uz, const double* ur) {
    if (!h || !rho) return LBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if (begin_init(h, rho, uz, ur) != cudaSuccess) return LBM_ERR_CUDA;
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return LBM_ERR_CUDA;
    h->initialized = true;
    h->pending = LBM_OK;
    return LBM_OK;
}

int lbm_axi_init(lbm_axi* h, const double* rho, const double* uz, const double* ur) {
    if (!h || !rho) return LBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    const size_t n = (size_t)h->nz * h->nr;
    double* d_rho = h->mout;
    double* d_uz = uz ? h->mout + n : nullptr;
    double* d_ur = ur ? h->mout + 2 * n : nullptr;
    cudaError_t e = cudaMemcpyAsync(d_rho, rho, n * sizeof(double), cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess && uz) e = cudaMemcpyAsync(d_uz, uz, n * sizeof(double), cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess && ur) e = cudaMemcpyAsync(d_ur, ur, n * sizeof(double), cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    return lbm_axi_init_device(h, d_rho, d_uz, d_ur);
}

// One stream order without a wait between: f^eq(rho, u), its fluid velocity into the field planes, then
// f^eq(rho, u - F / (2 rho)) unless the state raised an error.
int lbm_axi_init_physical_device(lbm_axi* h, const double* rho, const double* uz, const double* ur) {
    if (!h || !rho) return LBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    char* phys = static_cast<char*>(h->aux) + (size_t)h->plane * (h->precision == 32 ? 4 : 8);
    cudaError_t e = begin_init(h, rho, uz, ur);
    if (e == cudaSuccess) e = enqueue_fields(h, nullptr, nullptr, nullptr, nullptr, phys);
    if (e == cudaSuccess) e = enqueue_init(h, rho, uz, ur, phys);
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    h->initialized = true;
    h->pending = LBM_OK;
    return read_error(h);
}

int lbm_axi_init_physical(lbm_axi* h, const double* rho, const double* uz, const double* ur) {
    if (!h || !rho) return LBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    const size_t n = (size_t)h->nz * h->nr;
    double* d = h->mout;  // idle: the velocity between the two passes is in the field planes
    cudaError_t e = cudaMemcpyAsync(d, rho, n * sizeof(double), cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess && uz) e = cudaMemcpyAsync(d + n, uz, n * sizeof(double), cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess && ur)
        e = cudaMemcpyAsync(d + 2 * n, ur, n * sizeof(double), cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) {
        cudaStreamSynchronize(h->stream);
        return LBM_ERR_CUDA;
    }
    return lbm_axi_init_physical_device(h, d, uz ? d + n : nullptr, ur ? d + 2 * n : nullptr);
}

int lbm_axi_step_async(lbm_axi* h, long long n) {
    if (!h || n < 0) return LBM_ERR_INVALID_ARG;
    if (!h->initialized) return LBM_ERR_STATE;
    DeviceGuard g(h->device);
    if (n == 0) return LBM_OK;
    cudaError_t e = cudaSuccess;
    if (h->cur == 1) {  // graphs start from buffer 0
        e = enqueue_step(h);
        n--;
    }
    const int chunk = chunk_steps(h);
    if (e == cudaSuccess && n >= chunk && !one_by_one(h->stream)) {
        if (!h->graph || h->graph_steps != chunk) {
            int rc = build_graph(h, chunk);
            if (rc != LBM_OK) return rc;
        }
        while (n >= chunk && e == cudaSuccess) {
            e = cudaGraphLaunch(h->graph, h->stream);
            n -= chunk;
        }
    }
    while (n > 0 && e == cudaSuccess) {
        e = enqueue_step(h);
        n--;
    }
    if (e != cudaSuccess) {
        h->pending = LBM_ERR_CUDA;
        return LBM_ERR_CUDA;
    }
    return LBM_OK;
}

int lbm_axi_sync(lbm_axi* h) {
    if (!h) return LBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    int rc = read_error(h);
    if (h->pending != LBM_OK) rc = h->pending;
    h->pending = LBM_OK;
    return rc;
}

int lbm_axi_step(lbm_axi* h, long long n) {
    int rc = lbm_axi_step_async(h, n);
    if (rc != LBM_OK) {
        if (h && rc != LBM_ERR_INVALID_ARG && rc != LBM_ERR_STATE) lbm_axi_sync(h);
        return rc;
    }
    return lbm_axi_sync(h);
}

int lbm_axi_time_kernels(lbm_axi* h, long long n, double* ms) {
    if (!h || n < 0 || !ms) return LBM_ERR_INVALID_ARG;
    if (!h->initialized) return LBM_ERR_STATE;
    DeviceGuard g(h->device);
    cudaEvent_t ev[3];
    for (int q = 0; q < 3; q++) {
        if (cudaEventCreate(&ev[q]) != cudaSuccess) return LBM_ERR_CUDA;
    }
    double acc[2] = {0.0, 0.0};
    cudaError_t e = cudaSuccess;
    for (long long s = 0; s < n && e == cudaSuccess; s++) {
        const int c = h->cur;
        e = cudaEventRecord(ev[0], h->stream);
        if (e == cudaSuccess && h->path == LBM_PATH_SPLIT) e = enqueue_density(h);
        if (e == cudaSuccess) e = cudaEventRecord(ev[1], h->stream);
        if (e == cudaSuccess && h->path == LBM_PATH_FUSED) {
            e = enqueue_step(h);
            h->cur = c;
        } else if (e == cudaSuccess) {
            if (h->precision == 32)
                e = Ops<float>::update(h->pf, (const float*)h->f[c], (float*)h->f[c ^ 1],
                                       (const float*)h->aux, h->stream, link_planes<float>(h, c), guo_of(h));
            else
                e = Ops<double>::update(h->pdd, (const double*)h->f[c], (double*)h->f[c ^ 1],
                                        (const double*)h->aux, h->stream, link_planes<double>(h, c), guo_of(h));
        }
        if (e == cudaSuccess) e = cudaEventRecord(ev[2], h->stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(ev[2]);
        float t0 = 0.f, t1 = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t0, ev[0], ev[1]);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t1, ev[1], ev[2]);
        acc[0] += t0;
        acc[1] += t1;
        h->cur = c ^ 1;
    }
    for (int q = 0; q < 3; q++) cudaEventDestroy(ev[q]);
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    ms[0] = acc[0];
    ms[1] = acc[1];
    return read_error(h);
}

// Fields to arrays a kernel may write directly, else through the staging planes.
int lbm_axi_moments_device(lbm_axi* h, double* rho, double* uz, double* ur, double* p) {
    if (!h) return LBM_ERR_INVALID_ARG;
    if (!h->initialized) return LBM_ERR_STATE;
    DeviceGuard g(h->device);
    const size_t n = (size_t)h->nz * h->nr;
    double* dst[4] = {rho, uz, ur, p};
    double* to[4];
    DeviceRange r;  // looked up again only for a destination that is not in the last one's allocation
    for (int q = 0; q < 4; q++) {
        if (dst[q] && !r.holds(dst[q], n)) r = allocation_of(dst[q], h->device);
        to[q] = !dst[q] || r.holds(dst[q], n) ? dst[q] : h->mout + q * n;
    }
    cudaError_t e = enqueue_fields(h, to[0], to[1], to[2], to[3], nullptr);
    for (int q = 0; q < 4 && e == cudaSuccess; q++) {
        if (dst[q] && to[q] != dst[q])
            e = cudaMemcpyAsync(dst[q], to[q], n * sizeof(double), cudaMemcpyDefault, h->stream);
    }
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    return read_error(h);
}

int lbm_axi_moments(lbm_axi* h, double* rho, double* uz, double* ur, double* p) {
    return lbm_axi_moments_device(h, rho, uz, ur, p);
}

// ------------------------------------------------------- checkpoint --
// Blob: StateHeader, then the 9 population planes (nr x nz each, z fastest) in
// the storage precision, exactly as the next step will read them.  The header
// records the grid, precision, reference density and every parameter of the
// dynamics, so that a blob only resumes a solve that continues the same run.
namespace {
struct StateHeader {
    char magic[8];  // "LBMAXIS1"
    int32_t version, precision, nz, nr;
    double rho_ref;
    int32_t cur, link_planes, reserved[6];
    // dynamics (format version 2)
    double tau, A, T, T_over_Tc, a, b, R, lambda, g_z;
    int32_t eos_kind, top_bc, axis_terms, multiphase, kappa_mode, hr_sign, h_eval, forcing;
    int32_t axis_a_term, reserved2[5];
};
static_assert(sizeof(StateHeader) == 192, "checkpoint header layout");
const char kStateMagic[8] = {'L', 'B', 'M', 'A', 'X', 'I', 'S', '1'};
constexpr int32_t kStateVersion = 2;

void fill_header(const lbm_axi* h, StateHeader* hd) {
    memset(hd, 0, sizeof(*hd));
    memcpy(hd->magic, kStateMagic, sizeof(kStateMagic));
    hd->version = kStateVersion;
    hd->precision = h->precision;
    hd->nz = h->nz;
    hd->nr = h->nr;
    hd->rho_ref = stored_rho_ref(h);
    hd->cur = h->cur;
    hd->link_planes = h->hb[0] ? 1 : 0;
    hd->tau = h->tau;
    hd->A = h->A;
    hd->T = h->T;
    hd->T_over_Tc = h->opts.multiphase ? h->eos.T_over_Tc : 0.0;
    hd->a = h->opts.multiphase ? h->eos.a : 0.0;
    hd->b = h->opts.multiphase ? h->eos.b : 0.0;
    hd->R = h->opts.multiphase ? h->eos.R : 0.0;
    hd->lambda = h->opts.multiphase ? h->eos.lambda : 0.0;
    hd->g_z = h->opts.g_z;
    hd->eos_kind = h->opts.multiphase ? h->eos.kind : -1;
    hd->top_bc = h->opts.top_bc;
    hd->axis_terms = h->opts.axis_terms ? 1 : 0;
    hd->multiphase = h->opts.multiphase ? 1 : 0;
    hd->kappa_mode = h->opts.kappa_mode;
    hd->hr_sign = h->opts.hr_sign;
    hd->h_eval = h->opts.h_eval;
    hd->forcing = h->opts.forcing;
    hd->axis_a_term = h->opts.axis_a_term;
}

// The blob continues this solve: same layout and the same dynamics, bit for bit.
bool header_matches(const lbm_axi* h, const StateHeader& hd) {
    StateHeader mine;
    fill_header(h, &mine);
    return memcmp(hd.magic, mine.magic, sizeof(mine.magic)) == 0 && hd.version == mine.version &&
           hd.precision == mine.precision && hd.nz == mine.nz && hd.nr == mine.nr && hd.rho_ref == mine.rho_ref &&
           (hd.cur == 0 || hd.cur == 1) && hd.link_planes == mine.link_planes && hd.tau == mine.tau &&
           hd.A == mine.A && hd.T == mine.T && hd.T_over_Tc == mine.T_over_Tc && hd.a == mine.a &&
           hd.b == mine.b && hd.R == mine.R && hd.lambda == mine.lambda && hd.g_z == mine.g_z &&
           hd.eos_kind == mine.eos_kind && hd.top_bc == mine.top_bc && hd.axis_terms == mine.axis_terms &&
           hd.multiphase == mine.multiphase && hd.kappa_mode == mine.kappa_mode && hd.hr_sign == mine.hr_sign &&
           hd.h_eval == mine.h_eval && hd.forcing == mine.forcing && hd.axis_a_term == mine.axis_a_term;
}

// planes in the blob: the 9 populations, then (link-midpoint source) the 3 source planes
int state_planes(const lbm_axi* h) { return h->hb[0] ? 12 : 9; }
size_t state_bytes(const lbm_axi* h) {
    return sizeof(StateHeader) + (size_t)state_planes(h) * h->nz * h->nr * (h->precision == 32 ? 4 : 8);
}
}  // namespace

int lbm_axi_state_bytes(const lbm_axi* h, size_t* bytes) {
    if (!h || !bytes) return LBM_ERR_INVALID_ARG;
    *bytes = state_bytes(h);
    return LBM_OK;
}

int lbm_axi_save(lbm_axi* h, void* buf, size_t bytes) {
    if (!h || !buf || bytes < state_bytes(h)) return LBM_ERR_INVALID_ARG;
    if (!h->initialized) return LBM_ERR_STATE;
    DeviceGuard g(h->device);
    StateHeader hd;
    fill_header(h, &hd);
    memcpy(buf, &hd, sizeof(hd));
    const size_t es = h->precision == 32 ? 4 : 8;
    char* dst = static_cast<char*>(buf) + sizeof(hd);
    const char* src = static_cast<const char*>(h->f[h->cur]);
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < state_planes(h) && e == cudaSuccess; i++) {
        const char* s = i < 9 ? src + (size_t)i * h->plane * es
                              : static_cast<const char*>(h->hb[h->cur]) + (size_t)(i - 9) * h->plane * es;
        e = cudaMemcpy2DAsync(dst + (size_t)i * h->nz * h->nr * es, h->nz * es, s, (size_t)h->pitch * es,
                              h->nz * es, h->nr, cudaMemcpyDeviceToHost, h->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    return read_error(h);
}

int lbm_axi_load(lbm_axi* h, const void* buf, size_t bytes) {
    if (!h || !buf || bytes < sizeof(StateHeader)) return LBM_ERR_INVALID_ARG;
    StateHeader hd;
    memcpy(&hd, buf, sizeof(hd));
    if (!header_matches(h, hd) || bytes < state_bytes(h)) return LBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    const size_t es = h->precision == 32 ? 4 : 8;
    const char* src = static_cast<const char*>(buf) + sizeof(hd);
    char* dst = static_cast<char*>(h->f[hd.cur]);
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < state_planes(h) && e == cudaSuccess; i++) {
        char* d = i < 9 ? dst + (size_t)i * h->plane * es
                        : static_cast<char*>(h->hb[hd.cur]) + (size_t)(i - 9) * h->plane * es;
        e = cudaMemcpy2DAsync(d, (size_t)h->pitch * es, src + (size_t)i * h->nz * h->nr * es, h->nz * es,
                              h->nz * es, h->nr, cudaMemcpyHostToDevice, h->stream);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(h->derr, 0, sizeof(int), h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    h->cur = hd.cur;
    h->initialized = true;
    h->pending = LBM_OK;
    return LBM_OK;
}

int lbm_axi_mass(lbm_axi* h, double* mass_rw, double* mass_plain) {
    if (!h || !mass_rw) return LBM_ERR_INVALID_ARG;
    if (!h->initialized) return LBM_ERR_STATE;
    DeviceGuard g(h->device);
    cudaError_t e;
    if (h->precision == 32)
        e = Ops<float>::mass(h->pf, (const float*)h->f[h->cur], link_planes<float>(h, h->cur), h->partial, h->hred,
                             h->derr, h->stream);
    else
        e = Ops<double>::mass(h->pdd, (const double*)h->f[h->cur], link_planes<double>(h, h->cur), h->partial, h->hred,
                              h->derr, h->stream);
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    int rc = read_error(h);
    if (rc != LBM_OK) return rc;
    // the sums are over rho - rho_ref
    const double n = (double)h->nz * h->nr, ref = stored_rho_ref(h);
    *mass_rw = h->hred[0] + ref * (0.5 * n * h->nr);
    if (mass_plain) *mass_plain = h->hred[1] + ref * n;
    return LBM_OK;
}

int lbm_axi_pressure_jump(lbm_axi* h, double zc, double rc, double rin, double rout, double* dp) {
    if (!h || !dp || !(rin > 0) || !(rout >= rin)) return LBM_ERR_INVALID_ARG;
    if (!h->initialized) return LBM_ERR_STATE;
    DeviceGuard g(h->device);
    cudaError_t e;
    if (h->precision == 32)
        e = Ops<float>::pjump(h->pf, h->pdd, (const float*)h->f[h->cur], link_planes<float>(h, h->cur), zc, rc, rin,
                              rout, h->partial, h->hred, h->derr, h->stream);
    else
        e = Ops<double>::pjump(h->pdd, h->pdd, (const double*)h->f[h->cur], link_planes<double>(h, h->cur), zc, rc,
                               rin, rout, h->partial, h->hred, h->derr, h->stream);
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    int rcode = read_error(h);
    if (rcode != LBM_OK) return rcode;
    if (!(h->hred[1] > 0) || !(h->hred[3] > 0)) return LBM_ERR_INVALID_ARG;
    *dp = h->hred[0] / h->hred[1] - h->hred[2] / h->hred[3];
    return LBM_OK;
}

void lbm_axi_destroy(lbm_axi* h) {
    if (!h) return;
    DeviceGuard g(h->device);
    cudaStreamSynchronize(h->stream);
    release_all(h);
    delete h;
}

int lbm_axi_get_tuning(const lbm_axi* h, lbm_axi_tuning* t) {
    if (!h || !t) return LBM_ERR_INVALID_ARG;
    t->path = h->path;
    t->rows_per_cta = h->rows_per_cta;
    return LBM_OK;
}

int lbm_axi_set_tuning(lbm_axi* h, const lbm_axi_tuning* t) {
    if (!h || !t) return LBM_ERR_INVALID_ARG;
    if (t->path != LBM_PATH_FUSED && t->path != LBM_PATH_SPLIT) return LBM_ERR_INVALID_ARG;
    if (t->path == LBM_PATH_FUSED && !fused_ok(h)) return LBM_ERR_INVALID_ARG;
    if (t->path == LBM_PATH_FUSED && fv_of(h) != 0 && t->rows_per_cta != 0) return LBM_ERR_INVALID_ARG;
    if (t->rows_per_cta < 0 || t->rows_per_cta > (1 << 20)) return LBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return LBM_ERR_CUDA;
    if (h->graph) {
        cudaGraphExecDestroy(h->graph);
        h->graph = nullptr;
    }
    h->path = t->path;
    h->rows_per_cta = t->rows_per_cta;
    return LBM_OK;
}

// As enqueue_step and step_fused choose.
const char* lbm_axi_step_kernels(const lbm_axi* h) {
    if (!h) return nullptr;
    if (h->path != LBM_PATH_FUSED) return "k_density,k_update";
    if (h->rows_per_cta > 0) return "k_step";
    if (h->tile != lbm::TILE_NONE) return "k_tile";
    if (lbm_by_phases(h->precision, lbm::phase_nodes(h->nz, h->nr))) return "k_phase_l,k_phase_u,k_phase_c";
    return fv_of(h) == 0 ? "k_step_warp" : "k_step_single";
}

int lbm_axi_temperature(const lbm_axi* h, double* T, double* Tc) {
    if (!h) return LBM_ERR_INVALID_ARG;
    if (T) *T = h->T;
    if (Tc) *Tc = h->Tc;
    return LBM_OK;
}

int lbm_axi_device_bytes(const lbm_axi* h, size_t* bytes) {
    if (!h || !bytes) return LBM_ERR_INVALID_ARG;
    *bytes = h->bytes;
    return LBM_OK;
}

int lbm_eos_critical_temperature(const lbm_eos* eos, double* Tc) {
    if (!eos || !Tc) return LBM_ERR_INVALID_ARG;
    double rc;
    return lbm::critical_point(*eos, Tc, &rc) ? LBM_OK : LBM_ERR_INVALID_ARG;
}

int lbm_eos_coexistence(const lbm_eos* eos, double* rho_v, double* rho_l) {
    if (!eos || !rho_v || !rho_l) return LBM_ERR_INVALID_ARG;
    const double T = lbm::absolute_temperature(*eos);
    if (!(T > 0)) return LBM_ERR_INVALID_ARG;
    return lbm::coexistence(*eos, T, rho_v, rho_l) ? LBM_OK : LBM_ERR_INVALID_ARG;
}

int lbm_eos_pressure(const lbm_eos* eos, double rho, double* p, double* dpdrho) {
    if (!eos || !p) return LBM_ERR_INVALID_ARG;
    const double T = lbm::absolute_temperature(*eos);
    if (!(T > 0)) return LBM_ERR_INVALID_ARG;
    double dp;
    lbm::eos_pressure(*eos, T, rho, p, &dp);
    if (dpdrho) *dpdrho = dp;
    return LBM_OK;
}

int lbm_axi_set_allocator(void* (*alloc)(size_t, void*), void (*release)(void*, void*), void* ctx) {
    if ((alloc == nullptr) != (release == nullptr)) return LBM_ERR_INVALID_ARG;
    g_alloc = alloc;
    g_release = release;
    g_alloc_ctx = ctx;
    return LBM_OK;
}

const char* lbm_axi_strerror(int code) {
    switch (code) {
        case LBM_OK: return "ok";
        case LBM_ERR_INVALID_ARG: return "invalid argument";
        case LBM_ERR_OOM: return "out of memory";
        case LBM_ERR_CUDA: return "CUDA error";
        case LBM_ERR_UNPHYSICAL: return "unphysical state (rho <= 0, psi^2 < 0 or non-finite value)";
        case LBM_ERR_TIMEOUT: return "device wait timed out";
        case LBM_ERR_STATE: return "call out of order (solve not initialised)";
        default: return "unknown error";
    }
}

}  // extern "C"
