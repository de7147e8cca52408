// A CUDA runtime and launchers that only keep books, so that the library's host code (lbm_axi.cu,
// lbm_batch.cu) can be driven on the CPU through failures that a GPU must not be driven through: an
// allocation that fails, a launch on a list that is gone.  Device memory is host memory; a launch checks
// that the lists it is given lie in live allocations.  One program, one check per argument.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <map>
#include <new>
#include <tuple>
#include <vector>

#include "lbm_axi.h"
#include "lbm_axi_batch.h"
#include "lbm_handle.h"
#include "lbm_launch.h"

namespace fake {
std::map<uintptr_t, size_t>* live = nullptr;  // device allocations
long long device_left = -1, host_left = -1;   // allocations until one fails (-1: none does)
int launches = 0, violations = 0;
const char* form = "";  // of the last step launched
bool track = false;
const void* last_rho = nullptr;   // where the last read wrote its density
cudaStream_t captured = nullptr;  // a stream that its owner is capturing

struct Untracked {  // the runtime's own bookkeeping does not count
    const bool was = track;
    Untracked() { track = false; }
    ~Untracked() { track = was; }
};

bool inside(const void* p, size_t bytes) {
    auto it = live->upper_bound((uintptr_t)p);
    if (it == live->begin()) return false;
    --it;
    return (uintptr_t)p + bytes <= it->first + it->second;
}
cudaError_t launch(const void* list, size_t bytes, const void* list2 = nullptr, size_t bytes2 = 0) {
    launches++;
    if (!inside(list, bytes) || (bytes2 && !inside(list2, bytes2))) {
        violations++;
        return cudaErrorIllegalAddress;
    }
    return cudaSuccess;
}
}  // namespace fake

void* operator new(size_t n) {
    if (fake::host_left >= 0 && fake::track && fake::host_left-- == 0) throw std::bad_alloc();
    void* p = malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

// ----------------------------------------------------------------- runtime --

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
    if (fake::device_left >= 0 && fake::device_left-- == 0) return cudaErrorMemoryAllocation;
    fake::Untracked u;
    *p = calloc(n, 1);
    (*fake::live)[(uintptr_t)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    fake::live->erase((uintptr_t)p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return *p = calloc(1, n), cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { return *p = calloc(1, n), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return memcpy(d, s, n), cudaSuccess; }
static CUresult address_range(CUdeviceptr* base, size_t* size, CUdeviceptr p) {
    auto it = fake::live->upper_bound(p);
    if (it == fake::live->begin()) return CUDA_ERROR_NOT_FOUND;
    --it;
    *base = it->first, *size = it->second;
    return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    const bool known = !strcmp(name, "cuMemGetAddressRange");
    *f = known ? (void*)address_range : nullptr;
    *q = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    // to an address in device memory: refused unless it all fits
    if (fake::inside(d, 1) && !fake::inside(d, n)) return cudaErrorInvalidValue;
    return memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    memset(a, 0, sizeof(*a));
    if (fake::inside(p, 1)) a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)malloc(1), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return free((void*)s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    return s == fake::captured || s == cudaStreamLegacy ? cudaErrorIllegalState : cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
    *st = s == fake::captured ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return *g = (cudaGraph_t)malloc(1), cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
    return *x = (cudaGraphExec_t)malloc(1), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return free((void*)g), cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { return free((void*)x), cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) {
    return s == fake::captured ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
}

// --------------------------------------------------------------- launchers --

namespace lbm {

TileForm tile_form(const int*, const int*, int, bool, bool, int) { return TILE_NONE; }
void tile_size(TileForm, int* tz, int* tr) { *tz = 16, *tr = 8; }

template <typename R>
cudaError_t Ops<R>::density(const Params<R>&, const R*, R*, int*, cudaStream_t, LinkPlanes<R>) { return cudaSuccess; }
template <typename R>
cudaError_t Ops<R>::update(const Params<R>&, const R*, R*, const R*, cudaStream_t, LinkPlanes<R>, bool) {
    return cudaSuccess;
}
template <typename R>
cudaError_t Ops<R>::fields(const BatchSolve<R>& v, LinkPlanes<R>, const Params<double>&, int, double* rho, double* uz,
                           double* ur, double* pk, R*, int*, cudaStream_t) {
    for (double* q : {rho, uz, ur, pk})
        if (q && !fake::inside(q, (size_t)v.p.nz * v.p.nr * sizeof(double))) fake::violations++;
    fake::last_rho = rho;
    return cudaSuccess;
}
template <typename R>
cudaError_t Ops<R>::init(const Params<R>&, double, const double*, const double*, const double*, R*, cudaStream_t,
                         const R*, const int*) {
    return cudaSuccess;
}
template <typename R>
cudaError_t Ops<R>::mass(const Params<R>&, const R*, LinkPlanes<R>, double*, double*, int*, cudaStream_t) {
    return cudaSuccess;
}
template <typename R>
cudaError_t Ops<R>::pjump(const Params<R>&, const Params<double>&, const R*, LinkPlanes<R>, double, double, double,
                          double, double*, double*, int*, cudaStream_t) {
    return cudaSuccess;
}
template <typename R>
cudaError_t Ops<R>::take_error(int*, int*, cudaStream_t) { return cudaSuccess; }
template <typename R>
cudaError_t Ops<R>::prepare() { return cudaSuccess; }
template <typename R>
cudaError_t Ops<R>::step(const Params<R>&, const R*, R*, int, int*, cudaStream_t) { return cudaSuccess; }
template <typename R>
cudaError_t Ops<R>::step_batch(const BatchSolve<R>*, const Tile* tiles, const int* first, int ncta, bool, bool, int, int,
                               int*, cudaStream_t) {
    fake::form = "ctas";
    if (ncta <= 0) return cudaErrorInvalidConfiguration;
    return fake::launch(first, (ncta + 1) * sizeof(int), tiles, sizeof(Tile));
}
template <typename R>
cudaError_t Ops<R>::step_single(const BatchSolve<R>&, const LinkSets<R>&, const Tile* tiles, const int* first, int ncta,
                                bool, bool, int, int*, cudaStream_t, int) {
    fake::form = "ctas";
    if (ncta <= 0) return cudaErrorInvalidConfiguration;
    return fake::launch(first, (ncta + 1) * sizeof(int), tiles, sizeof(Tile));
}
template <typename R>
cudaError_t Ops<R>::step_table(const BatchTable<R>&, const Tile* tiles, const int* first, int ncta, bool, bool, int, int,
                               int*, cudaStream_t) {
    fake::form = "ctas";
    if (ncta <= 0) return cudaErrorInvalidConfiguration;
    return fake::launch(first, (ncta + 1) * sizeof(int), tiles, sizeof(Tile));
}
template <typename R>
cudaError_t Ops<R>::phase_step(const BatchSolve<R>&, const LinkSets<R>&, bool, bool, int, int*, cudaStream_t, int) {
    fake::form = "phases";
    return fake::launches++, cudaSuccess;
}
template <typename R>
cudaError_t Ops<R>::phase_step_many(const BatchSolve<R>* solves, const PhaseTile* tiles, int ntiles, int nghost, int,
                                    bool, bool, int, int*, cudaStream_t) {
    fake::form = "phases";
    if (ntiles <= 0) return cudaErrorInvalidConfiguration;
    return fake::launch(tiles, (ntiles + nghost) * sizeof(PhaseTile), solves, sizeof(BatchSolve<R>));
}
template <typename R>
int Ops<R>::phase_tile_z() { return 64; }
template <typename R>
int Ops<R>::phase_rows(long long) { return 8; }
template <typename R>
int Ops<R>::batch_resident_ctas(int) { return 608; }
template <>
cudaError_t Ops<float>::tile_step(TileForm, const BatchSolve<float>&, bool, int, int*, cudaStream_t) {
    return fake::launches++, cudaSuccess;
}
template <>
cudaError_t Ops<float>::tile_step_many(TileForm, const BatchSolve<float>*, const PhaseTile* tiles, int n, bool, int, int*,
                                       cudaStream_t) {
    return fake::launch(tiles, n * sizeof(PhaseTile));
}
template <>
int Ops<float>::warp_slots() { return 1824; }
template <>
cudaError_t Ops<float>::step_warp(const BatchSolve<float>&, const Tile* tiles, int n, bool, bool, int, int*, cudaStream_t) {
    fake::form = "warps";
    return fake::launch(tiles, n * sizeof(Tile));
}
template <>
cudaError_t Ops<float>::step_warp_many(const BatchSolve<float>* solves, int, const Tile* tiles, int n, bool, bool, int, int*,
                                       cudaStream_t) {
    fake::form = "warps";
    if (n <= 0) return cudaErrorInvalidConfiguration;
    const cudaError_t e = fake::launch(tiles, n * sizeof(Tile), solves, sizeof(BatchSolve<float>));
    for (int i = 0; e == cudaSuccess && i < n; i++)  // the list is this form's: strips of its width, rows of the solve
        if (tiles[i].strip * kWarpStrip >= solves[tiles[i].solve].p.nz || tiles[i].jend > solves[tiles[i].solve].p.nr)
            fake::violations++;
    return e;
}
template <>
int Ops<float>::warp_kind(const Params<float>&) { return 0; }
template <>
int Ops<float>::warp_kind(int a, int) { return a; }
template struct Ops<float>;
template struct Ops<double>;

}  // namespace lbm

// ------------------------------------------------------------------ checks --

#define CHECK(c)                                              \
    do {                                                      \
        if (!(c)) {                                           \
            fprintf(stderr, "line %d: %s\n", __LINE__, #c);   \
            exit(1);                                          \
        }                                                     \
    } while (0)

static lbm_axi* solve(int nz, int nr, int precision, void* stream = nullptr, int forcing = LBM_FORCING_EDM) {
    lbm_axi_opts o;
    lbm_axi_default_opts(&o);
    o.precision = precision;
    o.stream = stream;
    o.forcing = forcing;
    lbm_eos e = {LBM_EOS_CS, 0.9, 1.0, 4.0, 1.0, 0.01};
    lbm_axi* h = nullptr;
    CHECK(lbm_axi_create(nz, nr, 1.0, &e, -0.152, &o, &h) == LBM_OK);
    double* rho = (double*)calloc((size_t)nz * nr, sizeof(double));
    CHECK(lbm_axi_init(h, rho, nullptr, nullptr) == LBM_OK);
    free(rho);
    return h;
}

// A change of a batch's tuning that runs out of device or host memory, at any of its allocations: the call
// reports it, the batch keeps the tuning it had and the next step launches over that tuning's lists.
static void batch_retune(int nz, int nr, int n, int precision, bool device) {
    lbm_axi* h[300];
    for (int i = 0; i < n; i++) h[i] = solve(nz, nr, precision);
    lbm_axi_batch* b = nullptr;
    CHECK(lbm_axi_batch_create(h, n, nullptr, &b) == LBM_OK);
    CHECK(lbm_axi_batch_step(b, 1) == LBM_OK);
    const lbm_axi_batch_tuning to[4] = {{64, 0}, {112, 0}, {112, 300}, {112, 0}};
    for (const lbm_axi_batch_tuning& t : to) {
        lbm_axi_batch_tuning had, has;
        lbm_axi_batch_get_tuning(b, &had);
        int failures = 0;
        for (int at = 0;; at++) {
            (device ? fake::device_left : fake::host_left) = at;
            fake::track = true;
            const int rc = lbm_axi_batch_set_tuning(b, &t);
            fake::track = false;
            fake::device_left = fake::host_left = -1;
            if (rc == LBM_OK) break;
            failures++;
            CHECK(rc == LBM_ERR_CUDA || rc == LBM_ERR_OOM);
            lbm_axi_batch_get_tuning(b, &has);
            CHECK(has.strip == had.strip && has.grid == had.grid);
            CHECK(lbm_axi_batch_step(b, 1) == LBM_OK && lbm_axi_batch_step(b, 3) == LBM_OK);
            CHECK(fake::violations == 0);
        }
        CHECK(failures > 0);
        lbm_axi_batch_get_tuning(b, &has);
        CHECK(has.strip == t.strip && has.grid == t.grid);
        CHECK(lbm_axi_batch_step(b, 5) == LBM_OK && fake::violations == 0);
    }
    lbm_axi_batch_destroy(b);
    for (int i = 0; i < n; i++) lbm_axi_destroy(h[i]);
    CHECK(fake::live->empty());
}

// A step of a large FP32 batch is one launch, whatever the number of solves.
static void batch_launches(int nz, int nr, int n) {
    lbm_axi* h[300];
    for (int i = 0; i < n; i++) h[i] = solve(nz, nr, 32);
    lbm_axi_batch* b = nullptr;
    CHECK(lbm_axi_batch_create(h, n, nullptr, &b) == LBM_OK);
    fake::launches = 0;
    CHECK(lbm_axi_batch_step(b, 1) == LBM_OK && fake::launches == 1);
    lbm_axi_batch_destroy(b);
    for (int i = 0; i < n; i++) lbm_axi_destroy(h[i]);
}

// Which form a grid steps by: what counts is its nodes in whole tiles of 64 columns and 8 rows.
static void forms() {
    struct {
        int nz, nr, n;
        const char *edm, *other;  // other: Guo forcing, single solves only
    } const cases[] = {{640, 1248, 1, "phases", "phases"}, {640, 1251, 1, "warps", "ctas"}, {65, 6248, 1, "phases", "phases"},
                       {65, 6251, 1, "warps", "ctas"},     {65, 9000, 1, "warps", "ctas"},  {2, 12496, 1, "phases", "phases"},
                       {2, 150000, 1, "warps", "ctas"},    {64, 32, 299, "phases", nullptr}, {66, 33, 156, "phases", nullptr},
                       {66, 33, 157, "warps", nullptr}};
    for (const auto& c : cases)
        for (int forcing = 0; forcing < (c.other ? 2 : 1); forcing++) {
            lbm_axi* h[300];
            for (int i = 0; i < c.n; i++) h[i] = solve(c.nz, c.nr, 32, nullptr, forcing);
            CHECK(lbm_axi_step(h[0], 1) == LBM_OK);
            if (c.n == 1) {
                const char *form = forcing ? c.other : c.edm, *k = lbm_axi_step_kernels(h[0]);
                CHECK(!strcmp(fake::form, form));
                CHECK(!strcmp(k, !strcmp(form, "phases") ? "k_phase_l,k_phase_u,k_phase_c"
                                                         : (!strcmp(form, "warps") ? "k_step_warp" : "k_step_single")));
            }
            if (!forcing) {
                lbm_axi_batch* b = nullptr;
                CHECK(lbm_axi_batch_create(h, c.n, nullptr, &b) == LBM_OK && lbm_axi_batch_step(b, 1) == LBM_OK);
                CHECK(!strcmp(fake::form, c.edm) && fake::violations == 0);
                lbm_axi_batch_destroy(b);
            }
            for (int i = 0; i < c.n; i++) lbm_axi_destroy(h[i]);
        }
}

// Steps enqueued while the caller captures the solve's stream: one launch each, whatever their number, before
// and after the solve has built a graph of its own.
static void step_under_capture(int precision) {
    cudaStream_t s = (cudaStream_t)malloc(1);
    lbm_axi* h = solve(64, 64, precision, s);
    for (int round = 0; round < 2; round++) {
        for (int n : {1, 31, 32, 64, 200, 255, 256, 400}) {
            fake::captured = s;
            fake::launches = 0;
            CHECK(lbm_axi_step_async(h, n) == LBM_OK && fake::launches == n);
            fake::captured = nullptr;
        }
        CHECK(lbm_axi_step_async(h, 600) == LBM_OK);
    }
    lbm_axi_destroy(h);
    free((void*)s);
}

// Fields wanted in device memory that is too short for them: refused, as the copy that checks it does, and no
// kernel is given the address.  Memory that fits, from its start or within, is written directly.
static void moments_to_short_memory(int precision) {
    const int nz = 37, nr = 18, n = nz * nr;
    lbm_axi* h = solve(nz, nr, precision);
    double* d;
    cudaMalloc((void**)&d, (2 * n + 1) * sizeof(double));
    for (int at : {0, 1, n, n + 1}) {
        CHECK(lbm_axi_moments_device(h, d + at, nullptr, nullptr, nullptr) == LBM_OK && fake::last_rho == d + at);
        CHECK(fake::violations == 0);
    }
    for (int at : {n + 2, 2 * n}) {
        CHECK(lbm_axi_moments_device(h, d + at, nullptr, nullptr, nullptr) == LBM_ERR_CUDA);
        CHECK(lbm_axi_moments_device(h, nullptr, d, nullptr, d + at) == LBM_ERR_CUDA);
        CHECK(fake::violations == 0);
    }
    cudaFree(d);
    lbm_axi_destroy(h);
}

// A solve whose creation runs out of device or host memory, at any of its allocations: an error code, and nothing
// stays allocated.
static void create_out_of_memory(int nz, int nr, int precision, int forcing) {
    lbm_axi_opts o;
    lbm_axi_default_opts(&o);
    o.precision = precision;
    o.forcing = forcing;
    lbm_eos e = {LBM_EOS_CS, 0.9, 1.0, 4.0, 1.0, 0.01};
    for (bool device : {true, false})
        for (int at = 0;; at++) {
            lbm_axi* h = nullptr;
            (device ? fake::device_left : fake::host_left) = at;
            fake::track = true;
            const int rc = lbm_axi_create(nz, nr, 1.0, &e, -0.152, &o, &h);
            fake::track = false;
            fake::device_left = fake::host_left = -1;
            if (rc == LBM_OK) {
                CHECK(h && at > 0);
                lbm_axi_destroy(h);
                CHECK(fake::live->empty());
                break;
            }
            CHECK(rc == LBM_ERR_OOM && !h && fake::live->empty());
        }
}

// A solve on the legacy stream, which cannot be captured.
static void step_on_the_legacy_stream() {
    for (int precision : {32, 64}) {
        lbm_axi* h = solve(64, 64, precision, cudaStreamLegacy);
        for (int n : {1, 31, 32, 100, 255, 256, 700}) {
            fake::launches = 0;
            CHECK(lbm_axi_step(h, n) == LBM_OK && fake::launches == n);
        }
        lbm_axi_destroy(h);
    }
}

// The warps' plan against the general one on the same strips: the same tiles, the tallest first, and no slower than
// the general plan of a march on wide strips.
static void warp_plan() {
    unsigned seed = 1;
    auto rnd = [&](int lo, int hi) { return lo + (int)((seed = seed * 1664525u + 1013904223u) >> 8) % (hi - lo + 1); };
    auto key = [](const lbm::Tile& t) { return std::make_tuple(t.solve, t.strip, t.j0, t.jend); };
    for (int round = 0; round < 120; round++) {
        const int n = round < 40 ? 1 : rnd(2, 300), slots = round % 3 ? 1824 : rnd(1, 4000);
        std::vector<int> nz(n), nr(n), first;
        for (int i = 0; i < n; i++) nz[i] = rnd(1, n == 1 ? 5000 : 600), nr[i] = rnd(16, n == 1 ? 100000 : 400);
        std::vector<lbm::Tile> a, b;
        CHECK(lbm::plan_warp_tiles(nz.data(), nr.data(), n, slots, a) == LBM_OK);
        CHECK(lbm::plan_tiles(nz.data(), nr.data(), n, lbm::kWarpStrip, slots, b, first, nullptr, lbm::kWarpFillRows) == LBM_OK);
        for (size_t i = 1; i < a.size(); i++) CHECK(a[i - 1].jend - a[i - 1].j0 >= a[i].jend - a[i].j0);
        auto less = [&](const lbm::Tile& x, const lbm::Tile& y) { return key(x) < key(y); };
        std::sort(a.begin(), a.end(), less);
        std::sort(b.begin(), b.end(), less);
        CHECK(a.size() == b.size());
        for (size_t i = 0; i < a.size(); i++) CHECK(key(a[i]) == key(b[i]));
    }
    const int nz = 4096, nr = 2048;
    double best[2] = {1e9, 1e9};
    for (int i = 0; i < 20; i++)
        for (int which = 0; which < 2; which++) {
            std::vector<lbm::Tile> t;
            std::vector<int> first;
            const auto t0 = std::chrono::steady_clock::now();
            if (which) lbm::plan_warp_tiles(&nz, &nr, 1, 1824, t);
            else lbm::plan_tiles(&nz, &nr, 1, lbm::kStripWide, 608, t, first, nullptr);
            best[which] = std::min(best[which], std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count());
        }
    CHECK(best[1] <= best[0]);
}

int main(int argc, char** argv) {
    fake::live = new std::map<uintptr_t, size_t>();
    const char* what = argc > 1 ? argv[1] : "";
    if (!strcmp(what, "retune_device_warps")) return batch_retune(1040, 400, 3, 32, true), 0;
    if (!strcmp(what, "retune_host_warps")) return batch_retune(1040, 400, 3, 32, false), 0;
    if (!strcmp(what, "retune_host_many")) return batch_retune(64, 48, 280, 32, false), 0;
    if (!strcmp(what, "retune_device_phases")) return batch_retune(100, 40, 3, 32, true), 0;
    if (!strcmp(what, "retune_host_fp64")) return batch_retune(100, 40, 3, 64, false), 0;
    if (!strcmp(what, "capture32")) return step_under_capture(32), 0;
    if (!strcmp(what, "capture64")) return step_under_capture(64), 0;
    if (!strcmp(what, "short32")) return moments_to_short_memory(32), 0;
    if (!strcmp(what, "short64")) return moments_to_short_memory(64), 0;
    if (!strcmp(what, "create_phases")) return create_out_of_memory(64, 64, 32, 0), 0;
    if (!strcmp(what, "create_fp64")) return create_out_of_memory(64, 64, 64, 0), 0;
    if (!strcmp(what, "create_warps")) return create_out_of_memory(1040, 800, 32, 0), 0;
    if (!strcmp(what, "create_ctas")) return create_out_of_memory(1040, 800, 32, 1), 0;
    if (!strcmp(what, "legacy_stream")) return step_on_the_legacy_stream(), 0;
    if (!strcmp(what, "warp_plan")) return warp_plan(), 0;
    if (!strcmp(what, "forms")) return forms(), 0;
    if (!strcmp(what, "launches")) {
        batch_launches(1040, 400, 2);
        batch_launches(64, 52, 256);
        batch_launches(64, 52, 257);
        batch_launches(64, 52, 300);
        return 0;
    }
    fprintf(stderr, "unknown check %s\n", what);
    return 2;
}
