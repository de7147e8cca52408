// Definitions of Ops<R>; included once per precision.
#pragma once

#include "lbm_early.cuh"
#include "lbm_kernels.cuh"
#include "lbm_launch.h"
#include "lbm_phase.cuh"
#include "lbm_read.cuh"
#include "lbm_step.cuh"

namespace lbm {

// Tile of kernel (b) per precision: TZ nodes along z (coalesced) x TR rows.
template <typename R>
struct UpdateTile;
template <>
struct UpdateTile<float> {
    // 32 x 32: 512 us per launch through the C ABI on the 4096 x 2048 wave against
    // 559 us for 32 x 16 (less halo work); wider tiles lose occupancy (64 x 16: +19 %)
    static constexpr int TZ = 32, TR = 32;
};
template <>
struct UpdateTile<double> {
    static constexpr int TZ = 32, TR = 8;
};

template <typename R>
size_t Ops<R>::update_smem() {
    using T = UpdateTile<R>;
    return sizeof(R) * (size_t)TileShape<T::TZ, T::TR>::elems;
}

// Strip width and rows per iteration of the fused kernel per precision.
template <typename R>
struct StepTile;
// CP: columns per thread (2: march2, pairs of nodes with packed FP32 arithmetic).
template <>
struct StepTile<float> {
    static constexpr int TZ = 112, RR = 2, CP = 2, MINB = 4;  // 128 threads, 45.3 KB of rings
};
template <>
struct StepTile<double> {
    static constexpr int TZ = 64, RR = 2, CP = 1, MINB = 2;  // 160 threads, 71.7 KB of rings
};

template <typename R>
static size_t step_smem() {
    return sizeof(R) * (size_t)StepShape<StepTile<R>::TZ, StepTile<R>::RR>::elems;
}

// The four compiled forms of the fused kernel (force on/off x axis terms on/off).
template <typename R, bool MP, bool AX>
static auto step_kernel() {
    return k_step<R, StepTile<R>::TZ, StepTile<R>::RR, StepTile<R>::CP, StepTile<R>::MINB, MP, AX>;
}

template <typename R>
static cudaError_t set_step_attr(int smem) {
    cudaError_t e = cudaFuncSetAttribute(step_kernel<R, true, true>(), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(step_kernel<R, true, false>(), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(step_kernel<R, false, true>(), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(step_kernel<R, false, false>(), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e;
}

template <typename R>
static cudaError_t single_prepare();
template <typename R, int TZ>
static cudaError_t table_prepare();

template <typename R>
cudaError_t Ops<R>::prepare() {
    using T = UpdateTile<R>;
    const int smem = (int)update_smem();
    cudaError_t e = cudaFuncSetAttribute(k_update<R, T::TZ, T::TR>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_update<R, T::TZ, T::TR, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = set_step_attr<R>((int)step_smem<R>());
    // the marching forms (FP32): attributes and occupancy are settled here, outside any stream capture
    if constexpr (sizeof(R) == 4) {
        if (e == cudaSuccess && (batch_resident_ctas(kStripNarrow) <= 0 || batch_resident_ctas(kStripWide) <= 0))
            e = cudaErrorInvalidConfiguration;
        if (e == cudaSuccess) e = single_prepare<R>();
        if (e == cudaSuccess) e = table_prepare<R, kStripNarrow>();
        if (e == cudaSuccess) e = table_prepare<R, kStripWide>();
    }
    return e;
}

template <typename R>
cudaError_t Ops<R>::step(const Params<R>& p, const R* f, R* fout, int rows_per_cta, int* err, cudaStream_t s) {
    constexpr int TZ = StepTile<R>::TZ, RR = StepTile<R>::RR, CP = StepTile<R>::CP;
    constexpr int NT = StepShape<TZ, RR, CP>::NT;
    const dim3 grid((p.nz + TZ - 1) / TZ, (p.nr + rows_per_cta - 1) / rows_per_cta);
    const size_t smem = step_smem<R>();
    if (p.multiphase && p.axis)
        step_kernel<R, true, true>()<<<grid, NT, smem, s>>>(p, f, fout, rows_per_cta, err);
    else if (p.multiphase)
        step_kernel<R, true, false>()<<<grid, NT, smem, s>>>(p, f, fout, rows_per_cta, err);
    else if (p.axis)
        step_kernel<R, false, true>()<<<grid, NT, smem, s>>>(p, f, fout, rows_per_cta, err);
    else
        step_kernel<R, false, false>()<<<grid, NT, smem, s>>>(p, f, fout, rows_per_cta, err);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Ops<R>::density(const Params<R>& p, const R* f, R* aux, int* err, cudaStream_t s, LinkPlanes<R> lk) {
    dim3 block(32, 8), grid((p.nz + 31) / 32, (p.nr + 7) / 8);
    k_density<R><<<grid, block, 0, s>>>(p, f, aux, err, lk);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Ops<R>::update(const Params<R>& p, const R* f, R* fout, const R* aux, cudaStream_t s, LinkPlanes<R> lk,
                           bool guo) {
    using T = UpdateTile<R>;
    const size_t smem = update_smem();
    dim3 grid((p.nz + T::TZ - 1) / T::TZ, (p.nr + T::TR - 1) / T::TR);
    if (guo)
        k_update<R, T::TZ, T::TR, true><<<grid, 256, smem, s>>>(p, f, fout, aux, lk);
    else
        k_update<R, T::TZ, T::TR><<<grid, 256, smem, s>>>(p, f, fout, aux, lk);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Ops<R>::init(const Params<R>& p, double rho_ref, const double* rho, const double* uz, const double* ur,
                         R* f, cudaStream_t s, const R* phys, const int* err) {
    dim3 block(32, 8), grid((p.nz + 31) / 32, (p.nr + 7) / 8);
    k_init<R><<<grid, block, 0, s>>>(p, rho_ref, rho, uz, ur, f, phys, err);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Ops<R>::mass(const Params<R>& p, const R* f, LinkPlanes<R> lk, double* partial, double* out, int* err,
                         cudaStream_t s) {
    const int blocks = reduce_blocks((long long)p.nz * p.nr);
    k_mass<R><<<blocks, 256, 0, s>>>(p, f, lk, partial, err);
    k_reduce_final<2><<<1, 256, 0, s>>>(partial, blocks, out);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Ops<R>::pjump(const Params<R>& p, const Params<double>& pd, const R* f, LinkPlanes<R> lk, double zc,
                          double rc, double rin, double rout, double* partial, double* out, int* err,
                          cudaStream_t s) {
    const int blocks = reduce_blocks((long long)p.nz * p.nr);
    k_pjump<R><<<blocks, 256, 0, s>>>(p, pd, f, lk, zc, rc, rin, rout, partial, err);
    k_reduce_final<4><<<1, 256, 0, s>>>(partial, blocks, out);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Ops<R>::take_error(int* err, int* host, cudaStream_t s) {
    return launch_early(k_take_error, 1, 1, s, err, host);
}

// Batched marching forms (FP32): strip width kStripNarrow or kStripWide (the autotuner picks), force and
// axis terms compiled in or out.
// Resident CTAs per SM the launch bounds ask for: what shared memory allows at each width (45.3 KB /
// 26.9 KB of rings).
template <typename R, int TZ>
struct BatchMinBlocks {
    static constexpr int value = TZ == kStripWide ? 4 : 5;
};

template <typename R, int TZ>
struct BatchTile {
    static constexpr int RR = 2;
    static constexpr int CP = StepTile<R>::CP;
    static constexpr int MINB = BatchMinBlocks<R, TZ>::value;
    static constexpr int NT = StepShape<TZ, RR, CP>::NT;
    static size_t smem() { return sizeof(R) * (size_t)StepShape<TZ, RR, CP>::elems; }
};

template <typename R, int TZ, bool MP, bool AX>
static auto batch_kernel() {
    return k_step_batch<R, TZ, BatchTile<R, TZ>::RR, BatchTile<R, TZ>::CP, BatchTile<R, TZ>::MINB, MP, AX>;
}

template <typename R, int FV>
static auto single_kernel() {
    constexpr int TZ = kStripWide;
    return k_step_single<R, TZ, BatchTile<R, TZ>::RR, BatchTile<R, TZ>::CP, BatchTile<R, TZ>::MINB, FV>;
}

template <typename R>
static cudaError_t single_prepare() {
    const int smem = (int)BatchTile<R, kStripWide>::smem();
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(single_kernel<R, FV_GUO>(), a, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(single_kernel<R, FV_LINK>(), a, smem);
    return e == cudaSuccess ? cudaFuncSetAttribute(single_kernel<R, FV_GUO | FV_LINK>(), a, smem) : e;
}

template <typename R, int TZ>
static cudaError_t batch_prepare() {
    const int smem = (int)BatchTile<R, TZ>::smem();
    cudaError_t e = cudaFuncSetAttribute(batch_kernel<R, TZ, true, true>(),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(batch_kernel<R, TZ, true, false>(), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(batch_kernel<R, TZ, false, true>(), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(batch_kernel<R, TZ, false, false>(),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e;
}

template <typename R, int TZ, bool MP, bool AX>
static auto table_kernel() {
    return k_step_table<R, TZ, BatchTile<R, TZ>::RR, BatchTile<R, TZ>::CP, BatchTile<R, TZ>::MINB, MP, AX>;
}

template <typename R, int TZ>
static cudaError_t table_prepare() {
    const int smem = (int)BatchTile<R, TZ>::smem();
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(table_kernel<R, TZ, true, true>(), a, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(table_kernel<R, TZ, true, false>(), a, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(table_kernel<R, TZ, false, true>(), a, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(table_kernel<R, TZ, false, false>(), a, smem);
    return e;
}

template <typename R, int TZ>
static cudaError_t launch_table(const BatchTable<R>& table, const Tile* tiles, const int* first, int ncta, bool mp,
                                bool ax, int parity, int* err, cudaStream_t s) {
    using T = BatchTile<R, TZ>;
    const size_t smem = T::smem();
    if (mp && ax)
        table_kernel<R, TZ, true, true>()<<<ncta, T::NT, smem, s>>>(table, tiles, first, parity, err);
    else if (mp)
        table_kernel<R, TZ, true, false>()<<<ncta, T::NT, smem, s>>>(table, tiles, first, parity, err);
    else if (ax)
        table_kernel<R, TZ, false, true>()<<<ncta, T::NT, smem, s>>>(table, tiles, first, parity, err);
    else
        table_kernel<R, TZ, false, false>()<<<ncta, T::NT, smem, s>>>(table, tiles, first, parity, err);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Ops<R>::step_table(const BatchTable<R>& table, const Tile* tiles, const int* first, int ncta, bool mp,
                               bool ax, int parity, int strip, int* err, cudaStream_t s) {
    if constexpr (sizeof(R) == 4) {
        if (ncta <= 0) return cudaErrorInvalidConfiguration;
        return strip == kStripNarrow
                   ? launch_table<R, kStripNarrow>(table, tiles, first, ncta, mp, ax, parity, err, s)
                   : launch_table<R, kStripWide>(table, tiles, first, ncta, mp, ax, parity, err, s);
    } else {
        return cudaErrorNotSupported;
    }
}

template <typename R>
int Ops<R>::batch_resident_ctas(int strip) {
    if constexpr (sizeof(R) == 8) {
        return 0;  // FP64 steps by phases
    } else {
    static int cached[2] = {0, 0};
    const int slot = strip == kStripNarrow ? 0 : 1;
    if (cached[slot] > 0) return cached[slot];
    if ((strip == kStripNarrow ? batch_prepare<R, kStripNarrow>() : batch_prepare<R, kStripWide>()) != cudaSuccess) return 0;
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    cudaError_t e = strip == kStripNarrow ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                      &per_sm, batch_kernel<R, kStripNarrow, true, true>(), BatchTile<R, kStripNarrow>::NT,
                                      BatchTile<R, kStripNarrow>::smem())
                                : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                      &per_sm, batch_kernel<R, kStripWide, true, true>(), BatchTile<R, kStripWide>::NT,
                                      BatchTile<R, kStripWide>::smem());
    if (e != cudaSuccess || per_sm < 1) per_sm = 1;
    cached[slot] = sms * per_sm;
    return cached[slot];
    }
}

template <typename R, int TZ>
static cudaError_t launch_batch(const BatchSolve<R>* solves, const Tile* tiles, const int* first, int ncta, bool mp,
                                bool ax, int parity, int* err, cudaStream_t s) {
    using T = BatchTile<R, TZ>;
    const size_t smem = T::smem();
    if (mp && ax)
        batch_kernel<R, TZ, true, true>()<<<ncta, T::NT, smem, s>>>(solves, tiles, first, parity, err);
    else if (mp)
        batch_kernel<R, TZ, true, false>()<<<ncta, T::NT, smem, s>>>(solves, tiles, first, parity, err);
    else if (ax)
        batch_kernel<R, TZ, false, true>()<<<ncta, T::NT, smem, s>>>(solves, tiles, first, parity, err);
    else
        batch_kernel<R, TZ, false, false>()<<<ncta, T::NT, smem, s>>>(solves, tiles, first, parity, err);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Ops<R>::step_single(const BatchSolve<R>& solve, const LinkSets<R>& h, const Tile* tiles, const int* first,
                                int ncta, bool mp, bool ax, int parity, int* err, cudaStream_t s, int fv) {
    if constexpr (sizeof(R) == 4) {
        using T = BatchTile<R, kStripWide>;
        if (ncta <= 0) return cudaErrorInvalidConfiguration;
        const size_t smem = T::smem();
        if (fv == 0 || !(mp && ax)) return cudaErrorInvalidValue;
        if (fv == FV_GUO)
            single_kernel<R, FV_GUO>()<<<ncta, T::NT, smem, s>>>(solve, h, tiles, first, parity, err);
        else if (fv == FV_LINK)
            single_kernel<R, FV_LINK>()<<<ncta, T::NT, smem, s>>>(solve, h, tiles, first, parity, err);
        else
            single_kernel<R, FV_GUO | FV_LINK>()<<<ncta, T::NT, smem, s>>>(solve, h, tiles, first, parity, err);
        return cudaGetLastError();
    } else {
        return cudaErrorNotSupported;
    }
}

template <typename R>
cudaError_t Ops<R>::step_batch(const BatchSolve<R>* solves, const Tile* tiles, const int* first, int ncta, bool mp,
                               bool ax, int parity, int strip, int* err, cudaStream_t s) {
    if constexpr (sizeof(R) == 4) {
        if (ncta <= 0) return cudaErrorInvalidConfiguration;
        return strip == kStripNarrow
                   ? launch_batch<R, kStripNarrow>(solves, tiles, first, ncta, mp, ax, parity, err, s)
                   : launch_batch<R, kStripWide>(solves, tiles, first, ncta, mp, ax, parity, err, s);
    } else {
        return cudaErrorNotSupported;
    }
}

// ------------------------------------------------------------ phase launches --

template <typename R, int TR, bool MP, bool AX, int FV>
static cudaError_t phases(const PhaseOne<R>& a, unsigned grid, cudaStream_t s) {
    const unsigned ghost = AX && a.s.p.top != TOP_PERIODIC ? a.across : 0;
    // the gather and the collision read no halo of their own rows: 4 rows per block keep more warps resident
    // (1023 x 511 Guo 21.6 -> 20.3 us)
    const unsigned grid4 = a.across * (unsigned)((a.s.p.nr + 3) / 4);
    cudaError_t e = launch_early(k_phase_l<R, 4, MP, (FV & FV_LINK) != 0>, grid4, 128, s, a);
    if (e == cudaSuccess) e = launch_early(k_phase_u<R, TR, MP, AX>, grid + ghost, 32 * TR, s, a);
    if (e == cudaSuccess) e = launch_early(k_phase_c<R, 4, AX, FV>, grid4, 128, s, a);
    return e;
}
template <typename R, int TR>
static cudaError_t phases_of(const BatchSolve<R>& v, const LinkSets<R>& h, bool mp, bool ax, int parity, int* err,
                             cudaStream_t s, int fv) {
    const int across = (v.p.nz + PhaseShape<R>::TZ - 1) / PhaseShape<R>::TZ;
    const unsigned grid = (unsigned)across * (unsigned)((v.p.nr + TR - 1) / TR);
    const PhaseOne<R> a{v, parity ? h.h_b : h.h_a, parity ? const_cast<R*>(h.h_a) : h.h_b, parity, across, err};
    if (fv == FV_GUO && mp && ax) return phases<R, TR, true, true, FV_GUO>(a, grid, s);
    if (fv == FV_LINK && mp && ax) return phases<R, TR, true, true, FV_LINK>(a, grid, s);
    if (fv == (FV_GUO | FV_LINK) && mp && ax) return phases<R, TR, true, true, FV_GUO | FV_LINK>(a, grid, s);
    if (fv != 0) return cudaErrorInvalidValue;
    if (mp && ax) return phases<R, TR, true, true, 0>(a, grid, s);
    if (mp) return phases<R, TR, true, false, 0>(a, grid, s);
    if (ax) return phases<R, TR, false, true, 0>(a, grid, s);
    return phases<R, TR, false, false, 0>(a, grid, s);
}

template <typename R, int TR, bool MP, bool AX>
static cudaError_t phases_many(const PhaseMany<R>& a, unsigned grid, unsigned ghost, cudaStream_t s) {
    cudaError_t e = launch_early(k_phase_l_many<R, TR, MP>, grid, 32 * TR, s, a);
    if (e == cudaSuccess) e = launch_early(k_phase_u_many<R, TR, MP, AX>, grid + (AX ? ghost : 0), 32 * TR, s, a);
    if (e == cudaSuccess) e = launch_early(k_phase_c_many<R, TR, AX>, grid, 32 * TR, s, a);
    return e;
}
template <typename R, int TR>
static cudaError_t phases_many_of(const PhaseMany<R>& a, unsigned grid, unsigned ghost, bool mp, bool ax,
                                  cudaStream_t s) {
    if (mp && ax) return phases_many<R, TR, true, true>(a, grid, ghost, s);
    if (mp) return phases_many<R, TR, true, false>(a, grid, ghost, s);
    if (ax) return phases_many<R, TR, false, true>(a, grid, ghost, s);
    return phases_many<R, TR, false, false>(a, grid, ghost, s);
}

template <typename R>
int Ops<R>::phase_tile_z() {
    return PhaseShape<R>::TZ;
}

// Rows per tile: 8, or 4 while 8 would leave SMs without a tile or, in FP64, unevenly loaded (its blocks are
// bound by their SM's arithmetic rate, and 8 rows compute less halo: 500 x 250 70 us per step with 4 rows and
// 78 with 8, 512 x 512 147 and 143, 1024 x 512 282 and 275).
template <typename R>
int Ops<R>::phase_rows(long long nodes) {
    return nodes <= 152LL * 8 * PhaseShape<R>::TZ * (sizeof(R) == 8 ? 4 : 1) ? 4 : 8;
}

template <typename R>
cudaError_t Ops<R>::phase_step(const BatchSolve<R>& v, const LinkSets<R>& h, bool mp, bool ax, int parity, int* err,
                               cudaStream_t s, int fv) {
    return phase_rows((long long)v.p.nz * v.p.nr) == 4 ? phases_of<R, 4>(v, h, mp, ax, parity, err, s, fv)
                                                       : phases_of<R, 8>(v, h, mp, ax, parity, err, s, fv);
}

template <typename R>
cudaError_t Ops<R>::phase_step_many(const BatchSolve<R>* solves, const PhaseTile* tiles, int ntiles, int nghost,
                                    int rows, bool mp, bool ax, int parity, int* err, cudaStream_t s) {
    if (ntiles <= 0) return cudaErrorInvalidConfiguration;
    const PhaseMany<R> a{solves, tiles, parity, err};
    return rows == 4 ? phases_many_of<R, 4>(a, (unsigned)ntiles, (unsigned)nghost, mp, ax, s)
                     : phases_many_of<R, 8>(a, (unsigned)ntiles, (unsigned)nghost, mp, ax, s);
}

// -------------------------------------------------------------- field passes --

template <int TR>
static cudaError_t fields64(const BatchSolve<double>& v, const LinkPlanes<double>& lk, const Params<double>& pd,
                            int parity, const FieldsOut<double>& out, int* err, cudaStream_t s) {
    const int across = (v.p.nz + PhaseShape<double>::TZ - 1) / PhaseShape<double>::TZ;
    const unsigned grid = (unsigned)across * (unsigned)((v.p.nr + TR - 1) / TR);
    const PhaseOne<double> a{v, lk.src, lk.dst, parity, across, err, true};
    const bool mp = v.p.multiphase != 0, ax = v.p.axis != 0;
    cudaError_t e;
    if (mp)
        e = lk.src ? launch_early(k_phase_l<double, TR, true, true>, grid, 32 * TR, s, a)
                   : launch_early(k_phase_l<double, TR, true, false>, grid, 32 * TR, s, a);
    else
        e = lk.src ? launch_early(k_phase_l<double, TR, false, true>, grid, 32 * TR, s, a)
                   : launch_early(k_phase_l<double, TR, false, false>, grid, 32 * TR, s, a);
    if (e != cudaSuccess) return e;
    if (mp && ax) return launch_early(k_fields64<TR, true, true>, grid, 32 * TR, s, a, out, pd);
    if (mp) return launch_early(k_fields64<TR, true, false>, grid, 32 * TR, s, a, out, pd);
    return launch_early(k_fields64<TR, false, false>, grid, 32 * TR, s, a, out, pd);
}

template <typename R>
cudaError_t Ops<R>::fields(const BatchSolve<R>& v, LinkPlanes<R> lk, const Params<double>& pd, int parity, double* rho,
                           double* uz, double* ur, double* pk, R* u, int* err, cudaStream_t s) {
    const FieldsOut<R> out{rho, uz, ur, pk, u};
    if constexpr (sizeof(R) == 8) {
        return phase_rows((long long)v.p.nz * v.p.nr) == 4 ? fields64<4>(v, lk, pd, parity, out, err, s)
                                                           : fields64<8>(v, lk, pd, parity, out, err, s);
    } else {
        // 16 rows per block, 8 while that leaves SMs without one
        const int across = (v.p.nz + 31) / 32;
        const R* f = parity ? v.f_b : v.f_a;
        if ((long long)v.p.nz * v.p.nr <= 2 * 152 * 512)
            return launch_early(k_fields<8>, across * ((v.p.nr + 7) / 8), 256, s, v.p, pd, f, lk, out, err);
        if ((long long)v.p.nz * v.p.nr > 1000000)
            return launch_early(k_fields<32>, across * ((v.p.nr + 31) / 32), 256, s, v.p, pd, f, lk, out, err);
        return launch_early(k_fields<16>, across * ((v.p.nr + 15) / 16), 256, s, v.p, pd, f, lk, out, err);
    }
}

}  // namespace lbm
