// Host-side launchers of the kernels, one explicit instantiation per
// precision (kernels_f32.cu, kernels_f64.cu).
#pragma once

#include <cuda_runtime.h>

#include "lbm_device.cuh"
#include "lbm_tiles.h"

namespace lbm {

// Blocks of 256 threads of a reduction over n nodes: 8 x 152 SMs (all that fit), fewer while that leaves some
// without a node; by the size alone, so reductions are reproducible.
constexpr int reduce_blocks(long long n) { return n > 1216 * 256 ? 1216 : (int)((n + 255) / 256); }
constexpr int kStepMinRows = 16;    // the fused forms need single reflections at the walls
// FP32 solves and batches up to this many nodes, counted in whole tiles (phase_nodes), step by phases, larger
// ones by warps (with the link source or Guo forcing, a solve by CTAs).  us per step, phases and warps, by
// such nodes: 256k (500 x 500) 14.0 and 23.2, 576k 22.5 and 28.2, 749k (800 x 900) 27.0 and 29.5, 768k (65 x
// 6000) 28.8 and 29.6, 845k (900 x 880) 30.2 and 30.5, 1.15M (65 x 9000) 40.9 and 30.1, 1.28M (33 x 20000) 50 and
// 39; batches: 707k (138 x 66 x 33) 29.4 and 25.0, 774k 33.6 and 29.6, 791k (386 x 64 x 32) 34.9 and 38.1,
// 1.04M 42.8 and 31.3, 1.41M (276 x 66 x 33) 54.5 and 33.0.
constexpr long long kPhaseMaxNodes = 800000;
// z-columns per CTA of the two compiled forms of the batched kernel (the wide
// one is the default; the autotuner may pick the narrow one for small grids).
// 112: with 128 threads of two columns each, stages L, D, U and C fill 124,
// 120, 116 and 112 of them, and strip origins stay 64-byte aligned; measured
// fastest of the even widths 96 ... 116 on the 4096 x 2048 wave.
constexpr int kStripNarrow = 64, kStripWide = 112;

// Forms of the one-launch tile step (lbm_tile.cuh, FP32 with the force on) for n solves together, by their
// sizes; TILE_NONE: another kernel is faster or the form is not compiled.  tile_size: nodes of a tile.
enum TileForm { TILE_NONE, TILE_A, TILE_B, TILE_C, TILE_D };
TileForm tile_form(const int* nz, const int* nr, int n, bool mp, bool ax, int fv);
void tile_size(TileForm f, int* tz, int* tr);

template <typename R>
struct Ops {
    // kernel (a): gather, rho/j, psi; raises bits in *err.
    // lk: the link-midpoint source planes (null: h_i at the node).
    static cudaError_t density(const Params<R>& p, const R* f, R* aux, int* err, cudaStream_t s,
                               LinkPlanes<R> lk = {nullptr, nullptr});
    // kernel (b): the fused stream + force + EDM + axisymmetric source + collide step
    // (guo: Guo forcing in place of the EDM shift).
    static cudaError_t update(const Params<R>& p, const R* f, R* fout, const R* aux, cudaStream_t s,
                              LinkPlanes<R> lk = {nullptr, nullptr}, bool guo = false);
    // rho, physical u, P_k of the state in v.f_a (parity 0) or v.f_b: FP64 arrays [j * nz + k] on the device,
    // and u into two pitched planes of R (each may be null).  lk: as for density.
    static cudaError_t fields(const BatchSolve<R>& v, LinkPlanes<R> lk, const Params<double>& pd, int parity,
                              double* rho, double* uz, double* ur, double* pk, R* u, int* err, cudaStream_t s);
    // f^eq(rho, u); with phys (u + F / (2 rho) of that state, two pitched planes) f^eq(rho, u - F / (2 rho))
    // unless *err is set.
    static cudaError_t init(const Params<R>& p, double rho_ref, const double* rho, const double* uz,
                            const double* ur, R* f, cudaStream_t s, const R* phys = nullptr,
                            const int* err = nullptr);
    // kernel (c): out[0] = sum (j+1/2) (rho - rho_ref), out[1] = sum (rho - rho_ref) (host-mapped or device).
    static cudaError_t mass(const Params<R>& p, const R* f, LinkPlanes<R> lk, double* partial, double* out, int* err,
                            cudaStream_t s);
    // out[0..3] = sum P_k inside, count inside, sum P_k outside, count outside.
    static cudaError_t pjump(const Params<R>& p, const Params<double>& pd, const R* f, LinkPlanes<R> lk, double zc,
                             double rc, double rin, double rout, double* partial, double* out, int* err,
                             cudaStream_t s);
    // *host (pinned) = *err, *err = 0.
    static cudaError_t take_error(int* err, int* host, cudaStream_t s);
    // dynamic shared memory of one k_update CTA, bytes
    static size_t update_smem();
    // one-time kernel attributes (shared-memory opt-in); call outside stream capture
    static cudaError_t prepare();
    // kernel (b'): the whole step in one pass (needs nr >= kStepMinRows); rows_per_cta > 0
    // rows of each z-strip per CTA.
    static cudaError_t step(const Params<R>& p, const R* f, R* fout, int rows_per_cta, int* err, cudaStream_t s);
    // Batched fused step: ncta CTAs, CTA c marching tiles first[c] .. first[c + 1] - 1
    // (device arrays planned by plan_tiles for this strip width); strip: kStripNarrow
    // or kStripWide z-columns per CTA.  FP32 only (cudaErrorNotSupported in FP64, like
    // step_single and step_table: FP64 steps by phases).
    static cudaError_t step_batch(const BatchSolve<R>* solves, const Tile* tiles, const int* first, int ncta,
                                  bool mp, bool ax, int parity, int strip, int* err, cudaStream_t s);
    // The fused step of one solve with Guo forcing or the link source (fv; mp && ax),
    // descriptor by value, kStripWide tiles.
    static cudaError_t step_single(const BatchSolve<R>& solve, const LinkSets<R>& h, const Tile* tiles,
                                   const int* first, int ncta, bool mp, bool ax, int parity, int* err,
                                   cudaStream_t s, int fv = 0);
    // The fused step by warps (lbm_march.cuh; FP32 only): tile t on block t (plan_warp_tiles for warp_slots()),
    // of one solve or of many (EDM, h_i at the node).  kind: what the parameters of many have in common
    // (warp_kind of one, of two kinds).
    static cudaError_t step_warp(const BatchSolve<R>& solve, const Tile* tiles, int ntiles, bool mp, bool ax, int parity,
                                 int* err, cudaStream_t s);
    static cudaError_t step_warp_many(const BatchSolve<R>* solves, int kind, const Tile* tiles, int ntiles, bool mp,
                                      bool ax, int parity, int* err, cudaStream_t s);
    static int warp_kind(const Params<R>& p);
    static int warp_kind(int a, int b);
    static int warp_slots();
    // The batched step with the descriptors as one kernel argument (FP32; n <=
    // BatchTable<R>::N solves; cudaErrorNotSupported in FP64).
    static cudaError_t step_table(const BatchTable<R>& table, const Tile* tiles, const int* first, int ncta,
                                  bool mp, bool ax, int parity, int strip, int* err, cudaStream_t s);
    // The step as three phase launches (lbm_phase.cuh) of one solve, or of the tiles of
    // many (device arrays; tiles of phase_tile_z() x rows nodes, rows of phase_rows).
    static cudaError_t phase_step(const BatchSolve<R>& solve, const LinkSets<R>& h, bool mp, bool ax, int parity,
                                  int* err, cudaStream_t s, int fv = 0);
    // The list ends with nghost tiles at j0 = -2: the two rows beyond the axis of each
    // solve without a periodic top (axis terms on).
    static cudaError_t phase_step_many(const BatchSolve<R>* solves, const PhaseTile* tiles, int ntiles, int nghost,
                                       int rows, bool mp, bool ax, int parity, int* err, cudaStream_t s);
    static cudaError_t tile_step(TileForm f, const BatchSolve<R>& solve, bool ax, int parity, int* err, cudaStream_t s);
    static cudaError_t tile_step_many(TileForm f, const BatchSolve<R>* solves, const PhaseTile* tiles, int ntiles,
                                      bool ax, int parity, int* err, cudaStream_t s);
    static int phase_tile_z();
    static int phase_rows(long long nodes);
    static int batch_resident_ctas(int strip);
};

template <>
cudaError_t Ops<float>::tile_step(TileForm, const BatchSolve<float>&, bool, int, int*, cudaStream_t);
template <>
cudaError_t Ops<float>::tile_step_many(TileForm, const BatchSolve<float>*, const PhaseTile*, int, bool, int, int*,
                                       cudaStream_t);
template <>
int Ops<float>::warp_slots();
template <>
cudaError_t Ops<float>::step_warp(const BatchSolve<float>&, const Tile*, int, bool, bool, int, int*, cudaStream_t);
template <>
cudaError_t Ops<float>::step_warp_many(const BatchSolve<float>*, int, const Tile*, int, bool, bool, int, int*, cudaStream_t);
template <>
int Ops<float>::warp_kind(const Params<float>&);
template <>
int Ops<float>::warp_kind(int, int);

}  // namespace lbm
