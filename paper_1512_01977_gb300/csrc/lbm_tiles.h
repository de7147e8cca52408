// Internal: tiles of the batched step kernel and their planner (lbm_tiles.cu).
#pragma once

#include <vector>

namespace lbm {

// Rows [j0, jend) of z-strip `strip` of solve `solve`.
struct Tile {
    int solve, strip, j0, jend;
};

// A tile of the phase kernels: columns from k0 and rows from j0 of solve `solve`.
struct PhaseTile {
    int solve, k0, j0;
};

// Columns of an FP32 phase tile, and the nodes of a grid with its last tiles (of 8 rows) counted whole: what
// the phases' time goes by, as a tile computes all its nodes.
constexpr int kPhaseColumns = 64;
inline long long phase_nodes(int nz, int nr) {
    return (long long)((nz + kPhaseColumns - 1) / kPhaseColumns) * kPhaseColumns * ((nr + 7) / 8) * 8;
}

// Pipeline rows a tile costs beyond its own: 6 halo rows above it and the 12-row
// lag between the first and the last marching stage.
constexpr int kTileFillRows = 18;
// The same of the warp march (lbm_march.cuh), and the columns a warp stores.
constexpr int kWarpFillRows = 13, kWarpStrip = 52;

// Plan for n solves (nz[i] x nr[i]), z-strips of `strip` columns, `slots` CTAs:
// tiles in CTA order, first[c] .. first[c + 1] those of CTA c (first has one entry
// per CTA with work, plus one).  Returns LBM_OK, LBM_ERR_INVALID_ARG or LBM_ERR_OOM.
// fill: pipeline rows a tile costs beyond its own.
int plan_tiles(const int* nz, const int* nr, int n, int strip, int slots, std::vector<Tile>& tiles,
               std::vector<int>& first, long long* makespan, int fill = kTileFillRows);

// Tiles of the warp march for `slots` resident warps, one block each, the tallest first (the hardware
// starts a block wherever one ends, which deals them as plan_tiles does).
int plan_warp_tiles(const int* nz, const int* nr, int n, int slots, std::vector<Tile>& tiles);

}  // namespace lbm
