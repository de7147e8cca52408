// Launchers of the one-launch tile step (FP32; a translation unit of its own to compile beside the others).
#include "lbm_early.cuh"
#include "lbm_launch.h"
#include "lbm_tile.cuh"

namespace lbm {

namespace {

template <int TZ, int TR, int NT>
struct Form {
    static constexpr int tz = TZ, tr = TR, nt = NT;
};
using TileA = Form<16, 8, 288>;
using TileB = Form<16, 16, 416>;
using TileC = Form<32, 16, 320>;
using TileD = Form<32, 8, 256>;

template <typename F, bool AX>
cudaError_t one(const BatchSolve<float>& v, int parity, int* err, cudaStream_t s) {
    const int across = (v.p.nz + F::tz - 1) / F::tz;
    const unsigned grid = (unsigned)across * (unsigned)((v.p.nr + F::tr - 1) / F::tr);
    return launch_early(k_tile<F::tz, F::tr, F::nt, true, AX>, grid, F::nt, s,
                        PhaseOne<float>{v, nullptr, nullptr, parity, across, err});
}
template <typename F, bool AX>
cudaError_t many(const PhaseMany<float>& a, int ntiles, cudaStream_t s) {
    return launch_early(k_tile_many<F::tz, F::tr, F::nt, true, AX>, (unsigned)ntiles, F::nt, s, a);
}

}  // namespace

// us per step of A (16 x 8 nodes per CTA), B (16 x 16), C (32 x 16), D (32 x 8) and the phases, axis terms
// on: 64 x 64 3.1, 3.6, 5.5, 4.6, 6.2; 256 x 128 4.1, 3.7, 6.3, 4.6, 7.1; 300 x 200 6.9, 5.6, 6.7, 5.7, 8.0;
// 512 x 256 11, 9.3, 7.8, 10, 9.3; 512 x 512 19, 17, 14, 16, 13.9.  So: the smallest tile that gives no SM
// two of them, 16 x 16 while none has three, then the one with the least halo.  Axis terms off (psi one
// row and column around): 500 x 500 11.7, 10.4, 7.9, 6.7, 9.8; 700 x 700 20, 18, 13.9, 11.1, 15.4.
TileForm tile_form(const int* nz, const int* nr, int n, bool mp, bool ax, int fv) {
    if (!mp || fv) return TILE_NONE;
    constexpr long long kSms = 152, kMost = 200000;
    long long a = 0, b = 0, nodes = 0;
    for (int i = 0; i < n; i++) {
        if (nr[i] < kStepMinRows) return TILE_NONE;
        a += (long long)((nz[i] + 15) / 16) * ((nr[i] + 7) / 8);
        b += (long long)((nz[i] + 15) / 16) * ((nr[i] + 15) / 16);
        nodes += (long long)nz[i] * nr[i];
    }
    if (a <= kSms) return TILE_A;
    if (!ax) return nodes <= kPhaseMaxNodes ? TILE_D : TILE_NONE;
    if (b <= 2 * kSms) return TILE_B;
    return nodes <= kMost ? TILE_C : TILE_NONE;
}

void tile_size(TileForm f, int* tz, int* tr) {
    *tz = f == TILE_C || f == TILE_D ? 32 : 16;
    *tr = f == TILE_A || f == TILE_D ? 8 : 16;
}

template <>
cudaError_t Ops<float>::tile_step(TileForm f, const BatchSolve<float>& v, bool ax, int parity, int* err, cudaStream_t s) {
    if (!ax) return f == TILE_A ? one<TileA, false>(v, parity, err, s) : one<TileD, false>(v, parity, err, s);
    return f == TILE_A ? one<TileA, true>(v, parity, err, s)
                       : (f == TILE_B ? one<TileB, true>(v, parity, err, s) : one<TileC, true>(v, parity, err, s));
}

template <>
cudaError_t Ops<float>::tile_step_many(TileForm f, const BatchSolve<float>* solves, const PhaseTile* tiles, int ntiles,
                                       bool ax, int parity, int* err, cudaStream_t s) {
    if (ntiles <= 0) return cudaErrorInvalidConfiguration;
    const PhaseMany<float> a{solves, tiles, parity, err};
    if (!ax) return f == TILE_A ? many<TileA, false>(a, ntiles, s) : many<TileD, false>(a, ntiles, s);
    return f == TILE_A ? many<TileA, true>(a, ntiles, s)
                       : (f == TILE_B ? many<TileB, true>(a, ntiles, s) : many<TileC, true>(a, ntiles, s));
}

}  // namespace lbm
