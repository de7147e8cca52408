// Launchers of the warp march (FP32; a translation unit of its own to compile beside the others).
#include "lbm_launch.h"
#include "lbm_march.cuh"

namespace lbm {

namespace {

int kind_of(const Params<float>& p) {
    return (p.eos == EOS_VDW ? WARP_VDW : WARP_CS) | (p.axis && p.kappa == KAPPA_LATTICE ? 1 : 0);
}

// One solve's kernel.  Without F_axis kappa is not used; without the force nor is the EOS.
using One = void (*)(const BatchSolve<float>, const Tile*, int, int*);
One one_mp_ax(int kind) {
    switch (kind) {
        case WARP_CS: return k_step_warp<true, true, WARP_CS>;
        case WARP_CS_LATTICE: return k_step_warp<true, true, WARP_CS_LATTICE>;
        case WARP_VDW: return k_step_warp<true, true, WARP_VDW>;
        default: return k_step_warp<true, true, WARP_VDW_LATTICE>;
    }
}
One one(const Params<float>& p, bool mp, bool ax) {
    if (mp && ax) return one_mp_ax(kind_of(p));
    if (mp) return p.eos == EOS_VDW ? k_step_warp<true, false, WARP_VDW> : k_step_warp<true, false, WARP_CS>;
    return ax ? k_step_warp<false, true, WARP_CS> : k_step_warp<false, false, WARP_CS>;
}

using Many = void (*)(const BatchSolve<float>*, const Tile*, int, int*);
Many many(int kind, bool mp, bool ax) {
    if (mp && ax) {
        switch (kind) {
            case WARP_CS: return k_step_warp_many<true, true, WARP_CS>;
            case WARP_CS_LATTICE: return k_step_warp_many<true, true, WARP_CS_LATTICE>;
            case WARP_VDW: return k_step_warp_many<true, true, WARP_VDW>;
            case WARP_VDW_LATTICE: return k_step_warp_many<true, true, WARP_VDW_LATTICE>;
            default: return k_step_warp_many<true, true, WARP_MIXED>;
        }
    }
    if (mp && kind == WARP_MIXED) return k_step_warp_many<true, false, WARP_MIXED>;
    if (mp) return kind == WARP_VDW ? k_step_warp_many<true, false, WARP_VDW> : k_step_warp_many<true, false, WARP_CS>;
    return ax ? k_step_warp_many<false, true, WARP_CS> : k_step_warp_many<false, false, WARP_CS>;
}

}  // namespace

template <>
int Ops<float>::warp_slots() {
    static int cached = 0;
    if (cached > 0) return cached;
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_step_warp<true, true, WARP_CS>, 32, 0) != cudaSuccess)
        return 0;
    return cached = sms * (per_sm > 0 ? per_sm : 1);
}

template <>
cudaError_t Ops<float>::step_warp(const BatchSolve<float>& v, const Tile* tiles, int ntiles, bool mp, bool ax, int parity,
                                  int* err, cudaStream_t s) {
    if (ntiles <= 0) return cudaErrorInvalidConfiguration;
    one(v.p, mp, ax)<<<ntiles, 32, 0, s>>>(v, tiles, parity, err);
    return cudaGetLastError();
}

template <>
int Ops<float>::warp_kind(const Params<float>& p) {
    return kind_of(p);
}
template <>
int Ops<float>::warp_kind(int a, int b) {
    return a == b ? a : (int)WARP_MIXED;
}

template <>
cudaError_t Ops<float>::step_warp_many(const BatchSolve<float>* solves, int kind, const Tile* tiles, int ntiles, bool mp,
                                       bool ax, int parity, int* err, cudaStream_t s) {
    if (ntiles <= 0) return cudaErrorInvalidConfiguration;
    many(kind, mp, ax)<<<ntiles, 32, 0, s>>>(solves, tiles, parity, err);
    return cudaGetLastError();
}

}  // namespace lbm
