// One FP32 time step as one launch over tiles of nodes, for the smallest grids.
//
// Three phase launches (lbm_phase.cuh) cost about 2 us each however little they
// do.  Here a CTA gathers its tile with 6 columns and rows around it and takes
// all stages in shared memory: more work in all (L runs on (TZ + 12)(TR + 12)
// nodes for TZ x TR results), one launch.  What bounds it is the latency of the
// four stages in a row, so every stage has one item per thread or little more,
// and the collision's own populations are gathered first of all.  us per step,
// phases -> tiles: 64 x 64 6.2 -> 3.1, 512 x 256 9.3 -> 7.8; tile_form has more.
//
// The packed operations and their order are those of march2 (lbm_step.cuh), so
// the results are the same bits.  (Not with Guo forcing: the compiler fuses a
// sum of its longer collision differently here, which grows to 5e-5 of the
// velocities in 200 steps; those solves step by phases and, when large, by
// marching CTAs.)
#pragma once

#include "lbm_phase.cuh"

namespace lbm {

// TZ x TR nodes per CTA of NT threads.
template <int TZ_, int TR_, int NT_, bool AX>
struct TileStep {
    static constexpr int TZ = TZ_, TR = TR_, NT = NT_;
    // halo of psi (columns, rows), of its derivatives, of rho, j and u
    static constexpr int LZ = AX ? 6 : 2, LR = AX ? 6 : 1, D = 4, U = AX ? 2 : 0;
    static constexpr int WL = TZ + 2 * LZ, HL = TR + 2 * LR;
    static constexpr int WD = TZ + 2 * D, HD = TR + 2 * D;
    static constexpr int WU = TZ + 2 * U, HU = TR + 2 * U;
    static constexpr int elems = WL * HL + (AX ? 2 * WD * HD : 0) + 5 * WU * HU;
    static_assert(TZ * TR / 2 <= NT, "one collision item per thread");
};

// Populations arriving at row j for the pair of columns c[1], c[2] between c[0] and c[3] (all wrapped).
template <bool EDGE>
__device__ __forceinline__ void pull_pair(const Params<float>& p, const float* __restrict__ f, int j, const int (&c)[4],
                                          float2 (&fi)[Q]) {
    const PullRow q = pull_row(p, j);
#pragma unroll
    for (int i = 0; i < Q; i++) {
        const float* r = f + q.o[i];
        const int s = (i == 6 || i == 7) && q.stay ? 1 : 1 - cz_of(i);
        if (cz_of(i) == 0 && !EDGE)
            fi[i] = *reinterpret_cast<const float2*>(r + c[1]);
        else
            fi[i] = s == 0 ? pk(r[c[0]], r[c[1]]) : (s == 1 ? pk(r[c[1]], r[c[2]]) : pk(r[c[2]], r[c[3]]));
    }
}

template <typename S, bool MP, bool AX, bool EDGE>
__device__ __forceinline__ void tile_step(const Params<float>& p, const PhaseWork<float>& w, float* smem, int word) {
    using T = float2;
    constexpr int NT = S::NT, LZ = S::LZ, LR = S::LR, WL = S::WL, WD = S::WD, WU = S::WU;
    float* sPsi = smem;
    float* sRho = sPsi + WL * S::HL;
    float* sJz = sRho + WU * S::HU;
    float* sJr = sJz + WU * S::HU;
    float* sUz = sJr + WU * S::HU;
    float* sUr = sUz + WU * S::HU;
    float* sPz = sUr + WU * S::HU;
    float* sPr = sPz + WD * S::HD;
    const int tid = threadIdx.x, nz = p.nz, nr = p.nr, k0 = w.k0, j0 = w.j0;
    const bool periodic = p.top == TOP_PERIODIC;
    const int jn = min(S::TR, nr - j0), kn = EDGE ? min(S::TZ, nz - k0) : S::TZ;
    const T zero = pk(0.0f, 0.0f), ref = pk(p.rho_ref, p.rho_ref);
    const T la[3] = {zero, zero, zero};  // no link source in this form
    // columns k - 1 .. k + 2, wrapped: by one period unless the grid is narrower than the tile
    auto columns = [&](int k, int(&c)[4]) {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            c[q] = k - 1 + q;
            if (EDGE) c[q] = nz >= S::TZ + 16 ? wrap_small(c[q], nz) : wrap_any(c[q], nz);
        }
    };
    int bad = 0;
    // the collision's own populations
    const int ct = tid / (S::TZ / 2), cc = 2 * (tid - ct * (S::TZ / 2)), crow = j0 + ct;
    const bool collides = ct < jn && cc < kn;
    T cf[Q];
    if (collides) {
        int c[4];
        columns(k0 + cc, c);
        pull_pair<EDGE>(p, w.f, crow, c, cf);
    }
    // ---- rho, j, psi
    for (int i = tid; i < WL / 2 * S::HL; i += NT) {
        const int a = i / (WL / 2), b = 2 * (i - a * (WL / 2)), row = j0 - LR + a;
        if (a >= jn + 2 * LR || b >= kn + 2 * LZ) continue;
        const int iu = a - (LR - S::U), bu = b - (LZ - S::U);
        const bool own = iu >= 0 && iu < jn + 2 * S::U && bu >= 0 && bu < WU;
        if (!MP && !own) continue;
        int c[4];
        columns(k0 - LZ + b, c);
        T f[Q], drho, jz, jr;
        pull_pair<EDGE>(p, w.f, mirror_row(row, nr, periodic), c, f);
        moments2<false, float>(f, la, drho, jz, jr);
        const T psi = psi2<MP>(p, drho, true, bad);
        if (MP) st2(sPsi + a * WL, b, psi);
        if (own) {
            st2(sRho + iu * WU, bu, drho);
            st2(sJz + iu * WU, bu, jz);
            st2(sJr + iu * WU, bu, !periodic && (row < 0 || row >= nr) ? psub(zero, jr) : jr);
        }
    }
    __syncthreads();
    // ---- psi_z, psi_r
    if (MP && AX) {
        for (int i = tid; i < WD / 2 * S::HD; i += NT) {
            const int a = i / (WD / 2), b = 2 * (i - a * (WD / 2));
            if (a >= jn + 2 * S::D || b >= kn + 2 * S::D) continue;
            int er = j0 - S::D + a;
            const bool above = !periodic && er >= nr;  // beyond the wall: the mirror row, psi_r odd
            if (above) er = 2 * nr - 1 - er;
            const float* m = sPsi + (er - j0 + LR) * WL;
            T dz, dr;
            fd_both2<float>(m - 2 * WL, m - WL, m, m + WL, m + 2 * WL, b + (LZ - S::D), dz, dr);
            st2(sPz + a * WD, b, dz);
            st2(sPr + a * WD, b, above ? psub(zero, dr) : dr);
        }
        __syncthreads();
    }
    // ---- force and u
    for (int i = tid; i < WU / 2 * S::HU; i += NT) {
        const int a = i / (WU / 2), b = 2 * (i - a * (WU / 2)), row = j0 - S::U + a;
        if (a >= jn + 2 * S::U || b >= kn + 2 * S::U || (!periodic && row >= nr)) continue;
        const T rho = padd(ld2<T>(sRho + a * WU, b), ref);
        T fz = pmul(rho, pk(p.gz, p.gz)), fr = zero;
        if (MP) {
            const float* m = sPsi + (row - j0 + LR) * WL;
            const int c = b + (LZ - S::U);
            const Tri<T> z0 = ld3<T>(m, c), zm = ld3<T>(m - WL, c), zq = ld3<T>(m + WL, c);
            force_k2(p, zm, z0, zq, fz, fr);
            if (AX) {
                const float* r = sPr + (row - j0 + S::D) * WD;
                const float* z = sPz + (row - j0 + S::D) * WD;
                const int d = b + (S::D - S::U);
                const T prr = fd_r2<float, T>(r - 2 * WD, r - WD, r + WD, r + 2 * WD, d);
                const T prz = fd_r2<float, T>(z - 2 * WD, z - WD, z + WD, z + 2 * WD, d);
                const int rrow = periodic ? mirror_row(row, nr, true) : row;
                force_axis2(p, rho, z0.b, ld2<T>(z, d), ld2<T>(r, d), prr, prz, rrow, fz, fr);
            }
        }
        T vz, vr;
        velocity2<float>(rho, ld2<T>(sJz + a * WU, b), ld2<T>(sJr + a * WU, b), fz, fr, vz, vr);
        st2(sUz + a * WU, b, vz);
        st2(sUr + a * WU, b, vr);
    }
    __syncthreads();
    // ---- collide
    const int earlier = earlier_error(word, w.parity);
    bad |= earlier;
    if (bad) atomicOr(w.err, err_of_step(bad, w.parity));
    if (!collides || earlier) return;
    const int b = cc + S::U;
    const int o0 = (ct + S::U) * WU;
    const T drho = ld2<T>(sRho + o0, b), uz = ld2<T>(sUz + o0, b), ur = ld2<T>(sUr + o0, b);
    T Hz = zero, Hr = zero, mir = zero, rur = zero;
    if (AX) {
        Tri<T> z[5], r[5];
#pragma unroll
        for (int q = 0; q < 5; q++) {
            const int row = crow + q - 2;
            const bool above = !periodic && row >= nr;  // beyond the wall: the mirror row with signs
            const int o = ((above ? 2 * nr - 1 - row : row) - j0 + S::U) * WU;
            r[q] = ld3<T>(sUr + o, b);
            if (above) r[q] = {psub(zero, r[q].a), psub(zero, r[q].b), psub(zero, r[q].c)};
            if (q == 2) continue;
            z[q] = ld3<T>(sUz + o, b);
            if (above && p.top == TOP_NOSLIP) z[q] = {psub(zero, z[q].a), psub(zero, z[q].b), psub(zero, z[q].c)};
        }
        const T duz_dr = fd_r3<float, T>(z[0], z[1], z[3], z[4]);
        T dur_dz, dur_dr;
        fd_both3<float>(r[0], r[1], r[2], r[3], r[4], dur_dz, dur_dr);
        source2(p, padd(drho, ref), uz, ur, duz_dr, dur_dz, dur_dr, crow, Hz, Hr, mir, rur);
    }
    const int plane = (int)p.plane, k = k0 + cc;
    float* out = w.fout + (crow * p.pitch + k);
    collide2<0>(
        p, cf, la, drho, ld2<T>(sJz + o0, b), ld2<T>(sJr + o0, b), uz, ur, Hz, Hr, mir, rur,
        [&](int q, T v) {
            if (!EDGE || k + 1 < nz)
                st2(out + q * plane, 0, v);
            else
                out[q * plane] = v.x;
        },
        [](int, T) {});
}

template <typename S, bool MP, bool AX>
__device__ __forceinline__ void tile_step(const Params<float>& p, const PhaseWork<float>& w) {
    __shared__ __align__(16) float smem[S::elems];
    const int word = error_word(w.err);
    if (w.k0 >= 8 && w.k0 + S::TZ + 8 <= p.nz)
        tile_step<S, MP, AX, false>(p, w, smem, word);
    else
        tile_step<S, MP, AX, true>(p, w, smem, word);
}

template <int TZ, int TR, int NT, bool MP, bool AX>
__global__ void __launch_bounds__(NT) k_tile(const PhaseOne<float> a) {
    const int ti = blockIdx.x / a.across, tk = blockIdx.x - ti * a.across;
    phase_wait();
    tile_step<TileStep<TZ, TR, NT, AX>, MP, AX>(a.s.p, phase_work(a.s, a.parity, a.err, tk * TZ, ti * TR));
}
template <int TZ, int TR, int NT, bool MP, bool AX>
__global__ void __launch_bounds__(NT) k_tile_many(const PhaseMany<float> a) {
    const PhaseTile tl = a.tiles[blockIdx.x];
    const Params<float> p = a.s[tl.solve].p;
    phase_wait();
    tile_step<TileStep<TZ, TR, NT, AX>, MP, AX>(p, phase_work(a.s[tl.solve], a.parity, a.err + tl.solve, tl.k0, tl.j0));
}

}  // namespace lbm
