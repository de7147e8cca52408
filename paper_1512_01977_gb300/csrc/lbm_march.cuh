// The single-pass step for large FP32 grids: one warp marches one z-strip down
// its rows, every lane owning a pair of columns, and nothing is shared between
// warps.
//
// The turn that reads row l does
//
//   L  row l      gathers 9 populations: rho, j, psi
//   D  row l - 2  psi_z, psi_r and the Kupershtokh force from psi rows l-4 .. l
//   U  row l - 5  F_axis from the psi derivatives of rows l-7 .. l-3, F, u
//   C  row l - 7  velocity gradients from u of rows l-9 .. l-5, H, collision
//
// Vertical neighbours are the lane's own values of the last rows, in registers
// or in shared memory that only the lane itself reads back; horizontal ones
// come from the neighbouring lanes by shuffles of the column sums and
// differences, which every lane forms once for its own pair.  A warp of 32
// pairs loses one pair on each side per stage: 64 columns in, 52 out.  There
// are no barriers.  Global traffic is the populations only (72 B per node plus
// the strip's halo; C gathers again, mostly from L1 and L2).
//
// What bounds it: with 168 registers 12 warps fit an SM, which issue on 54 % of
// the cycles; the LSU data pipe (shuffles, gathers, the ring) is 68 % busy.  So
// the turn of an interior row is one straight line without a condition (EOS
// and kappa known to the compiler), in which L -> D and U -> C are independent
// chains; u sits in registers and only psi_z, psi_r, rho and j in the ring.
// 4096 x 2048: 153 us per step, 54,800 MLUPS; march2 with its barriers and 48
// shared-memory reads per node takes 208.  Measured on the way: conditions in
// the loop 198-211, u in the ring too 168, 15 warps of 128 registers 247 (the
// gathers of C then miss L1), 8 warps 174, rows unrolled by 2 168 (spills) and
// by 5 262 (instruction fetch).
//
// The packed operations and their order are those of march2 (lbm_step.cuh), so
// the results are the same bits.  (Not with Guo forcing: the compiler fuses a
// sum of its longer collision differently here, which grows to 5e-5 of the
// velocities in 200 steps; those solves step by phases and, when large, by
// marching CTAs.)
#pragma once

#include <type_traits>

#include "lbm_phase.cuh"

namespace lbm {

struct WarpShape {
    static constexpr int TZ = kWarpStrip;  // columns a warp stores
    static constexpr int kFirst = 3;       // the lanes that store: kFirst .. 31 - kFirst
    static constexpr int kRing = 8;        // rows of the ring: rho, j (l - 7 .. l), psi_z, psi_r (l - 7 .. l - 2)
    static constexpr int kRow = 160;       // pairs of a ring row
    static constexpr int kWarps = 12;      // per SM: 168 registers
};

__device__ __forceinline__ float from_left(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float from_right(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float2 from_left(float2 v) { return pk(from_left(v.x), from_left(v.y)); }
__device__ __forceinline__ float2 from_right(float2 v) { return pk(from_right(v.x), from_right(v.y)); }

// D_r from the row differences of the own pair, d1 = row r+1 - row r-1 and d2 = row r+2 - row r-2 (fd_r3).
__device__ __forceinline__ float2 lane_dr(float2 d1, float2 d2, float d1l, float d1r) {
    const float t = d1.x + d1.y;
    const float2 n1 = pk(d1l + t, d1r + t);
    const float2 n2 = padd(padd(from_left(d2), d2), from_right(d2));
    return pfma(n1, pk(8.0f / 36.0f, 8.0f / 36.0f), pmul(n2, pk(-1.0f / 36.0f, -1.0f / 36.0f)));
}
// D_z from the row sums s1 (r, r+1, r-1) and s2 (r, r+2, r-2) of the own pair (fd_both3).
__device__ __forceinline__ float2 lane_dz(float2 s1, float2 s2) {
    const float2 n1 = pk(s1.y - from_left(s1.y), from_right(s1.x) - s1.x);
    const float2 n2 = psub(from_right(s2), from_left(s2));
    return pfma(n1, pk(8.0f / 36.0f, 8.0f / 36.0f), pmul(n2, pk(-1.0f / 36.0f, -1.0f / 36.0f)));
}

// Where the lane's populations come from: the nine planes shifted to their source rows (uniform), the
// wrapped columns k - 1, k, k + 1, k + 2.
struct LaneSource {
    const float* base[Q];
    int c[4];
};

// Populations arriving at the lane's nodes of row j.  LAST: the last read of these values in the step.
template <bool FULL, bool PAIR, bool LAST>
__device__ __forceinline__ void lane_pull(const Params<float>& p, const float* __restrict__ f, const LaneSource& s,
                                          int j, float2 (&fi)[Q]) {
    auto ld = [](const float* a) { return LAST ? __ldcs(a) : *a; };
    if (FULL || (j >= 1 && j + 1 < p.nr)) {
        unsigned o[4];
#pragma unroll
        for (int q = 0; q < 4; q++) o[q] = (unsigned)(j * p.pitch + s.c[q]);
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const int q = cz_of(i) > 0 ? 0 : (cz_of(i) < 0 ? 2 : 1);
            if (PAIR && q == 1) {
                const float2* a = reinterpret_cast<const float2*>(s.base[i] + o[1]);
                fi[i] = LAST ? __ldcs(a) : *a;
            } else {
                fi[i] = pk(ld(s.base[i] + o[q]), ld(s.base[i] + o[q + 1]));
            }
        }
    } else {
        const PullRow r = pull_row(p, j);
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const int q = (i == 6 || i == 7) && r.stay ? 1 : (cz_of(i) > 0 ? 0 : (cz_of(i) < 0 ? 2 : 1));
            const float* b = f + r.o[i];
            fi[i] = q == 0 ? pk(ld(b + s.c[0]), ld(b + s.c[1]))
                           : (q == 1 ? pk(ld(b + s.c[1]), ld(b + s.c[2])) : pk(ld(b + s.c[2]), ld(b + s.c[3])));
        }
    }
}

// First moments of the Kupershtokh force at a row from its own pair's rows m, z, q (r-1, r, r+1), their
// difference dd = q - m and the neighbours' (kup_moments2).
__device__ __forceinline__ void lane_kup(float2 m, float2 z, float2 q, float2 dd, float dl, float dr, float2& sz,
                                         float2& sr) {
    const float2 c9 = pk(1.0f / 9.0f, 1.0f / 9.0f), c36 = pk(1.0f / 36.0f, 1.0f / 36.0f);
    const float2 v = pfma(z, c9, pmul(padd(q, m), c36));
    sz = pk(v.y - from_left(v.y), from_right(v.x) - v.x);
    sr = pfma(dd, c9, pmul(pk(dl + dd.y, dd.x + dr), c36));
}

// The last N values of a lane's pair down its column, the newest last.
template <int N>
struct Column {
    float2 a[N];
    __device__ __forceinline__ void push(float2 v) {
#pragma unroll
        for (int q = 0; q + 1 < N; q++) a[q] = a[q + 1];
        a[N - 1] = v;
    }
    __device__ __forceinline__ float2 operator[](int q) const { return a[q]; }
};

template <bool MP, bool AX, int EOS, bool LATTICE>
__device__ __forceinline__ void march_warp(const Params<float>& pp, const float* __restrict__ f, float* __restrict__ fout,
                                           int strip, int j0, int jend, float2* __restrict__ ring, int& bad) {
    using T = float2;
    using S = WarpShape;
    Params<float> p = pp;  // with what the compiler is to know
    if (EOS >= 0) p.eos = EOS;
    if (LATTICE) p.kappa = KAPPA_LATTICE;
    const int lane = threadIdx.x & 31, nz = p.nz, nr = p.nr, plane = (int)p.plane;
    const int k = strip * S::TZ + 2 * (lane - S::kFirst);  // the lane's first column, not wrapped
    const bool periodic = p.top == TOP_PERIODIC, noslip = p.top == TOP_NOSLIP;
    const bool stores = lane >= S::kFirst && lane <= 31 - S::kFirst && k < nz;
    const bool v1 = k + 1 < nz;
    LaneSource src;
#pragma unroll
    for (int i = 0; i < 4; i++) src.c[i] = wrap_any(k - 1 + i, nz);
#pragma unroll
    for (int i = 0; i < Q; i++) src.base[i] = f + (i * plane - cr_of(i) * p.pitch);
    const T zero = pk(0.0f, 0.0f), ref = pk(p.rho_ref, p.rho_ref);
    const T la[3] = {zero, zero, zero};  // no link source in this form
    Column<6> psi = {};
    Column<4> fz = {}, fr = {};
    Column<5> uz = {}, ur = {};
    T lf[Q];
    lane_pull<false, false, false>(p, f, src, mirror_row(j0 - 6, nr, periodic), lf);
    auto rj = [&](int row) { return ring + (row & (S::kRing - 1)) * S::kRow + lane; };          // rho, j
    auto rp = [&](int row) { return ring + (row & (S::kRing - 1)) * S::kRow + (96 + lane); };  // psi_z, psi_r

    // The iteration that reads row l.  full: every stage runs on an interior row.
    auto turn = [&](int l, auto full, auto pairs) {
        constexpr bool kFull = decltype(full)::value, kPair = decltype(pairs)::value;
        T cf[Q];
        const bool doC = kFull || l >= j0 + 7;
        if (doC) lane_pull<kFull, kPair, true>(p, f, src, l - 7, cf);
        // ---- L, row l
        if (kFull || l < jend + 6) {
            T drho, jz, jr;
            moments2<false, float>(lf, la, drho, jz, jr);
            psi.push(psi2<MP>(p, drho, true, bad));
            T* o = rj(l);
            o[0] = drho;
            o[32] = jz;
            o[64] = !kFull && !periodic && l < 0 ? psub(zero, jr) : jr;
            if (kFull)
                lane_pull<true, kPair, false>(p, f, src, l + 1, lf);
            else if (l + 1 < jend + 6)
                lane_pull<false, false, false>(p, f, src, mirror_row(l + 1, nr, periodic), lf);
        } else {
            psi.push(zero);
        }

        // ---- D, row l - 2: psi rows l-4 .. l (1 .. 5); F_K pushed
        if (MP && (kFull || l >= j0 - 2)) {
            const int d = l - 2;
            T npz = zero, npr = zero;
            if (kFull || periodic || d < nr) {
                const T z0 = psi[3], zp = psi[4], zm = psi[2], d1 = psub(zp, zm);
                const float dl = from_left(d1.y), dr = from_right(d1.x);
                if (AX) {
                    const T z2p = psi[5], z2m = psi[1];
                    npz = lane_dz(padd(padd(z0, zp), zm), padd(padd(z0, z2p), z2m));
                    npr = lane_dr(d1, psub(z2p, z2m), dl, dr);
                }
                // Kupershtokh force (force_k2) on top of rho g
                T s1z, s1r, s2z, s2r;
                lane_kup(zm, z0, zp, d1, dl, dr, s1z, s1r);
                const T qm = pmul(zm, zm), q0 = pmul(z0, z0), qp = pmul(zp, zp), dq = psub(qp, qm);
                lane_kup(qm, q0, qp, dq, from_left(dq.y), from_right(dq.x), s2z, s2r);
                const T gz = pmul(padd(rj(d)[0], ref), pk(p.gz, p.gz));
                const float kB = 1.0f - 2.0f * p.A;
                const T bk = pmul(pk(6.0f * kB, 6.0f * kB), z0), a6k = pk(6.0f * p.A, 6.0f * p.A);
                fz.push(pfma(a6k, s2z, pfma(bk, s1z, gz)));
                fr.push(pfma(a6k, s2r, pfma(bk, s1r, zero)));
            } else {  // beyond the wall psi_z is even, psi_r odd: rows nr - 1, nr - 2
                if (AX) {
                    const T* m = rp(d == nr ? d - 1 : d - 3);
                    npz = m[0];
                    npr = psub(zero, m[32]);
                }
                fz.push(zero);
                fr.push(zero);
            }
            if (AX) rp(d)[0] = npz, rp(d)[32] = npr;
        }

        // ---- U, row l - 5: psi derivatives of rows l-7 .. l-3
        T nuz = zero, nur = zero;
        if (kFull || l >= j0 + 3) {
            const int u = l - 5;
            if (kFull || periodic || u < nr) {
                const T* o = rj(u);
                const T rho = padd(o[0], ref);
                T Fz = fz[0], Fr = fr[0];
                if (!MP) Fz = pmul(rho, pk(p.gz, p.gz)), Fr = zero;
                if (MP && AX) {
                    const T *q1 = rp(u - 2), *q2 = rp(u - 1), *q3 = rp(u), *q4 = rp(u + 1), *q5 = rp(u + 2);
                    const T r1 = psub(q4[32], q2[32]), z1 = psub(q4[0], q2[0]);
                    const T prr = lane_dr(r1, psub(q5[32], q1[32]), from_left(r1.y), from_right(r1.x));
                    const T prz = lane_dr(z1, psub(q5[0], q1[0]), from_left(z1.y), from_right(z1.x));
                    const int row = kFull ? u : (periodic ? mirror_row(u, nr, true) : u);
                    force_axis2(p, rho, psi[0], q3[0], q3[32], prr, prz, row, Fz, Fr);
                }
                velocity2<float>(rho, o[32], o[64], Fz, Fr, nuz, nur);
            } else {  // beyond the wall: rows nr - 1, nr - 2
                const T mz = u == nr ? uz[4] : uz[2], mr = u == nr ? ur[4] : ur[2];
                nuz = noslip ? psub(zero, mz) : mz;
                nur = psub(zero, mr);
            }
            uz.push(nuz);
            ur.push(nur);
        }

        // ---- C, row l - 7: u of rows l-9 .. l-5
        if (doC) {
            const int row = l - 7;
            const T* o = rj(row);
            const T drho = o[0], rho = padd(drho, ref);
            T Hz = zero, Hr = zero, mir = zero, rur = zero;
            const T cuz = uz[2], cur = ur[2], u1 = ur[0], u2 = ur[1], u4 = ur[3], v1_ = uz[0], v2_ = uz[1], v4_ = uz[3];
            if (AX) {
                const T z1 = psub(v4_, v2_), r1 = psub(u4, u2);
                const T duz_dr = lane_dr(z1, psub(nuz, v1_), from_left(z1.y), from_right(z1.x));
                const T dur_dz = lane_dz(padd(padd(cur, u4), u2), padd(padd(cur, nur), u1));
                const T dur_dr = lane_dr(r1, psub(nur, u1), from_left(r1.y), from_right(r1.x));
                source2(p, rho, cuz, cur, duz_dr, dur_dz, dur_dr, row, Hz, Hr, mir, rur);
            }
            float* out = fout + (row * p.pitch + k);
            collide2<0>(
                p, cf, la, drho, o[32], o[64], cuz, cur, Hz, Hr, mir, rur,
                [&](int q, T v) { cf[q] = v; }, [](int, T) {});
            if (stores && v1) {
#pragma unroll
                for (int q = 0; q < Q; q++) __stcs(reinterpret_cast<T*>(out + q * plane), cf[q]);
            } else if (stores) {
#pragma unroll
                for (int q = 0; q < Q; q++) __stcs(out + q * plane, cf[q].x);
            }
        }
    };

    // interior turns: every stage on, no row gathered at the axis or the top
    const int a = max(j0 + 7, 8), b = min(jend + 5, nr - 2);
    // pairs are aligned: an even nz, or no column of the strip wraps
    const bool pairs = (nz & 1) == 0 || (strip * S::TZ >= 8 && strip * S::TZ + 60 <= nz);
    int l = j0 - 6;
#pragma unroll 1
    while (l < jend + 7) {
        if (l >= a && l < b) {
            if (pairs) {
#pragma unroll 1
                for (; l < b; l++) turn(l, std::true_type(), std::true_type());
            } else {
#pragma unroll 1
                for (; l < b; l++) turn(l, std::true_type(), std::false_type());
            }
        } else {
            turn(l, std::false_type(), std::false_type());
            l++;
        }
    }
}

// What a kernel knows of its solves' parameters: the EOS and whether kappa is the lattice constant.
// With axis terms WARP_MIXED knows neither and asks in the loop, which costs 0 to 3 % (100 solves of 1.1M nodes
// 39.8 us per step with mixed EOS and 39.0 with one); a copy of the loop for each kind costs more as soon as their
// warps meet on an SM, whose instruction cache does not hold them: 76.6.  Without axis terms (a shorter loop) two
// copies are better: 256 solves of 6.3M nodes 157 us, 173 asking in the loop, 139 with one EOS.
enum WarpKind { WARP_CS = 0, WARP_CS_LATTICE = 1, WARP_VDW = 2, WARP_VDW_LATTICE = 3, WARP_MIXED = 4 };

// One tile of one solve.
template <bool MP, bool AX, int KIND>
__device__ __forceinline__ void march_tile(const BatchSolve<float>& s, const Tile& t, int parity, int* __restrict__ err) {
    __shared__ float2 ring[WarpShape::kRing * WarpShape::kRow];
    int bad = earlier_error(error_word(err), parity);
    const float* f = parity ? s.f_b : s.f_a;
    float* fo = parity ? const_cast<float*>(s.f_a) : s.f_b;
    if (bad) {
        // the solve already went unphysical: the step is left out, and so will the next one be
    } else if constexpr (KIND != WARP_MIXED) {
        march_warp<MP, AX, (KIND & 2) ? EOS_VDW : EOS_CS, (KIND & 1) != 0>(s.p, f, fo, t.strip, t.j0, t.jend, ring, bad);
    } else if constexpr (AX) {
        march_warp<MP, AX, -1, false>(s.p, f, fo, t.strip, t.j0, t.jend, ring, bad);
    } else if (s.p.eos == EOS_VDW) {
        march_warp<MP, AX, EOS_VDW, false>(s.p, f, fo, t.strip, t.j0, t.jend, ring, bad);
    } else {
        march_warp<MP, AX, EOS_CS, false>(s.p, f, fo, t.strip, t.j0, t.jend, ring, bad);
    }
    if (bad) atomicOr(err, err_of_step(bad, parity));
}

// Block b marches tile b.  The tile is the same for the whole warp: said by a
// shuffle, so that its rows stay uniform values.
__device__ __forceinline__ Tile warp_tile(const Tile* __restrict__ tiles) {
    const Tile t = tiles[blockIdx.x];
    return {__shfl_sync(0xffffffffu, t.solve, 0), __shfl_sync(0xffffffffu, t.strip, 0),
            __shfl_sync(0xffffffffu, t.j0, 0), __shfl_sync(0xffffffffu, t.jend, 0)};
}

template <bool MP, bool AX, int KIND>
__global__ void __launch_bounds__(32, WarpShape::kWarps)
    k_step_warp(const BatchSolve<float> s, const Tile* __restrict__ tiles, int parity, int* __restrict__ err) {
    march_tile<MP, AX, KIND>(s, warp_tile(tiles), parity, err);
}

// The tiles of any number of solves in one launch, their descriptors read from device memory once per tile
// (164 registers, as with a solve's own in the constant bank; a table of them as the launch's argument holds 256
// and takes 42.0 us on 256 solves of 1.1M nodes in all where this takes 41.3; 1200 solves of 2.9M nodes 109 us in
// one launch and 186 in five).
template <bool MP, bool AX, int KIND>
__global__ void __launch_bounds__(32, WarpShape::kWarps)
    k_step_warp_many(const BatchSolve<float>* __restrict__ solves, const Tile* __restrict__ tiles, int parity,
                     int* __restrict__ err) {
    const Tile t = warp_tile(tiles);
    const BatchSolve<float> s = solves[t.solve];
    march_tile<MP, AX, KIND>(s, t, parity, err + t.solve);
}

}  // namespace lbm
