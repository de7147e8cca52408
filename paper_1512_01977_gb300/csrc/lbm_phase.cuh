// One time step as three launches over tiles of nodes, without recomputed halos:
//
//   k_phase_l  gather, rho, j, psi            -> aux planes
//   k_phase_u  psi derivatives, force, u      -> u planes
//   k_phase_c  velocity gradients, H, collide -> the other population buffer
//
// The marching kernel (lbm_step.cuh) moves less memory but is a serial chain: a
// tile of 16 rows takes 17 iterations of all four stages whatever else the GPU
// has to do, and every tile recomputes 12 extra rows.  Here every node of a
// stage is independent, so a small grid fills the SMs and a step costs three
// short launches.  us per step, marching kernel -> phases (GB300): FP32 64 x 64
// 24.9 -> 6.1, 512 x 256 22.5 -> 9.4, 1023 x 511 (Guo) 32.4 -> 20.4; FP64 64 x 64
// 182 -> 16.3, 500 x 250 212 -> 70, 1024 x 512 495 -> 275.  (The smallest FP32
// grids are faster still in one launch, lbm_tile.cuh.)
//
// FP32 runs node pairs with the arithmetic of march2 (the update of a node pair
// in lbm_step.cuh), in the same order, so both give the same bits.  FP64 is
// bound by its arithmetic rate (1.9 DFMA lanes per clock and SM measured), so
// its kernels run one node per lane on the expressions with the fewest
// operations (34 + 116 + 104 FP64 instructions per node in the three phases,
// 437 in the marching kernel) and take reciprocals and roots from the hardware's
// FP64 approximations (rcp.approx.ftz.f64, rsqrt.approx.ftz.f64) and one
// correction each instead of a division.
#pragma once

#include "lbm_step.cuh"

namespace lbm {

// Columns of a tile (every kernel), rows by the launch.
template <typename R>
struct PhaseShape;
template <>
struct PhaseShape<float> {
    static constexpr int TZ = kPhaseColumns;  // a node pair per lane: one warp per tile row
};
template <>
struct PhaseShape<double> {
    static constexpr int TZ = 32;  // a node per lane
};

// The launches carry the programmatic attribute but no trigger: a trigger at the start lets the next
// kernel's waiting blocks fill whichever SMs have room, and it then runs unevenly (500 x 250 FP64: 97 us
// per step with it, 70 without; 512 x 256 FP32: 11.6 and 9.4).
__device__ __forceinline__ void phase_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// What a phase kernel works on: one solve (the tile by the block index) or the
// tiles of many (PhaseTile list, parameters from the device table).
template <typename R>
struct PhaseOne {
    BatchSolve<R> s;
    const R* h_src;  // link source planes (FV_LINK)
    R* h_dst;
    int parity;
    int across;  // tiles along z
    int* err;
    bool read = false;  // the gather of a field read: of the state as it is, failed or not
};
template <typename R>
struct PhaseMany {
    const BatchSolve<R>* s;
    const PhaseTile* tiles;
    int parity;
    int* err;
};

template <typename R>
struct PhaseWork {
    const R* f;
    R* fout;
    R* aux;
    R* u;  // u planes
    int* err;
    int k0, j0, parity;
};
template <typename R>
__device__ __forceinline__ PhaseWork<R> phase_work(const BatchSolve<R>& s, int parity, int* err, int k0, int j0) {
    return {parity ? s.f_b : s.f_a, parity ? const_cast<R*>(s.f_a) : s.f_b, s.aux, s.stage, err, k0, j0, parity};
}

// `word` below: the error word, read with a launch's other loads and looked at before its stores only.
// The gather passes an earlier error on as its own step's, so that the next step sees it too.

// u planes, in the staging planes of the moments pass (4 nz nr doubles, idle during a step): u_z, u_r
// (and 1 / rho in FP64), each of nr + 2 rows, the first two being rows -2 and -1 (beyond the axis:
// evaluated in place from mirrored rows, as the marching kernel does).  FP32 rows keep pairs aligned.
template <typename R>
__host__ __device__ inline int u_stride(int nz) {
    return sizeof(R) == 4 ? (nz + 1) & ~1 : nz;
}
template <typename R>
__host__ __device__ inline long long u_plane(int nz, int nr) {
    return (long long)u_stride<R>(nz) * (nr + 2);
}
constexpr int kGhostRows = 2;

// A row of psi within four rows of the grid: its mirror (even) or wrapped image.
__device__ __forceinline__ int mirror_row(int row, int nr, bool periodic) {
    while (row < 0 || row >= nr) {  // once unless nr is smaller than the halo (the field pass takes any nr)
        if (row < 0)
            row = periodic ? row + nr : -1 - row;
        else
            row = periodic ? row - nr : 2 * nr - 1 - row;
    }
    return row;
}

// The source planes and rows of the populations that arrive at row j (pull_slot for all nine): element
// offsets without the column, and whether the two diagonals from above arrive unshifted (no-slip).
struct PullRow {
    int o[Q];
    bool stay;
};
template <typename R>
__device__ __forceinline__ PullRow pull_row(const Params<R>& p, int j) {
    const int plane = (int)p.plane, pitch = p.pitch, r = j * pitch;
    const bool periodic = p.top == TOP_PERIODIC;
    const bool ax = j == 0 && !periodic, top = j + 1 == p.nr && !periodic, ns = top && p.top == TOP_NOSLIP;
    const int up = j > 0 ? r - pitch : (periodic ? (p.nr - 1) * pitch : 0);
    const int dn = j + 1 < p.nr ? r + pitch : (periodic ? 0 : r);
    PullRow q;
    q.o[0] = r;
    q.o[1] = plane + r;
    q.o[2] = 2 * plane + r;
    q.o[3] = (ax ? 4 : 3) * plane + up;
    q.o[5] = (ax ? 7 : 5) * plane + up;
    q.o[8] = (ax ? 6 : 8) * plane + up;
    q.o[4] = (top ? 3 : 4) * plane + dn;
    q.o[7] = (ns ? 8 : (top ? 5 : 7)) * plane + dn;
    q.o[6] = (ns ? 5 : (top ? 8 : 6)) * plane + dn;
    q.stay = ns;
    return q;
}

// The five rows of u that the gradients at row `row` read, as element offsets of u_z's plane; those
// beyond a top wall are mirror rows whose values change sign (`above`: how many of the last two).
struct URows {
    long long o[5];
    int above;
};
template <typename R>
__device__ __forceinline__ URows u_rows(const Params<R>& p, int row) {
    const bool periodic = p.top == TOP_PERIODIC;
    const int st = u_stride<R>(p.nz);
    URows u;
#pragma unroll
    for (int q = 0; q < 5; q++) {
        int r = row + q - 2;
        if (q > 2) r = mirror_row(r, p.nr, periodic);
        if (q < 2 && r < 0 && periodic) r += p.nr;
        u.o[q] = (long long)(r + kGhostRows) * st;
    }
    u.above = periodic ? 0 : max(0, row + 3 - p.nr);
    return u;
}

// ================================================================== FP32 ==

// Populations arriving at nodes (k, j) and (k+1, j).  EDGE: columns may wrap in z (else k >= 1 and
// k + 2 < nz); an odd row's last pair reads its second lane from the row's padding or a wrapped
// column, and that lane is not used.
template <bool EDGE, typename R, typename T>
__device__ __forceinline__ void pull2(const Params<R>& p, const R* __restrict__ f, int j, int k, T (&fi)[Q]) {
    const PullRow q = pull_row(p, j);
    const int km = EDGE && k == 0 ? p.nz - 1 : k - 1;
    const int kp = EDGE && k + 1 >= p.nz ? k + 1 - p.nz : k + 1;
    const int kq = EDGE ? wrap_any(k + 2, p.nz) : k + 2;
    fi[0] = ld2<T>(f + q.o[0], k);
    fi[3] = ld2<T>(f + q.o[3], k);
    fi[4] = ld2<T>(f + q.o[4], k);
    fi[1] = pk(f[q.o[1] + km], f[q.o[1] + k]);
    fi[5] = pk(f[q.o[5] + km], f[q.o[5] + k]);
    fi[2] = pk(f[q.o[2] + kp], f[q.o[2] + kq]);
    fi[8] = pk(f[q.o[8] + kp], f[q.o[8] + kq]);
    if (!q.stay) {
        fi[7] = pk(f[q.o[7] + km], f[q.o[7] + k]);
        fi[6] = pk(f[q.o[6] + kp], f[q.o[6] + kq]);
    } else {
        fi[7] = ld2<T>(f + q.o[7], k);
        fi[6] = ld2<T>(f + q.o[6], k);
    }
}

// The tile's columns and their neighbours need no wrap (the same for the whole CTA).
template <typename R>
__device__ __forceinline__ bool phase_inner(const Params<R>& p, int k0) {
    return k0 >= 4 && k0 + PhaseShape<R>::TZ + 4 <= p.nz;
}

template <bool MP, bool LINK, bool EDGE, typename R>
__device__ __forceinline__ void phase_l2(const Params<R>& p, const PhaseWork<R>& w, const R* h_src, int word) {
    using T = typename PairOf<R>::T;
    const int row = w.j0 + (threadIdx.x >> 5), k = w.k0 + 2 * (threadIdx.x & 31);
    if (row >= p.nr || k >= p.nz) return;
    T f[Q], la[3];
    pull2<EDGE>(p, w.f, row, k, f);
    if (LINK) link2<R>(p, h_src, row, k, !EDGE, la);
    T drho, jz, jr;
    int bad = 0;
    moments2<LINK, R>(f, la, drho, jz, jr);
    const T psi = psi2<MP>(p, drho, k + 1 < p.nz, bad);
    const int earlier = earlier_error(word, w.parity);
    bad |= earlier;
    if (bad) atomicOr(w.err, err_of_step(bad, w.parity));
    if (earlier) return;
    // the second lane of an odd row's last pair goes to the row's padding
    R* o = w.aux + (row * p.pitch + k);
    const int plane = (int)p.plane;
    st2(o, 0, drho);
    st2(o + plane, 0, jz);
    st2(o + 2 * plane, 0, jr);
    if (MP) st2(o + 3 * plane, 0, psi);
}

// Tile plus 4 columns and rows of psi (F on the tile needs psi_rr, which needs psi_r on a 2-ring).
template <int TR>
struct PhaseU2 {
    static constexpr int TZ = PhaseShape<float>::TZ, WP = TZ + 8, WD = TZ + 4;
    static constexpr int elems = WP * (TR + 8) + 2 * WD * (TR + 4);
};

template <int TR, bool MP, bool AX, bool EDGE, typename R>
__device__ __forceinline__ void phase_u2(const Params<R>& p, const PhaseWork<R>& w, R* smem, int word) {
    using T = typename PairOf<R>::T;
    using S = PhaseU2<TR>;
    constexpr int TZ = S::TZ, WP = S::WP, WD = S::WD, NT = 32 * TR;
    R* sPsi = smem;
    R* sPz = sPsi + WP * (TR + 8);
    R* sPr = sPz + WD * (TR + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nz = p.nz, nr = p.nr, k0 = w.k0;
    const int plane = (int)p.plane;
    const bool periodic = p.top == TOP_PERIODIC;
    // rows [j0, jb): a tile that begins beyond the axis holds the ghost rows only
    const int j0 = w.j0, jb = j0 < 0 ? 0 : min(j0 + TR, nr);
    const int kn = EDGE ? min(TZ, nz - k0) : TZ, c = 2 * lane, row = j0 + warp;
    const bool mine = row < jb && c < kn;
    T drho = pk(R(0), R(0)), jz = drho, jr = drho;
    if (mine) {
        const R* a = w.aux + ((row < 0 ? -1 - row : row) * p.pitch + k0 + c);
        drho = ld2<T>(a, 0);
        jz = ld2<T>(a + plane, 0);
        jr = ld2<T>(a + 2 * plane, 0);
    }
    if (MP) {
        const R* psi = w.aux + 3 * plane;
        // lane's pairs of a row: columns c and, for the first four lanes, TZ + c (from k0 - 4)
        int ka = k0 - 4 + c, kb = k0 - 4 + TZ + c, ka1 = ka + 1, kb1 = kb + 1;
        if (EDGE) ka = wrap_any(ka, nz), ka1 = wrap_any(ka1, nz), kb = wrap_any(kb, nz), kb1 = wrap_any(kb1, nz);
#pragma unroll
        for (int q = 0; q < (TR + 8 + TR - 1) / TR; q++) {
            const int a = warp + q * TR;
            if (a < jb - j0 + 8) {
                const R* m = psi + mirror_row(j0 - 4 + a, nr, periodic) * p.pitch;
                st2(sPsi + a * WP, c, EDGE ? pk(m[ka], m[ka1]) : ld2<T>(m, ka));
                if (lane < 4) st2(sPsi + a * WP, TZ + c, EDGE ? pk(m[kb], m[kb1]) : ld2<T>(m, kb));
            }
        }
        __syncthreads();
    }
    if (MP && AX) {
        constexpr int HD = WD / 2;
        for (int i = tid; i < (jb - j0 + 4) * HD; i += NT) {
            const int a = i / HD, b = 2 * (i - a * HD);
            int er = j0 - 2 + a;
            const bool above = !periodic && er >= nr;
            if (above) er = 2 * nr - 1 - er;
            const R* m = sPsi + (er - j0 + 4) * WP;
            T dz, dr;
            fd_both2<R>(m - 2 * WP, m - WP, m, m + WP, m + 2 * WP, b + 2, dz, dr);
            st2(sPz + a * WD, b, dz);
            st2(sPr + a * WD, b, above ? psub(pk(R(0), R(0)), dr) : dr);
        }
        __syncthreads();
    }
    if (!mine || earlier_error(word, w.parity)) return;
    if (row < 0) jr = psub(pk(R(0), R(0)), jr);
    const T rho = padd(drho, pk(p.rho_ref, p.rho_ref));
    T fz = pmul(rho, pk(p.gz, p.gz)), fr = pk(R(0), R(0));
    if (MP) {
        const R* m = sPsi + (warp + 4) * WP;
        const Tri<T> z0 = ld3<T>(m, c + 4), zm = ld3<T>(m - WP, c + 4), zq = ld3<T>(m + WP, c + 4);
        force_k2(p, zm, z0, zq, fz, fr);
        if (AX) {
            const R* a = sPr + (warp + 2) * WD;
            const R* b = sPz + (warp + 2) * WD;
            const T prr = fd_r2<R, T>(a - 2 * WD, a - WD, a + WD, a + 2 * WD, c + 2);
            const T prz = fd_r2<R, T>(b - 2 * WD, b - WD, b + WD, b + 2 * WD, c + 2);
            force_axis2(p, rho, z0.b, ld2<T>(b, c + 2), ld2<T>(a, c + 2), prr, prz, row, fz, fr);
        }
    }
    T vz, vr;
    velocity2<R>(rho, jz, jr, fz, fr, vz, vr);
    R* o = w.u + ((long long)(row + kGhostRows) * u_stride<R>(nz) + k0 + c);
    st2(o, 0, vz);
    st2(o + u_plane<R>(nz, nr), 0, vr);
}

template <bool AX, int FV, bool EDGE, typename R>
__device__ __forceinline__ void phase_c2(const Params<R>& p, const PhaseWork<R>& w, const R* h_src, R* h_dst,
                                         int word) {
    using T = typename PairOf<R>::T;
    constexpr bool link = (FV & FV_LINK) != 0;
    const int row = w.j0 + (threadIdx.x >> 5), k = w.k0 + 2 * (threadIdx.x & 31);
    if (row >= p.nr || k >= p.nz) return;
    const int nz = p.nz;
    T f[Q], la[3], drho, jz, jr;
    pull2<EDGE>(p, w.f, row, k, f);
    if (link) link2<R>(p, h_src, row, k, !EDGE, la);
    T uz, ur, Hz = pk(R(0), R(0)), Hr = Hz, mir = Hz, rur = Hz;
    T duz_dr = Hz, dur_dz = Hz, dur_dr = Hz;
    const R* Ur = w.u + u_plane<R>(nz, p.nr);
    if (AX) {
        const URows ru = u_rows(p, row);
        int ka = k - 2, ka1 = k - 1, kc = k + 2, kc1 = k + 3;
        if (EDGE) ka = wrap_any(ka, nz), ka1 = wrap_any(ka1, nz), kc = wrap_any(kc, nz), kc1 = wrap_any(kc1, nz);
        // an odd row's last pair: column k + 1 wraps too
        const int kb1 = EDGE && k + 1 >= nz ? k + 1 - nz : k + 1;
        auto tri = [&](const R* m) -> Tri<T> {
            if (EDGE) return {pk(m[ka], m[ka1]), pk(m[k], m[kb1]), pk(m[kc], m[kc1])};
            return {ld2<T>(m, ka), ld2<T>(m, k), ld2<T>(m, kc)};
        };
        Tri<T> z[5], r[5];
#pragma unroll
        for (int q = 0; q < 5; q++) {
            r[q] = tri(Ur + ru.o[q]);
            if (q != 2) z[q] = tri(w.u + ru.o[q]);
        }
        uz = ld2<T>(w.u + ru.o[2], k);
        ur = r[2].b;
        if (ru.above > 0) {  // u_r is odd beyond the wall, u_z too beyond a no-slip one
            auto flip = [](Tri<T>& t) {
                const T o = pk(R(0), R(0));
                t = {psub(o, t.a), psub(o, t.b), psub(o, t.c)};
            };
            flip(r[4]);
            if (ru.above > 1) flip(r[3]);
            if (p.top == TOP_NOSLIP) {
                flip(z[4]);
                if (ru.above > 1) flip(z[3]);
            }
        }
        duz_dr = fd_r3<R, T>(z[0], z[1], z[3], z[4]);
        fd_both3<R>(r[0], r[1], r[2], r[3], r[4], dur_dz, dur_dr);
    } else {
        const long long o = (long long)(row + kGhostRows) * u_stride<R>(nz) + k;
        uz = ld2<T>(w.u + o, 0);
        ur = ld2<T>(Ur + o, 0);
    }
    moments2<link, R>(f, la, drho, jz, jr);
    if (AX) source2(p, padd(drho, pk(p.rho_ref, p.rho_ref)), uz, ur, duz_dr, dur_dz, dur_dr, row, Hz, Hr, mir, rur);
    if (earlier_error(word, w.parity)) return;
    const int plane = (int)p.plane;
    R* o = w.fout + (row * p.pitch + k);
    R* hq = link ? h_dst + (row * p.pitch + k) : nullptr;
    auto put = [&](R* q, T v) {
        if (!EDGE || k + 1 < nz)
            st2(q, 0, v);
        else
            *q = v.x;
    };
    collide2<FV>(
        p, f, la, drho, jz, jr, uz, ur, Hz, Hr, mir, rur, [&](int i, T v) { put(o + i * plane, v); },
        [&](int q, T v) { put(hq + q * plane, v); });
}

// ================================================================== FP64 ==

// A product that stays one: where it is added to something the compiler may or
// may not fuse the two, differently in the kernels for one solve and for many,
// whose results have to be the same.
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }

// 1/x: the hardware's approximation y (relative error e below 2^-19.9) and one
// third-order step, y (1 + e + e^2) with e = 1 - x y: within 1 ulp of the
// quotient, 3 operations where a division takes the time of 17.  Zeros, subnormal values and results, infinities
// and NaN are left to the division.
__device__ __forceinline__ double rcp3(double x) {
    // by the bits: |x| in [2^-1022, 2^1020)
    if ((unsigned)(__double2hiint(x) & 0x7fffffff) - 0x00100000u >= 0x7fa00000u) return 1.0 / x;
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
// sqrt(x), 0 for x <= 0: with y the approximate inverse root and s = x y, the root is s + r / (2 s) (1 - r /
// (4 s^2)) for the remainder r = x - s^2, and with e = 1 - s y that is s + r (y/2) (1 + 3 e/4), 6 operations:
// correctly rounded but for 6 roots in 10,000.  (The series of (1 - e)^(-1/2) alone, 5 operations, keeps half of
// the rounding of s: a unit off in one root of eight.)  Zeros, negative,
// tiny and non-finite values are told by the bits (an FP64 comparison costs as much as two operations).
__device__ __forceinline__ double sqrt3(double x) {
    const int hi = __double2hiint(x);
    // below 2^-959 the remainder would lose digits
    if ((unsigned)hi - 0x04000000u >= 0x7ff00000u - 0x04000000u) return x > 0.0 ? sqrt(x) : 0.0;
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double s = x * y, e = fma(-s, y, 1.0), r = fma(-s, s, x);
    const double half_y = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));
    return fma(r * half_y, fma(0.75, e, 1.0), s);
}
// x > 0 and x >= 0 (NaN: false), by the bits.
__device__ __forceinline__ bool positive(double x) {
    return (unsigned long long)__double_as_longlong(x) - 1ull < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool nonnegative(double x) { return positive(x) || x == 0.0; }

__device__ __forceinline__ double eos_p3(const Params<double>& p, double rho) {
    if (p.eos == EOS_VDW) return p.lambda * rho * fma(8.0 * p.T, rcp3(3.0 - rho), -3.0 * rho);
    const double e = mul(p.b * 0.25, rho), om = 1.0 - e;
    const double num = fma(e, fma(e, om, 1.0), 1.0);
    return rho * fma(p.Rg * p.T * num, rcp3(om * om * om), -p.a * rho);
}
__device__ __forceinline__ double kappa3(const Params<double>& p, double rho) {  // 3 kappa
    if (p.kappa == KAPPA_LATTICE) return 1.0 / 3.0;
    double c2;
    if (p.eos == EOS_VDW) {
        const double d = 3.0 - rho;
        c2 = p.lambda * fma(24.0 * p.T, rcp3(d * d), -6.0 * rho);
    } else {
        const double e = mul(p.b * 0.25, rho), om = 1.0 - e, om2 = mul(om, om);
        const double num = fma(e, fma(e, fma(e, e - 4.0, 4.0), 4.0), 1.0);
        c2 = fma(p.Rg * p.T * num, rcp3(om2 * om2), -2.0 * p.a * rho);
    }
    return p.kappa == KAPPA_MIXED ? c2 : 3.0 * c2 * c2;
}

// Populations arriving at node (k, j).
__device__ __forceinline__ void pull1(const Params<double>& p, const double* __restrict__ f, int j, int k,
                                      double (&fi)[Q]) {
    const PullRow q = pull_row(p, j);
    const int km = k == 0 ? p.nz - 1 : k - 1, kp = k + 1 == p.nz ? 0 : k + 1;
    fi[0] = f[q.o[0] + k];
    fi[3] = f[q.o[3] + k];
    fi[4] = f[q.o[4] + k];
    fi[1] = f[q.o[1] + km];
    fi[5] = f[q.o[5] + km];
    fi[2] = f[q.o[2] + kp];
    fi[8] = f[q.o[8] + kp];
    fi[7] = f[q.o[7] + (q.stay ? k : km)];
    fi[6] = f[q.o[6] + (q.stay ? k : kp)];
}

__device__ __forceinline__ void moments1(const double (&f)[Q], double& drho, double& jz, double& jr) {
    const double x = f[5] - f[6], y = f[7] - f[8];
    jz = (f[1] - f[2]) + (x + y);
    jr = (f[3] - f[4]) + (x - y);
    drho = (f[0] + ((f[1] + f[2]) + (f[3] + f[4]))) + ((f[5] + f[6]) + (f[7] + f[8]));
}
__device__ __forceinline__ bool finite1(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

template <bool MP, bool LINK>
__device__ __forceinline__ void phase_l1(const Params<double>& p, const PhaseWork<double>& w, const double* h_src,
                                         int word) {
    const int row = w.j0 + (threadIdx.x >> 5), k = w.k0 + (threadIdx.x & 31);
    if (row >= p.nr || k >= p.nz) return;
    double f[Q];
    pull1(p, w.f, row, k, f);
    double drho, jz, jr;
    moments1(f, drho, jz, jr);
    if (LINK) {
        double a[3];
        link3(p, h_src, row, k, a);
        drho = fma(0.5, a[0], drho);
        jz = fma(0.5, a[1], jz);
        jr = fma(0.5, a[2], jr);
    }
    const double rho = p.rho_ref + drho;
    int bad = (positive(rho) ? 0 : ERRBIT_RHO) | (finite1(jz) && finite1(jr) ? 0 : ERRBIT_NONFINITE);
    double psi = 0.0;
    if (MP) {
        const double arg = fma(rho, 1.0 / 3.0, -eos_p3(p, rho));
        if (!nonnegative(arg)) bad |= ERRBIT_PSI;
        psi = sqrt3(arg);
    }
    const int earlier = earlier_error(word, w.parity);
    bad |= earlier;
    if (bad) atomicOr(w.err, err_of_step(bad, w.parity));
    if (earlier) return;
    const int plane = (int)p.plane;
    double* o = w.aux + (row * p.pitch + k);
    o[0] = drho;
    o[plane] = jz;
    o[2 * plane] = jr;
    if (MP) o[3 * plane] = psi;
}

// psi with 4 columns and rows around the tile, the column sums of its stencils, and psi_z, psi_r with 2.
template <int TR>
struct PhaseU1 {
    static constexpr int TZ = PhaseShape<double>::TZ, WP = TZ + 8, WD = TZ + 4;
    static constexpr int elems = WP * (TR + 8) + 4 * WP * (TR + 4) + 2 * WD * (TR + 4);
};

// put(row, k, drho, u_z, u_r, 1/rho) takes the results.
template <int TR, bool MP, bool AX, typename P>
__device__ __forceinline__ void phase_u1(const Params<double>& p, const PhaseWork<double>& w, double* smem,
                                         int word, P&& put) {
    using S = PhaseU1<TR>;
    constexpr int TZ = S::TZ, WP = S::WP, WD = S::WD, NT = 32 * TR, NC = WP * (TR + 4);
    double* sPsi = smem;
    double* sS1 = sPsi + WP * (TR + 8);  // sums over rows r-1..r+1, of r-2, r, r+2; differences of r+-1, r+-2
    double* sPz = sS1 + 4 * NC;
    double* sPr = sPz + WD * (TR + 4);
    const int tid = threadIdx.x, warp = tid >> 5, c = tid & 31, nz = p.nz, nr = p.nr, k0 = w.k0;
    const int plane = (int)p.plane;
    const bool periodic = p.top == TOP_PERIODIC;
    const int j0 = w.j0, jb = j0 < 0 ? 0 : min(j0 + TR, nr), row = j0 + warp;
    const bool mine = row < jb && c < nz - k0;
    double drho = 0.0, jz = 0.0, jr = 0.0;
    if (mine) {
        const double* a = w.aux + ((row < 0 ? -1 - row : row) * p.pitch + k0 + c);
        drho = a[0];
        jz = a[plane];
        jr = a[2 * plane];
    }
    if (MP) {
        const double* psi = w.aux + 3 * plane;
        const int ka = wrap_any(k0 - 4 + c, nz), kb = wrap_any(k0 + TZ - 4 + c, nz);
#pragma unroll
        for (int q = 0; q < (TR + 8 + TR - 1) / TR; q++) {
            const int a = warp + q * TR;
            if (a < jb - j0 + 8) {
                const double* m = psi + mirror_row(j0 - 4 + a, nr, periodic) * p.pitch;
                sPsi[a * WP + c] = m[ka];
                if (c < 8) sPsi[a * WP + TZ + c] = m[kb];
            }
        }
        __syncthreads();
        if (AX) {
            for (int i = tid; i < (jb - j0 + 4) * WP; i += NT) {
                const int a = i / WP, b = i - a * WP;
                int er = j0 - 2 + a;
                if (!periodic && er >= nr) er = 2 * nr - 1 - er;
                const double* m = sPsi + (er - j0 + 4) * WP + b;
                const double z0 = m[0], zp = m[WP], zm = m[-WP], z2p = m[2 * WP], z2m = m[-2 * WP];
                sS1[i] = z0 + (zp + zm);
                sS1[NC + i] = z0 + (z2p + z2m);
                sS1[2 * NC + i] = zp - zm;
                sS1[3 * NC + i] = z2p - z2m;
            }
            __syncthreads();
            for (int i = tid; i < (jb - j0 + 4) * WD; i += NT) {
                const int a = i / WD, b = i - a * WD;
                const double* s1 = sS1 + a * WP + b + 2;
                const double* s2 = s1 + NC;
                const double* d1 = s2 + NC;
                const double* d2 = d1 + NC;
                const double n1r = d1[0] + (d1[-1] + d1[1]), n2r = d2[0] + (d2[-2] + d2[2]);
                const double dr = fma(n1r, 8.0 / 36.0, mul(n2r, -1.0 / 36.0));
                sPz[i] = fma(s1[1] - s1[-1], 8.0 / 36.0, mul(s2[2] - s2[-2], -1.0 / 36.0));
                sPr[i] = (!periodic && j0 - 2 + a >= nr) ? -dr : dr;  // psi_r is odd beyond the wall
            }
            __syncthreads();
        }
    }
    if (!mine || earlier_error(word, w.parity)) return;
    const double rho = p.rho_ref + drho;
    double fz = mul(rho, p.gz), fr = 0.0;
    if (MP) {
        // F_K with w(e) e^2 - w(w) w^2 = w (e - w)(e + w) for each opposite pair:
        // F = 6 sum over pairs of w c (d) [A (s) + (1 - 2A) psi], d and s its difference and sum
        const double* m = sPsi + (warp + 4) * WP + c + 4;
        const double bk = mul(1.0 - 2.0 * p.A, m[0]), A = p.A;
        const double e = m[1], wv = m[-1], n = m[WP], so = m[-WP];
        const double ne = m[WP + 1], nw = m[WP - 1], se = m[-WP + 1], sw = m[-WP - 1];
        const double gx = mul(ne - sw, fma(A, ne + sw, bk)), gy = mul(nw - se, fma(A, nw + se, bk));
        const double ge = mul(e - wv, fma(A, e + wv, bk)), gn = mul(n - so, fma(A, n + so, bk));
        fz = fma(1.0 / 6.0, fma(4.0, ge, gx - gy), fz);
        fr = mul(1.0 / 6.0, fma(4.0, gn, gx + gy));
        if (AX) {
            // F_axis; beyond the axis psi_r and 1/r are both odd, as the rows' own values have it
            const double* z = sPz + (warp + 2) * WD + c + 2;
            const double* r = sPr + (warp + 2) * WD + c + 2;
            const double prr = fd_r_rows(r - 2 * WD, r - WD, r + WD, r + 2 * WD, 0);
            const double prz = fd_r_rows(z - 2 * WD, z - WD, z + WD, z + 2 * WD, 0);
            const double ir = rcp3(row + 0.5), k3 = kappa3(p, rho), psr = r[0];
            const double a6 = mul(mul(mul(p.axis_a, A), ir), psr), pir = mul(m[0], ir);
            fz = fma(k3, fma(pir, prz, mul(a6, z[0])), fz);
            fr = fma(k3, fma(pir, fma(-psr, ir, prr), mul(a6, psr)), fr);
        }
    }
    const double irho = rcp3(rho);
    put(row, k0 + c, drho, mul(fma(0.5, fz, jz), irho), mul(fma(0.5, fr, row < 0 ? -jr : jr), irho), irho);
}

template <bool AX, int FV>
__device__ __forceinline__ void phase_c1(const Params<double>& p, const PhaseWork<double>& w, const double* h_src,
                                         double* h_dst, int word) {
    constexpr bool link = (FV & FV_LINK) != 0, guo = (FV & FV_GUO) != 0;
    const int row = w.j0 + (threadIdx.x >> 5), k = w.k0 + (threadIdx.x & 31), nz = p.nz;
    if (row >= p.nr || k >= nz) return;
    double f[Q];
    pull1(p, w.f, row, k, f);
    const long long n = u_plane<double>(nz, p.nr);
    const double* a = w.aux + (row * p.pitch + k);
    const double drho = a[0], jz = a[p.plane], jr = a[2 * p.plane];
    const double* u = w.u + (long long)(row + kGhostRows) * u_stride<double>(nz);
    const double uz = u[k], ur = u[n + k], irho = u[2 * n + k];
    const double rho = p.rho_ref + drho;
    double Hz = 0.0, Hr = 0.0, m0 = 0.0;
    if (AX) {
        const URows ru = u_rows(p, row);
        const int km = k == 0 ? nz - 1 : k - 1, kp = k + 1 == nz ? 0 : k + 1;
        const int km2 = wrap_any(k - 2, nz), kp2 = wrap_any(k + 2, nz);
        // rows beyond the wall: the mirror row's values with the sign changed (by the bits, no arithmetic)
        const bool n1 = ru.above > 1, n2 = ru.above > 0, ns = p.top == TOP_NOSLIP;
        auto sgn = [](bool neg, double v) {
            return neg ? __hiloint2double(__double2hiint(v) ^ 0x80000000, __double2loint(v)) : v;
        };
        double duz_dr;
        {
            const double *m2 = w.u + ru.o[0], *m1 = w.u + ru.o[1], *p1 = w.u + ru.o[3], *p2 = w.u + ru.o[4];
            const bool s1 = n1 && ns, s2 = n2 && ns;
            const double a1 = (sgn(s1, p1[k]) - m1[k]) + ((sgn(s1, p1[km]) - m1[km]) + (sgn(s1, p1[kp]) - m1[kp]));
            const double a2 =
                (sgn(s2, p2[k]) - m2[k]) + ((sgn(s2, p2[km2]) - m2[km2]) + (sgn(s2, p2[kp2]) - m2[kp2]));
            duz_dr = fma(a1, 8.0 / 36.0, mul(a2, -1.0 / 36.0));
        }
        // u_r: with x = ne - sw, y = nw - se the z sum is (e - w) + (x - y), the r sum (n - s) + (x + y)
        const double *m2 = w.u + n + ru.o[0], *m1 = w.u + n + ru.o[1], *z0 = w.u + n + ru.o[2];
        const double *p1 = w.u + n + ru.o[3], *p2 = w.u + n + ru.o[4];
        double x = sgn(n1, p1[kp]) - m1[km], y = sgn(n1, p1[km]) - m1[kp];
        const double n1z = (z0[kp] - z0[km]) + (x - y);
        const double n1r = (sgn(n1, p1[k]) - m1[k]) + (x + y);
        x = sgn(n2, p2[kp2]) - m2[km2], y = sgn(n2, p2[km2]) - m2[kp2];
        const double n2z = (z0[kp2] - z0[km2]) + (x - y);
        const double n2r = (sgn(n2, p2[k]) - m2[k]) + (x + y);
        const double dur_dz = fma(n1z, 8.0 / 36.0, mul(n2z, -1.0 / 36.0));
        const double dur_dr = fma(n1r, 8.0 / 36.0, mul(n2r, -1.0 / 36.0));
        const double ir = rcp3(row + 0.5), mu = mul(rho, p.nu), rur = mul(rho, ur);
        Hz = mul(fma(mu, duz_dr + dur_dz, -mul(rur, uz)), ir);
        Hr = mul(fma(2.0 * mu, fma(p.hr_sign * ir, ur, dur_dr), -mul(rur, ur)), ir);
        m0 = mul(-rur, ir);
    }
    if (earlier_error(word, w.parity)) return;
    const double om = p.tau_inv, om1 = 1.0 - p.tau_inv;
    const int plane = (int)p.plane;
    double* o = w.fout + (row * p.pitch + k);
    if (link) {
        double la[3];
        link3(p, h_src, row, k, la);
#pragma unroll
        for (int i = 0; i < Q; i++)
            f[i] = fma(0.5 * w_of<double>(i), fma(3.0, cz_of(i) * la[1] + cr_of(i) * la[2], la[0]), f[i]);
        double* h = h_dst + (row * p.pitch + k);
        h[0] = m0;
        h[plane] = Hz;
        h[2 * plane] = Hr;
        Hz *= 0.5;
        Hr *= 0.5;
        m0 *= 0.5;
    }
    // f*_i = (1 - omega) f_i + w_i (base + 4.5 c c : S) + 3 w_i c . M, the even part shared by opposite
    // directions: S = rho (u1 u1 - (1 - omega) u0 u0) or Guo's tensor, base its trace part with the
    // density and m0, M the odd part with H.
    const double u0z = mul(jz, irho), u0r = mul(jr, irho);
    double Szz, Srr, Szr, Mz, Mr, base;
    if (guo) {
        // omega rho u u + (1 - omega/2) (u F + F u), F = 2 rho (u - u0)
        const double g = 1.0 - 0.5 * om, Fz = 2.0 * rho * (uz - u0z), Fr = 2.0 * rho * (ur - u0r);
        const double mz = mul(om * rho, uz), mr = mul(om * rho, ur), gz = mul(g, Fz), gr = mul(g, Fr);
        Szz = fma(mz, uz, 2.0 * gz * uz);
        Srr = fma(mr, ur, 2.0 * gr * ur);
        Szr = fma(mz, ur, fma(gz, ur, gr * uz));
        Mz = mz + (gz + Hz);
        Mr = mr + (gr + Hr);
    } else {
        const double u1z = fma(2.0, uz, -u0z), u1r = fma(2.0, ur, -u0r);  // u0 + F / rho
        const double az = mul(om1, u0z), ar = mul(om1, u0r);
        Szz = mul(rho, fma(u1z, u1z, -az * u0z));
        Srr = mul(rho, fma(u1r, u1r, -ar * u0r));
        Szr = mul(rho, fma(u1z, u1r, -az * u0r));
        Mz = fma(rho, u1z - az, Hz);
        Mr = fma(rho, u1r - ar, Hr);
    }
    const double tr = Szz + Srr;
    base = fma(-1.5, tr, fma(om, drho, m0));
    o[0] = fma(om1, f[0], 4.0 / 9.0 * base);
    auto pair = [&](int i, double even, double w3, double M) {  // even, and 3 w_i times c_i . M
        o[i * plane] = fma(om1, f[i], fma(w3, M, even));
        o[(i + 1) * plane] = fma(om1, f[i + 1], fma(-w3, M, even));
    };
    pair(1, mul(1.0 / 9.0, fma(4.5, Szz, base)), 1.0 / 3.0, Mz);
    pair(3, mul(1.0 / 9.0, fma(4.5, Srr, base)), 1.0 / 3.0, Mr);
    const double diag = fma(4.5, tr, base);
    pair(5, mul(1.0 / 36.0, fma(9.0, Szr, diag)), 1.0 / 12.0, Mz + Mr);
    pair(7, mul(1.0 / 36.0, fma(-9.0, Szr, diag)), 1.0 / 12.0, Mz - Mr);
}

// =============================================================== kernels ==

template <typename R, bool MP, bool LINK>
__device__ __forceinline__ void phase_l(const Params<R>& p, const PhaseWork<R>& w, const R* h, bool read = false) {
    const int word = read ? 0 : error_word(w.err);
    if constexpr (sizeof(R) == 4) {
        if (phase_inner(p, w.k0))
            phase_l2<MP, LINK, false>(p, w, h, word);
        else
            phase_l2<MP, LINK, true>(p, w, h, word);
    } else {
        phase_l1<MP, LINK>(p, w, h, word);
    }
}
template <typename R, int TR, bool MP, bool AX>
__device__ __forceinline__ void phase_u(const Params<R>& p, const PhaseWork<R>& w) {
    const int word = error_word(w.err);
    if constexpr (sizeof(R) == 4) {
        __shared__ __align__(16) R smem[PhaseU2<TR>::elems];
        if (phase_inner(p, w.k0))
            phase_u2<TR, MP, AX, false>(p, w, smem, word);
        else
            phase_u2<TR, MP, AX, true>(p, w, smem, word);
    } else {
        __shared__ __align__(16) R smem[PhaseU1<TR>::elems];
        const long long n = u_plane<double>(p.nz, p.nr);
        phase_u1<TR, MP, AX>(p, w, smem, word, [&](int row, int k, double, double uz, double ur, double irho) {
            double* o = w.u + ((long long)(row + kGhostRows) * u_stride<double>(p.nz) + k);
            o[0] = uz;
            o[n] = ur;
            o[2 * n] = irho;
        });
    }
}
template <typename R, bool AX, int FV>
__device__ __forceinline__ void phase_c(const Params<R>& p, const PhaseWork<R>& w, const R* hs, R* hd) {
    const int word = error_word(w.err);
    if constexpr (sizeof(R) == 4) {
        if (phase_inner(p, w.k0))
            phase_c2<AX, FV, false>(p, w, hs, hd, word);
        else
            phase_c2<AX, FV, true>(p, w, hs, hd, word);
    } else {
        phase_c1<AX, FV>(p, w, hs, hd, word);
    }
}

// Tile of a block: by its index (the row beyond the last holds the ghost rows, k_phase_u's only), or
// from the list, which ends with the ghost rows' tiles.
#define LBM_PHASE_ONE(a)                                                                                     \
    const Params<R>& p = a.s.p;                                                                              \
    const int ti = blockIdx.x / a.across, tk = blockIdx.x - ti * a.across;                                   \
    phase_wait();                                                                                            \
    const PhaseWork<R> w = phase_work(a.s, a.parity, a.err, tk * PhaseShape<R>::TZ,                          \
                                      ti * TR < p.nr ? ti * TR : -kGhostRows)
#define LBM_PHASE_MANY(a)                                                                                    \
    const PhaseTile tl = a.tiles[blockIdx.x];                                                                \
    const Params<R> p = a.s[tl.solve].p;                                                                     \
    phase_wait();                                                                                            \
    const PhaseWork<R> w = phase_work(a.s[tl.solve], a.parity, a.err + tl.solve, tl.k0, tl.j0)

template <typename R, int TR, bool MP, bool LINK>
__global__ void __launch_bounds__(32 * TR) k_phase_l(const PhaseOne<R> a) {
    LBM_PHASE_ONE(a);
    phase_l<R, MP, LINK>(p, w, a.h_src, a.read);
}
template <typename R, int TR, bool MP, bool AX>
__global__ void __launch_bounds__(32 * TR) k_phase_u(const PhaseOne<R> a) {
    LBM_PHASE_ONE(a);
    phase_u<R, TR, MP, AX>(p, w);
}
template <typename R, int TR, bool AX, int FV>
__global__ void __launch_bounds__(32 * TR) k_phase_c(const PhaseOne<R> a) {
    LBM_PHASE_ONE(a);
    phase_c<R, AX, FV>(p, w, a.h_src, a.h_dst);
}
template <typename R, int TR, bool MP>
__global__ void __launch_bounds__(32 * TR) k_phase_l_many(const PhaseMany<R> a) {
    LBM_PHASE_MANY(a);
    phase_l<R, MP, false>(p, w, nullptr);
}
template <typename R, int TR, bool MP, bool AX>
__global__ void __launch_bounds__(32 * TR) k_phase_u_many(const PhaseMany<R> a) {
    LBM_PHASE_MANY(a);
    phase_u<R, TR, MP, AX>(p, w);
}
template <typename R, int TR, bool AX>
__global__ void __launch_bounds__(32 * TR) k_phase_c_many(const PhaseMany<R> a) {
    LBM_PHASE_MANY(a);
    phase_c<R, AX, 0>(p, w, nullptr, nullptr);
}
#undef LBM_PHASE_ONE
#undef LBM_PHASE_MANY

}  // namespace lbm
