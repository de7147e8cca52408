// Kernels of one time step of the axisymmetric multiphase D2Q9 update
// (arXiv:1512.01977), templated on the arithmetic type R (float or double).
//
// Storage (per solve, all planes with row pitch p.pitch, z contiguous):
//   f[2][9][nr][pitch]  populations, post-collision values of the previous
//                       step (pull streaming reads them shifted by -c_i);
//                       stored as deviations f_i - w_i rho_ref
//   aux[4][nr][pitch]   rho - rho_ref, j_z, j_r, psi of the current step
//
// One step of the two-kernel path = k_density (kernel a) + k_update (kernel b).
// The init pass uses the same maps; the passes that read a solve are in lbm_read.cuh.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

// ------------------------------------------------- kernel (a): rho, j, psi --
// rho - rho_ref, j_z, j_r of a node's arrived populations (Sec. II.A moments:
// rho = sum_i f_i, j = sum_i c_i f_i) and psi = sqrt(rho/3 - P_k(rho)) (Sec.
// II.C); returns error bits for rho <= 0, psi^2 < 0 and non-finite values.
template <typename R>
__device__ __forceinline__ int density_node(const Params<R>& p, const R (&f)[Q], const LinkPlanes<R>& lk, int j, int k,
                                            R& drho, R& jz, R& jr, R& psi) {
    drho = R(0), jz = R(0), jr = R(0), psi = R(0);
#pragma unroll
    for (int i = 0; i < Q; i++) {
        drho += f[i];
        jz += R(cz_of(i)) * f[i];
        jr += R(cr_of(i)) * f[i];
    }
    if (lk.src) {
        // arrival halves h_i(y)/2: zeroth moment S0/2, first moment H/2
        const long long o = (long long)j * p.pitch + k;
        drho += R(0.5) * lk.src[o];
        jz += R(0.5) * lk.src[p.plane + o];
        jr += R(0.5) * lk.src[2 * p.plane + o];
    }
    const R rho = p.rho_ref + drho;
    int bad = 0;
    if (!(rho > R(0))) bad |= ERRBIT_RHO;
    if (!isfinite(jz) || !isfinite(jr)) bad |= ERRBIT_NONFINITE;
    if (p.multiphase) {
        const R arg = rho * (R(1) / R(3)) - eos_p(p, rho);
        if (!(arg >= R(0))) bad |= ERRBIT_PSI;
        psi = sqrt(arg > R(0) ? arg : R(0));
    }
    return bad;
}

// Pull-gather the nine populations of node (k, j) and write rho - rho_ref, j_z,
// j_r, psi.  Raises error bits; never traps.
template <typename R>
__global__ void __launch_bounds__(256) k_density(Params<R> p, const R* __restrict__ f, R* __restrict__ aux,
                                                 int* __restrict__ err, LinkPlanes<R> lk) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (k >= p.nz || j >= p.nr) return;
    R fi[Q], drho, jz, jr, psi;
#pragma unroll
    for (int i = 0; i < Q; i++) fi[i] = f[pull_slot(p, k, j, i)];
    const int bad = density_node(p, fi, lk, j, k, drho, jz, jr, psi);
    if (bad) atomicOr(err, bad);
    const long long o = (long long)j * p.pitch + k;
    aux[o] = drho;
    aux[p.plane + o] = jz;
    aux[2 * p.plane + o] = jr;
    aux[3 * p.plane + o] = psi;
}

// ------------------------------------------------------ stencil helpers --
// Isotropic derivative, Eq. (fifthorderaccuratefinitedifference), on a
// shared-memory tile of row width W centred at m:
// d_z = 1/36 [8 (sum of the 3 nodes at dz=+1 - those at dz=-1)
//            - (sum of the 3 nodes at +2 c_i with c_z=+1 - those with c_z=-1)].
template <typename R, int W>
__device__ __forceinline__ R fd_z(const R* m) {
    const R n1 = (m[1] + m[1 + W] + m[1 - W]) - (m[-1] + m[-1 + W] + m[-1 - W]);
    const R n2 = (m[2] + m[2 + 2 * W] + m[2 - 2 * W]) - (m[-2] + m[-2 + 2 * W] + m[-2 - 2 * W]);
    return (R(8) * n1 - n2) * (R(1) / R(36));
}
template <typename R, int W>
__device__ __forceinline__ R fd_r(const R* m) {
    const R n1 = (m[W] + m[W + 1] + m[W - 1]) - (m[-W] + m[-W + 1] + m[-W - 1]);
    const R n2 = (m[2 * W] + m[2 * W + 2] + m[2 * W - 2]) - (m[-2 * W] + m[-2 * W + 2] + m[-2 * W - 2]);
    return (R(8) * n1 - n2) * (R(1) / R(36));
}

// Kupershtokh force, Eq. (kupershtokhforcing) with dt = 1:
// F = 6 [A sum_i w_i psi^2(x+c_i) c_i + (1-2A) psi(x) sum_i w_i psi(x+c_i) c_i].
template <typename R, int W>
__device__ __forceinline__ void kupershtokh(const R* m, R A, R& fz, R& fr) {
    const R e = m[1], w = m[-1], n = m[W], s = m[-W];
    const R ne = m[W + 1], nw = m[W - 1], se = m[-W + 1], sw = m[-W - 1];
    const R c9 = R(1) / R(9), c36 = R(1) / R(36);
    const R s1z = c9 * (e - w) + c36 * ((ne + se) - (nw + sw));
    const R s1r = c9 * (n - s) + c36 * ((ne + nw) - (se + sw));
    const R s2z = c9 * (e * e - w * w) + c36 * ((ne * ne + se * se) - (nw * nw + sw * sw));
    const R s2r = c9 * (n * n - s * s) + c36 * ((ne * ne + nw * nw) - (se * se + sw * sw));
    const R b = (R(1) - R(2) * A) * m[0];
    fz += R(6) * (A * s2z + b * s1z);
    fr += R(6) * (A * s2r + b * s1r);
}

// Total force and physical velocity of a node in row j from its psi tile (m, row width WP) and its
// psi_z, psi_r tiles (width WD); u = j / rho + F / (2 rho) (Sec. II.A, half-force shift).
template <int WP, int WD, typename R>
__device__ __forceinline__ void velocity_node(const Params<R>& p, const R* m, const R* pz, const R* pr, int j, R drho,
                                              R jz, R jr, bool mp, bool ax, R& fz, R& fr, R& uz, R& ur) {
    const R rho = p.rho_ref + drho;
    fz = rho * p.gz, fr = R(0);
    if (mp) {
        kupershtokh<R, WP>(m, p.A, fz, fr);
        if (ax) {
            // F_axis = 3 kappa [psi grad_c(psi_r / r) + (c A / r) psi_r grad_c psi],
            // Eq. (multiphasecorrections) (c = 6 as printed, 2 from the exact expansion);
            // psi_rr = D_r(psi_r), psi_rz = D_r(psi_z).
            const R psi = m[0], psz = pz[0], psr = pr[0];
            const R prr = fd_r<R, WD>(pr);
            const R prz = fd_r<R, WD>(pz);
            const R ir = R(1) / (R(j) + R(0.5));
            const R k3 = R(3) * kappa_of(p, rho);
            const R a6 = p.axis_a * p.A * ir * psr;
            fz += k3 * (psi * prz * ir + a6 * psz);
            fr += k3 * (psi * (prr - psr * ir) * ir + a6 * psr);
        }
    }
    uz = (jz + R(0.5) * fz) / rho;
    ur = (jr + R(0.5) * fr) / rho;
}

// ------------------------------------- kernel (b): the fused update step --
// One CTA owns a TZ x TR tile of nodes.  Staged in shared memory:
//   psi            tile + 6 (F on a 2-ring needs psi_rr, which needs psi_r on a 4-ring)
//   psi_z, psi_r   tile + 4
//   rho-rho_ref, j tile + 2
//   u (physical)   tile + 2 (velocity gradients of H)
//   F              tile
// Values of psi_z, psi_r and u beyond the axis or a wall are the mirror
// images of interior values with their parity (psi, psi_z, u_z even; psi_r,
// u_r odd; u_z odd at a no-slip wall), evaluated at the mirrored node.
template <int TZ, int TR>
struct TileShape {
    static constexpr int PW = TZ + 12, PH = TR + 12;
    static constexpr int DW = TZ + 8, DH = TR + 8;
    static constexpr int UW = TZ + 4, UH = TR + 4;
    static constexpr int elems = PW * PH + 2 * DW * DH + 5 * UW * UH + 2 * TZ * TR;
};

// GUO: Guo forcing (Sec. II.A) in place of the EDM shift.
template <typename R, int TZ, int TR, bool GUO = false>
__global__ void __launch_bounds__(256) k_update(Params<R> p, const R* __restrict__ f, R* __restrict__ fout,
                                                const R* __restrict__ aux, LinkPlanes<R> lk) {
    using S = TileShape<TZ, TR>;
    constexpr int PW = S::PW, PH = S::PH, DW = S::DW, DH = S::DH, UW = S::UW, UH = S::UH;
    constexpr int NT = 256;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R* sPsi = reinterpret_cast<R*>(smem_raw);
    R* sPz = sPsi + PW * PH;
    R* sPr = sPz + DW * DH;
    R* sRho = sPr + DW * DH;
    R* sJz = sRho + UW * UH;
    R* sJr = sJz + UW * UH;
    R* sUz = sJr + UW * UH;
    R* sUr = sUz + UW * UH;
    R* sFz = sUr + UW * UH;
    R* sFr = sFz + TZ * TR;

    const int tid = threadIdx.x;
    const int k0 = blockIdx.x * TZ, j0 = blockIdx.y * TR;
    const int kn = min(TZ, p.nz - k0), jn = min(TR, p.nr - j0);
    const bool mp = p.multiphase != 0, ax = p.axis != 0;
    const int uz_top = p.top == TOP_NOSLIP ? -1 : 1;

    // Stage 0: load psi (ring 6) and rho - rho_ref, j (ring 2).
    if (mp) {
        for (int idx = tid; idx < PW * PH; idx += NT) {
            const int a = idx / PW, b = idx - a * PW;
            if (a >= jn + 12 || b >= kn + 12) continue;
            int s;
            const int jm = map_row(p, j0 - 6 + a, 1, 1, s);
            const int km = wrap_any(k0 - 6 + b, p.nz);
            sPsi[idx] = aux[3 * p.plane + (long long)jm * p.pitch + km];
        }
    }
    for (int idx = tid; idx < UW * UH; idx += NT) {
        const int a = idx / UW, b = idx - a * UW;
        if (a >= jn + 4 || b >= kn + 4) continue;
        int s;
        const int jm = map_row(p, j0 - 2 + a, 1, 1, s);
        const int km = wrap_any(k0 - 2 + b, p.nz);
        const long long o = (long long)jm * p.pitch + km;
        sRho[idx] = aux[o];
        sJz[idx] = aux[p.plane + o];
        sJr[idx] = aux[2 * p.plane + o];
    }
    __syncthreads();

    // Stage 1: psi_z, psi_r on the 4-ring (needed for psi_rr, psi_rz of F_axis).
    if (mp && ax) {
        for (int idx = tid; idx < DW * DH; idx += NT) {
            const int a = idx / DW, b = idx - a * DW;
            if (a >= jn + 8 || b >= kn + 8) continue;
            int s;
            const int jm = map_row(p, j0 - 4 + a, -1, -1, s);
            // mirrored rows are evaluated at their interior image; wrapped rows in place
            const int jl = p.top == TOP_PERIODIC ? j0 - 4 + a : jm;
            const R* m = sPsi + (jl - j0 + 6) * PW + (b + 2);
            sPz[idx] = fd_z<R, PW>(m);
            sPr[idx] = R(s) * fd_r<R, PW>(m);
        }
        __syncthreads();
    }

    // Stage 2: total force and physical velocity on the 2-ring.
    for (int idx = tid; idx < UW * UH; idx += NT) {
        const int a = idx / UW, b = idx - a * UW;
        if (a >= jn + 4 || b >= kn + 4) continue;
        int s_ur, s_uz;
        const int jm = map_row(p, j0 - 2 + a, -1, -1, s_ur);
        map_row(p, j0 - 2 + a, 1, uz_top, s_uz);
        const int jl = p.top == TOP_PERIODIC ? j0 - 2 + a : jm;  // see stage 1
        const int lu = (jl - j0 + 2) * UW + b;
        R fz, fr, uz, ur;
        const int ld = (jl - j0 + 4) * DW + (b + 2);
        velocity_node<PW, DW>(p, sPsi + (jl - j0 + 6) * PW + (b + 4), sPz + ld, sPr + ld, jm, sRho[lu], sJz[lu], sJr[lu],
                              mp, ax, fz, fr, uz, ur);
        sUz[idx] = R(s_uz) * uz;
        sUr[idx] = R(s_ur) * ur;
        const int ti = a - 2, tk = b - 2;
        if (ti >= 0 && ti < jn && tk >= 0 && tk < kn) {
            sFz[ti * TZ + tk] = fz;
            sFr[ti * TZ + tk] = fr;
        }
    }
    __syncthreads();

    // Stage 3: collide the tile's own nodes.
    for (int idx = tid; idx < TZ * TR; idx += NT) {
        const int ti = idx / TZ, tk = idx - ti * TZ;
        if (ti >= jn || tk >= kn) continue;
        const int k = k0 + tk, j = j0 + ti;
        const int lu = (ti + 2) * UW + (tk + 2);
        const R drho = sRho[lu];
        const R rho = p.rho_ref + drho;
        const R uz = sUz[lu], ur = sUr[lu];
        const R irho = R(1) / rho;
        const R u0z = sJz[lu] / rho, u0r = sJr[lu] / rho;
        const R duz = sFz[ti * TZ + tk] * irho, dur = sFr[ti * TZ + tk] * irho;
        R Hz = R(0), Hr = R(0), m0 = R(0);
        if (ax) {
            // H of Eq. (axihz) with the c_i factors taken outside H and the
            // viscous hoop term 2 mu d_r(u_r/r) (hr_sign = -1).
            const R duz_dr = fd_r<R, UW>(sUz + lu);
            const R dur_dz = fd_z<R, UW>(sUr + lu);
            const R dur_dr = fd_r<R, UW>(sUr + lu);
            const R ir = R(1) / (R(j) + R(0.5));
            const R mu = rho * p.nu;
            Hz = (mu * (duz_dr + dur_dz) - rho * ur * uz) * ir;
            Hr = (R(2) * mu * (dur_dr + R(p.hr_sign) * ur * ir) - rho * ur * ur) * ir;
            m0 = -rho * ur * ir;
        }
        const R u0sq = u0z * u0z + u0r * u0r;
        const R sz = R(2) * u0z + duz, sr = R(2) * u0r + dur;  // u0 + u1
        const R dusum = duz * sz + dur * sr;                   // u1^2 - u0^2
        // Guo forcing: f^eq at the fluid velocity u, and
        // S_i = w_i (1 - 1/(2 tau)) [3 (c_i - u).F + 9 (c_i.u)(c_i.F)]
        const R Fz = sFz[ti * TZ + tk], Fr = sFr[ti * TZ + tk];
        const R usq = uz * uz + ur * ur, uF = uz * Fz + ur * Fr;
        const R gpre = R(1) - R(0.5) * p.tau_inv;
        const long long o = (long long)j * p.pitch + k;
        // link-midpoint source: arrival half of the previous step's h at this
        // node, departure half of this step's; this step's S0, H kept for the next
        R a0 = R(0), az = R(0), ar = R(0), hs = R(1);
        if (lk.src) {
            a0 = lk.src[o];
            az = lk.src[p.plane + o];
            ar = lk.src[2 * p.plane + o];
            lk.dst[o] = m0;
            lk.dst[p.plane + o] = Hz;
            lk.dst[2 * p.plane + o] = Hr;
            hs = R(0.5);
        }
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const R w = w_of<R>(i);
            const R cx = R(cz_of(i)), cy = R(cr_of(i));
            R fi = f[pull_slot(p, k, j, i)];
            if (lk.src) fi += R(0.5) * w * (a0 + R(3) * (cx * az + cy * ar));
            R feq, force;
            if (GUO) {
                const R cu = cx * uz + cy * ur, cF = cx * Fz + cy * Fr;
                feq = w * (drho + rho * (R(3) * cu + R(4.5) * cu * cu - R(1.5) * usq));
                force = w * gpre * (R(3) * (cF - uF) + R(9) * cu * cF);
            } else {
                const R cu0 = cx * u0z + cy * u0r;
                const R cdu = cx * duz + cy * dur;
                const R csum = cx * sz + cy * sr;
                // f^eq(rho, u0) - w_i rho_ref (Sec. II.A) and the EDM shift
                // f^eq(rho, u0 + F/rho) - f^eq(rho, u0) written as a difference
                feq = w * (drho + rho * (R(3) * cu0 + R(4.5) * cu0 * cu0 - R(1.5) * u0sq));
                force = w * rho * (R(3) * cdu + R(4.5) * cdu * csum - R(1.5) * dusum);
            }
            const R h = hs * w * (m0 + R(3) * (cx * Hz + cy * Hr));  // h_i (Sec. II.B)
            fout[i * p.plane + o] = fi + (feq - fi) * p.tau_inv + force + h;
        }
    }
}

// --------------------------------------------------------------- init --
// f_i = f_i^eq(rho, u) - w_i rho_ref, written to the slot from which the
// next pull reads population i of node (k, j).
template <typename R>
__global__ void __launch_bounds__(256) k_init(Params<R> p, double rho_ref, const double* __restrict__ rho,
                                              const double* __restrict__ uz, const double* __restrict__ ur,
                                              R* __restrict__ f, const R* __restrict__ phys,
                                              const int* __restrict__ err) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (k >= p.nz || j >= p.nr) return;
    const long long c = (long long)j * p.nz + k;
    const double d = rho[c];
    double vz = uz ? uz[c] : 0.0, vr = ur ? ur[c] : 0.0;
    if (phys) {
        // the fluid velocity is to be (vz, vr), and u + F / (2 rho) of f^eq(rho, u) is phys (two pitched
        // planes): the bare velocity u - F / (2 rho) = u - (phys - u).  A state that raised an error stays.
        if (*err) return;
        const R* q = phys + ((long long)j * p.pitch + k);
        vz = vz - ((double)q[0] - vz);
        vr = vr - ((double)q[p.plane] - vr);
    }
    if constexpr (sizeof(R) == 4) {
        // FP32 deviations f_i - w_i rho_ref = w_i [(rho - rho_ref) + rho (3 c.u + 4.5 (c.u)^2 - 1.5 u.u)]:
        // rho - rho_ref in FP64, the velocity part in FP32 (FP64 arithmetic would set this kernel's time)
        const float dr = (float)(d - rho_ref), rf = (float)d, zf = (float)vz, rrf = (float)vr;
        const float usq = zf * zf + rrf * rrf;
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const float cu = (float)cz_of(i) * zf + (float)cr_of(i) * rrf;
            f[pull_slot(p, k, j, i)] = w_of<float>(i) * (dr + rf * (3.0f * cu + 4.5f * cu * cu - 1.5f * usq));
        }
    } else {
        const double usq = vz * vz + vr * vr;
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const double cu = cz_of(i) * vz + cr_of(i) * vr;
            const double w = w_of<double>(i);
            const double feq = w * d * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq);
            f[pull_slot(p, k, j, i)] = (R)(feq - w * rho_ref);
        }
    }
}

// --------------------------------------------- kernel (c): reductions --
// FP64 sums; one partial per block, summed by k_reduce_final in a fixed order, so results are bitwise
// reproducible for a given grid.  block_sum adds over a block of 256 threads: one warp per value, 7
// additions and 5 shuffle steps for 256 terms.  (Five shuffle steps in each of 8 warps for every value take
// three times the FP64 pipe, which bounds the sums: mass of 2048 x 1024 45 us that way, 38 this way; the
// pressure jump 105 and 83.)
template <int N>
__device__ __forceinline__ void block_sum(double (&v)[N], double* out) {
    static_assert(N <= 8, "one warp per value");
    __shared__ double all[N][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < N; q++) all[q][threadIdx.x] = v[q];
    __syncthreads();
    if (warp < N) {
        double s = all[warp][lane];
#pragma unroll
        for (int i = 1; i < 8; i++) s += all[warp][lane + 32 * i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) out[warp] = s;
    }
}

// Final sum of the per-block partials by one block (launch <<<1, 256>>>): thread t
// adds partials t, t + 256, ... in that order, then block_sum combines the
// threads.  The order is fixed, so the result is bitwise reproducible for a
// given number of partials.
template <int N>
__global__ void __launch_bounds__(256) k_reduce_final(const double* __restrict__ partial, int nblocks,
                                                      double* __restrict__ out) {
    double s[N];
#pragma unroll
    for (int q = 0; q < N; q++) s[q] = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += 256) {
#pragma unroll
        for (int q = 0; q < N; q++) s[q] += partial[N * b + q];
    }
    block_sum<N>(s, out);
}

}  // namespace lbm
