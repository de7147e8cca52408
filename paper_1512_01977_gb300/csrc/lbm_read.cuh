// Reading a solve: fields (rho, u, P_k), masses and the pressure jump, each in
// one pass over the populations.  The moments of the arrived populations are
// gathered where they are used, so no field plane is written and read again,
// and results go straight to their destination.
//
// What bounds these passes is the FP64 arithmetic of P_k and of the sums (1.9
// lanes per clock and SM: 14 us per operation and node of a 4096 x 2048 solve),
// so P_k is evaluated in 10 or 11 operations (30 with its division), FP32 values
// are widened by their bits and distances are compared in FP32 where that
// decides.  What each read took and takes stands at its kernel, host call included.
#pragma once

#include "lbm_phase.cuh"

namespace lbm {

// FP32 -> FP64 by the bits (integer pipe); zero, subnormal and non-finite values by conversion.
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), e = (b >> 23) & 255u;
    if (e - 1u >= 254u) return (double)x;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

// P_k in FP64 (rho / 3 for a single-phase run), as exact as the formula with its quotient (units of 2^-53 of
// P_k + rho^2, rms over the coexistence range at 0.5 to 0.9 T_c: CS 0.6-0.8 and 1.3-1.5, vdW the same 0.12-0.04).
// vdW: the quotient is the product with the reciprocal and one correction by its remainder.  CS: with
// x = 1 - e, e = b rho / 4, the quotient (1 + e + e^2 - e^3) / x^3 is 1 + 2 e (x^-3 + x^-2), a sum of positive
// terms.  (Written 1 + 2 (x^-3 - x^-1) it cancels at low density: 2.4.)
__device__ __forceinline__ double pressure(const Params<double>& p, double rho) {
    if (!p.multiphase) {
        // rho / 3, correctly rounded (Markstein 1990: from the rounded 1/3 and the remainder), an infinity kept
        const double q = mul(rho, 1.0 / 3.0);
        return finite1(rho) ? fma(fma(-3.0, q, rho), 1.0 / 3.0, q) : q;
    }
    if (p.eos == EOS_VDW) {
        const double d = 3.0 - rho, r = rcp3(d), n = 8.0 * p.T * rho, q0 = mul(n, r);
        const double q = finite1(q0) ? fma(fma(-d, q0, n), r, q0) : q0;
        return mul(p.lambda, fma(-3.0 * rho, rho, q));
    }
    const double r = rcp3(fma(-0.25 * p.b, rho, 1.0)), r2 = mul(r, r), RT = p.Rg * p.T;
    return mul(rho, fma(-p.a, rho, fma(mul(0.5 * p.b * RT, rho), fma(r2, r, r2), RT)));
}

// Where a field pass writes: FP64 arrays [j * nz + k] (null: not wanted) and u in the storage type
// into two pitched planes (null: not wanted).
template <typename R>
struct FieldsOut {
    double *rho, *uz, *ur, *p;
    R* u;
};

template <typename R>
__device__ __forceinline__ void put_fields(const FieldsOut<R>& o, const Params<R>& p, const Params<double>& pd, int j,
                                           int k, R drho, R uz, R ur) {
    const long long c = (long long)j * p.nz + k;
    const double rho = pd.rho_ref + widen(drho);
    if (o.rho) o.rho[c] = rho;
    if (o.uz) o.uz[c] = widen(uz);
    if (o.ur) o.ur[c] = widen(ur);
    if (o.p) o.p[c] = pressure(pd, rho);
    if (o.u) {
        R* u = o.u + (j * p.pitch + k);
        u[0] = uz;
        u[p.plane] = ur;
    }
}

// Arrived populations of node (k, j).
template <typename R>
__device__ __forceinline__ void pull_node(const Params<R>& p, const R* __restrict__ f, int j, int k, R (&fi)[Q]) {
    const PullRow q = pull_row(p, j);
    const int km = k == 0 ? p.nz - 1 : k - 1, kp = k + 1 == p.nz ? 0 : k + 1;
#pragma unroll
    for (int i = 0; i < Q; i++) {
        const int col = cz_of(i) > 0 ? km : (cz_of(i) < 0 ? kp : k);
        fi[i] = f[q.o[i] + ((i == 6 || i == 7) && q.stay ? k : col)];
    }
}

// Density, momentum and psi of a node from its populations, with its error bits: FP32 as k_density
// has it, FP64 in phase_l1's operations.  PSI: psi itself is wanted, not only its check.
template <bool PSI>
__device__ __forceinline__ int node_moments(const Params<float>& p, const float* __restrict__ f,
                                            const LinkPlanes<float>& lk, int j, int k, float& drho, float& jz,
                                            float& jr, float& psi) {
    float fi[Q];
    pull_node(p, f, j, k, fi);
    return density_node(p, fi, lk, j, k, drho, jz, jr, psi);
}
template <bool PSI>
__device__ __forceinline__ int node_moments(const Params<double>& p, const double* __restrict__ f,
                                            const LinkPlanes<double>& lk, int j, int k, double& drho, double& jz,
                                            double& jr, double& psi) {
    double fi[Q];
    pull_node(p, f, j, k, fi);
    moments1(fi, drho, jz, jr);
    if (lk.src) {
        double a[3];
        link3(p, lk.src, j, k, a);
        drho = fma(0.5, a[0], drho);
        jz = fma(0.5, a[1], jz);
        jr = fma(0.5, a[2], jr);
    }
    const double rho = p.rho_ref + drho;
    int bad = (positive(rho) ? 0 : ERRBIT_RHO) | (finite1(jz) && finite1(jr) ? 0 : ERRBIT_NONFINITE);
    psi = 0.0;
    if (p.multiphase) {
        const double arg = fma(rho, 1.0 / 3.0, -eos_p3(p, rho));
        if (!nonnegative(arg)) bad |= ERRBIT_PSI;
        if (PSI) psi = sqrt3(arg);
    }
    return bad;
}

// Fields of an FP32 solve: 32 x TR nodes per block with 4 columns and rows of psi around them
// gathered again (F needs psi_rr).  The velocity is k_update's, operation for operation.
// 4096 x 2048: 277 us, and 598 as k_density, k_update's moments form and four copies (density alone 117).
// TR by size: the taller the tile, the less halo, and 32 rows beat 16 by 26 us there; 2048 x 1024 takes the
// same 100 us either way, and below 152 blocks' worth of nodes 8 rows give every SM one.
template <int TR>
struct FieldsShape {
    static constexpr int TZ = 32, WP = TZ + 8, WD = TZ + 4;
    static constexpr int elems = WP * (TR + 8) + 2 * WD * (TR + 4) + 3 * TZ * TR;
};
template <int TR>
__global__ void __launch_bounds__(256) k_fields(Params<float> p, Params<double> pd, const float* __restrict__ f,
                                                LinkPlanes<float> lk, FieldsOut<float> out, int* __restrict__ err) {
    using S = FieldsShape<TR>;
    constexpr int TZ = S::TZ, WP = S::WP, WD = S::WD, NT = 256;
    __shared__ float smem[S::elems];
    float* sPsi = smem;
    float* sPz = sPsi + WP * (TR + 8);
    float* sPr = sPz + WD * (TR + 4);
    float* sRho = sPr + WD * (TR + 4);
    float* sJz = sRho + TZ * TR;
    float* sJr = sJz + TZ * TR;
    const int tid = threadIdx.x, across = (p.nz + TZ - 1) / TZ, ti = blockIdx.x / across;
    const int k0 = (blockIdx.x - ti * across) * TZ, j0 = ti * TR;
    const int kn = min(TZ, p.nz - k0), jn = min(TR, p.nr - j0);
    const bool mp = p.multiphase != 0, ax = p.axis != 0, want_u = out.uz || out.ur || out.u;
    int bad = 0;
    phase_wait();
    for (int i = tid; i < WP * (TR + 8); i += NT) {
        const int a = i / WP, b = i - a * WP, tj = a - 4, tk = b - 4;
        const bool own = tj >= 0 && tj < jn && tk >= 0 && tk < kn;
        if (a >= jn + 8 || b >= kn + 8 || !((mp && want_u) || own)) continue;
        int s;
        const int jm = map_row(p, j0 + tj, 1, 1, s), km = wrap_any(k0 + tk, p.nz);
        float drho, jz, jr, psi;
        bad |= node_moments<true>(p, f, lk, jm, km, drho, jz, jr, psi);
        sPsi[i] = psi;
        if (own) {
            const int o = tj * TZ + tk;
            sRho[o] = drho;
            sJz[o] = jz;
            sJr[o] = jr;
        }
    }
    if (bad) atomicOr(err, bad);
    __syncthreads();
    if (!want_u) {
        for (int i = tid; i < TZ * TR; i += NT) {
            const int tj = i / TZ, tk = i - tj * TZ;
            if (tj < jn && tk < kn) put_fields(out, p, pd, j0 + tj, k0 + tk, sRho[i], 0.0f, 0.0f);
        }
        return;
    }
    if (mp && ax) {
        for (int i = tid; i < WD * (TR + 4); i += NT) {
            const int a = i / WD, b = i - a * WD;
            if (a >= jn + 4 || b >= kn + 4) continue;
            int s;
            const int jm = map_row(p, j0 - 2 + a, -1, -1, s);
            // mirrored rows are evaluated at their interior image; wrapped rows in place
            const int jl = p.top == TOP_PERIODIC ? j0 - 2 + a : jm;
            const float* m = sPsi + (jl - j0 + 4) * WP + (b + 2);
            sPz[i] = fd_z<float, WP>(m);
            sPr[i] = float(s) * fd_r<float, WP>(m);
        }
        __syncthreads();
    }
    for (int i = tid; i < TZ * TR; i += NT) {
        const int tj = i / TZ, tk = i - tj * TZ;
        if (tj >= jn || tk >= kn) continue;
        float uz, ur, fz, fr;
        velocity_node<WP, WD>(p, sPsi + (tj + 4) * WP + (tk + 4), sPz + (tj + 2) * WD + (tk + 2),
                              sPr + (tj + 2) * WD + (tk + 2), j0 + tj, sRho[i], sJz[i], sJr[i], mp, ax, fz, fr, uz, ur);
        put_fields(out, p, pd, j0 + tj, k0 + tk, sRho[i], uz, ur);
    }
}

// Fields of an FP64 solve: k_phase_l's planes, then its velocity phase writing to the destination.
// 1024 x 512: 210 us, and 437 as k_density, k_update's moments form and four copies.
template <int TR, bool MP, bool AX>
__global__ void __launch_bounds__(32 * TR) k_fields64(const PhaseOne<double> a, const FieldsOut<double> out,
                                                      const Params<double> pd) {
    __shared__ __align__(16) double smem[PhaseU1<TR>::elems];
    const int ti = blockIdx.x / a.across, tk = blockIdx.x - ti * a.across;
    phase_wait();
    const PhaseWork<double> w = phase_work(a.s, a.parity, a.err, tk * PhaseShape<double>::TZ, ti * TR);
    phase_u1<TR, MP, AX>(a.s.p, w, smem, 0, [&](int row, int k, double drho, double uz, double ur, double) {
        put_fields(out, a.s.p, pd, row, k, drho, uz, ur);
    });
}

// Sum of (j + 1/2) rho and of rho.  Summed over the deviations rho - rho_ref (one FP64 addition and
// one fused multiply per node); the reference's share is nz nr rho_ref and nz nr^2/2 rho_ref.
// 2048 x 1024: 38 us, and 78 as k_density, k_mass and the final sum; 4096 x 2048: 97.
template <typename R>
__global__ void __launch_bounds__(256) k_mass(Params<R> p, const R* __restrict__ f, LinkPlanes<R> lk,
                                              double* __restrict__ partial, int* __restrict__ err) {
    double v[2] = {0.0, 0.0};
    int bad = 0;
    const int n = p.nz * p.nr;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        const int j = c / p.nz, k = c - j * p.nz;
        R drho, jz, jr, psi;
        bad |= node_moments<false>(p, f, lk, j, k, drho, jz, jr, psi);
        const double d = widen(drho);
        v[0] = fma(__hiloint2double(0x43300000, j) - 4503599627370495.5, d, v[0]);  // 2^52 + j - (2^52 - 1/2)
        v[1] += d;
    }
    if (bad) atomicOr(err, bad);
    block_sum<2>(v, partial + 2 * blockIdx.x);
}

// Sums of P_k and node counts inside d < r_in and outside d > r_out.  The distance is compared in FP32
// unless it is within 1e-5 of a radius (relative; FP32 errs by a few 1e-7), then in FP64 as before.
// 2048 x 1024: 83 us, and 232 with k_density and an FP64 root and quotient per node.
template <typename R>
__global__ void __launch_bounds__(256) k_pjump(Params<R> p, Params<double> pd, const R* __restrict__ f,
                                               LinkPlanes<R> lk, double zc, double rc, double rin, double rout,
                                               double* __restrict__ partial, int* __restrict__ err) {
    double v[2] = {0.0, 0.0};
    int count[2] = {0, 0}, bad = 0;
    const int n = p.nz * p.nr;
    const float zf = (float)zc, rf = (float)rc, in2 = (float)(rin * rin), out2 = (float)(rout * rout);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        const int j = c / p.nz, k = c - j * p.nz;
        R drho, jz, jr, psi;
        bad |= node_moments<false>(p, f, lk, j, k, drho, jz, jr, psi);
        const float dz = (float)k + 0.5f - zf, dr = (float)j + 0.5f - rf, d2 = dz * dz + dr * dr;
        bool in = d2 < in2, out = d2 > out2;
        // how far the coordinates' own rounding may move d^2
        const float slack = 1e-5f * d2 + 1e-6f * (fabsf(dz) + fabsf(dr) + 1.0f) * (fabsf(zf) + fabsf(rf) + (float)k + (float)j);
        if (!(fabsf(d2 - in2) > slack && fabsf(d2 - out2) > slack)) {
            const double ez = k + 0.5 - zc, er = j + 0.5 - rc, d = sqrt(ez * ez + er * er);
            in = d < rin;
            out = d > rout;
        }
        if (in || out) {
            const double pk = pressure(pd, pd.rho_ref + widen(drho));
            if (in) {
                v[0] += pk;
                count[0]++;
            } else {
                v[1] += pk;
                count[1]++;
            }
        }
    }
    if (bad) atomicOr(err, bad);
    double w[4] = {v[0], (double)count[0], v[1], (double)count[1]};
    block_sum<4>(w, partial + 4 * blockIdx.x);
}

// The error word to the host, cleared on the device.
static __global__ void k_take_error(int* __restrict__ err, int* __restrict__ host) {
    phase_wait();
    *host = *err;
    *err = 0;
}

}  // namespace lbm
