"""The work this engine is used for, as cases that can be timed.

A case is one repeated piece of a user's program over the ctypes interface
(paper_1512_01977_gb300.lbm, .serve): advance a solve some steps and read its
fields, advance a batch and read every solve, start a solve and take its
diagnostics, serve a list of requests.  Stepped droplets and waves start at
rest, as the validation runs do, and lie in the stable range of density ratio
and tau, so a pass may be repeated on the same state any number of times.

Fields come back as doubles from the interface.  Those of an FP64 solve are
returned as they are; those of an FP32 solve hold FP32 numbers (the density as
its deviation from rho_ref, which is what an FP32 solve stores), so they are
kept as float32: rho - rho_ref, u_z, u_r, P_k.

exact() is the same method in plain torch, in 64 bits, written without the
package: pull streaming on whole-field arrays, ghost rows by concatenation.
"""
import math

import numpy as np
import torch

from paper_1512_01977_gb300 import lbm
from paper_1512_01977_gb300 import serve as srv

CS, VDW = "cs", "vdw"
LAM = 0.01
A_DEFAULT = -0.152
# one pass of any case moves at most this many nodes x steps (FP64 ones count 28 times,
# the ratio of the two arithmetic rates on this GPU)
MOST_NODE_STEPS = 20 * 4096 * 2048
FP64_WEIGHT = 28
DEV = "cuda"


# ---------------------------------------------------------------- the cases --

def _solve(name, field, nz, nr, steps, prec=32, eos=CS, T=0.8, tau=1.0, A=A_DEFAULT, top="freeslip", axis=1,
           forcing="edm", kappa="thermo", axis_a=6):
    return dict(name=name, kind="solve", field=field, nz=nz, nr=nr, steps=steps, prec=prec, eos=eos, T=T, tau=tau, A=A,
                top=top, axis=axis, forcing=forcing, kappa=kappa, axis_a=axis_a)


def listed():
    return [
        # the smallest solve in use (64 x 64 stationary droplet), sampled often: launches and latency
        _solve("droplet64_fp32", "droplet", 64, 64, 10),
        # the same droplet as the FP64 parity run, a longer stretch between two samples
        _solve("droplet64_fp64", "droplet", 64, 64, 200, prec=64),
        # mode-2 oscillation on 512 x 256, its axis extent sampled every 100 steps
        _solve("oscillation512_fp32", "droplet", 512, 256, 100, tau=0.8),
        # the vdW oscillation geometry of the validation runs in FP64 (500 x 250: ragged strips)
        _solve("oscillation500_vdw_fp64", "droplet", 500, 250, 20, prec=64, eos=VDW, T=0.85, A=0.0, kappa="lattice"),
        # the planar, fully periodic droplet that the surface-tension table compares the axisymmetric runs with
        _solve("planar500_fp32", "droplet2d", 500, 500, 50, eos=VDW, T=0.8, tau=1.5, top="periodic", axis=0),
        # radial wave in a pipe: one column of 2000 nodes, an axial stream, a no-slip wall
        _solve("radial_wave_fp32", "ring", 1, 2000, 100, eos=VDW, T=0.8, tau=0.6, top="noslip"),
        # the throughput run: a density wave on 4096 x 2048
        _solve("wave4096_fp32", "wave", 4096, 2048, 20, T=0.9, tau=0.6),
        # the same wave in FP64 on a smaller lattice, under a no-slip wall
        _solve("wave1024_fp64", "wave", 1024, 512, 10, prec=64, T=0.9, tau=0.6, top="noslip"),
        # Guo forcing with the exact A-term (the option the Laplace-law study uses), odd sizes
        _solve("guo1023_fp32", "droplet", 1023, 511, 30, T=0.85, forcing="guo", kappa="lattice", axis_a=2),
        # 256 droplets of uneven sizes advanced together, then every solve read
        dict(name="batch256_fp32", kind="batch", n=256, lo_z=64, lo_r=32, scale=8.0, steps=100, prec=32, pick=4),
        # starting a large solve with a given fluid velocity and taking its diagnostics (fields, masses, pressure jump)
        dict(name="start2048_fp32", kind="start", nz=2048, nr=1024, prec=32, eos=CS, T=0.85, tau=1.0),
        # continuous batching of a handful of short requests, solver creation and read-back included
        dict(name="serve12_fp32", kind="serve", n=12, most_z=1024, most_r=512, steps=300, prec=32, pick=5),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["solve"] * 7 + ["batch", "batch", "start", "serve"])
    prec = rng.choice([32, 32, 64])
    weight = FP64_WEIGHT if prec == 64 else 1
    if what == "batch":
        n = _logint(rng, 2, 320)
        scale = rng.uniform(2.0, 8.0)
        # mean nodes of a solve, sizes log-uniform between lo and scale lo on both axes
        mean = 64 * 32 * (scale * scale - 1) / (2 * math.log(scale))
        most = max(2, int(MOST_NODE_STEPS / 2 / (weight * n * mean)))
        return dict(kind="batch", n=n, lo_z=64, lo_r=32, scale=scale, steps=min(_logint(rng, 10, 150), most), prec=prec,
                    pick=rng.randrange(1000))
    if what == "start":
        return dict(kind="start", nz=_logint(rng, 64, 4096), nr=_logint(rng, 64, 2048), prec=prec, eos=rng.choice([CS, VDW]),
                    T=rng.uniform(0.82, 0.9), tau=rng.uniform(0.9, 1.5))
    if what == "serve":
        return dict(kind="serve", n=rng.randint(2, 16), most_z=rng.randint(128, 1024), most_r=rng.randint(64, 512),
                    steps=rng.randint(100, 300), prec=32, pick=rng.randrange(1000))
    field = rng.choice(["droplet", "droplet", "wave", "wave", "droplet2d", "ring"])
    c = _solve("", field, 1, 1, 1, prec=prec)
    del c["name"]
    c["eos"] = rng.choice([CS, VDW])
    c["T"], c["tau"] = rng.uniform(0.82, 0.9), rng.uniform(0.9, 1.5)
    c["kappa"] = rng.choice(["thermo", "lattice"])
    top = 1 << 18 if prec == 64 else 1 << 23
    if field == "ring":
        c.update(nz=rng.randint(1, 4), nr=_logint(rng, 200, 4000), top="noslip", T=0.8, tau=rng.uniform(0.6, 1.0))
    elif field == "droplet2d":
        c.update(nz=_logint(rng, 64, 512), nr=_logint(rng, 64, 512), axis=0, top="periodic")
    else:
        while True:
            c.update(nz=_logint(rng, 48, 4096), nr=_logint(rng, 40, 2048))
            if c["nz"] * c["nr"] <= top and c["nz"] >= c["nr"] / 4:
                break
    if field == "wave":
        c.update(T=0.9, tau=rng.uniform(0.6, 1.2), top=rng.choice(["freeslip", "noslip"]))
    if field == "droplet" and rng.random() < 0.3:
        c.update(forcing="guo", axis_a=rng.choice([2, 6]))
    most = MOST_NODE_STEPS / (weight * c["nz"] * c["nr"])
    c["steps"] = max(1, min(_logint(rng, 5, 200), int(most)))
    return c


# ------------------------------------------------- EOS, for initial states --

def _cs_Tc():
    """T_c of Carnahan-Starling with a = 1, b = 4, R = 1 from p' = p'' = 0 (e = rho b / 4):
    e N'(1 - e) + 4 e N = N (1 - e), N = 1 + 4e + 4e^2 - 4e^3 + e^4, and R T_c = 8 a e (1 - e)^4 / (b N)."""
    def g(e):
        n, dn = 1 + e * (4 + e * (4 + e * (-4 + e))), 4 + e * (8 + e * (-12 + 4 * e))
        return e * (dn * (1 - e) + 4 * n) - n * (1 - e)

    lo, hi = 0.05, 0.3
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if g(mid) < 0 else (lo, mid)
    e = 0.5 * (lo + hi)
    return 8 * e * (1 - e) ** 4 / (4 * (1 + e * (4 + e * (4 + e * (-4 + e)))))


def _T(eos, T):
    return T if eos == VDW else T * _cs_Tc()


def _p(eos, T, r):
    if eos == VDW:
        return LAM * (8 * r * T / (3 - r) - 3 * r * r)
    return r * T * (1 + r + r * r - r ** 3) / (1 - r) ** 3 - r * r


def _dp(eos, T, r):
    if eos == VDW:
        return LAM * (24 * T / (3 - r) ** 2 - 6 * r)
    return T * (1 + 4 * r + 4 * r ** 2 - 4 * r ** 3 + r ** 4) / (1 - r) ** 4 - 2 * r


def _mu(eos, T, r):
    if eos == VDW:
        return LAM * (8 * T / 3 * math.log(r / (3 - r)) - 3 * r) + _p(eos, T, r) / r
    return T * (math.log(r) + (4 * r - 3 * r * r) / (1 - r) ** 2) - r + _p(eos, T, r) / r


def _bisect(f, lo, hi, n=200):
    s = f(lo) > 0
    for _ in range(n):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if (f(mid) > 0) == s else (lo, mid)
    return 0.5 * (lo + hi)


def _coexistence(eos, T_over_Tc):
    """Vapour and liquid densities of equal pressure and chemical potential."""
    T = _T(eos, T_over_Tc)
    mid, top = (1.0, 3 - 1e-9) if eos == VDW else (0.130443884, 1 - 1e-9)
    sv = _bisect(lambda r: _dp(eos, T, r), 1e-12, mid)  # spinodals
    sl = _bisect(lambda r: _dp(eos, T, r), mid, top)

    def at(p):
        return (_bisect(lambda r: _p(eos, T, r) - p, 1e-14, sv, 80), _bisect(lambda r: _p(eos, T, r) - p, sl, top, 80))

    p = _bisect(lambda q: _mu(eos, T, at(q)[0]) - _mu(eos, T, at(q)[1]), max(1e-15, _p(eos, T, sl) + 1e-15),
                _p(eos, T, sv), 80)
    return at(p)


# -------------------------------------------------------------- the inputs --

def _rng(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 60))
    return g


def _grid(nz, nr):
    z = torch.arange(nz, dtype=torch.float64, device=DEV) + 0.5
    r = torch.arange(nr, dtype=torch.float64, device=DEV) + 0.5
    return z[None, :], r[:, None]


def _density(c, seed):
    """Initial density (nr, nz) and the reference density of an FP32 solve: a tanh droplet of width 2 with a
    P2 perturbation, a density wave with noise, or a Gaussian ring; radius, centre, noise and phase by the seed."""
    nz, nr = c["nz"], c["nr"]
    rng = np.random.default_rng(int(seed))
    rv, rl = _coexistence(c["eos"], c["T"])
    field = c.get("field", "droplet")
    Z, R = _grid(nz, nr)
    if field == "wave":
        noise = torch.rand((nr, nz), dtype=torch.float64, device=DEV, generator=_rng(seed))
        ph = rng.uniform(0, 2 * math.pi)
        return rl * (1 + 0.01 * torch.sin(2 * math.pi * Z / nz + ph)) + 1e-4 * (2 * noise - 1), rl
    if field == "ring":
        r0 = 1.8 if c["eos"] == VDW else rl
        rc = rng.uniform(0.05, 0.1) * nr + 20
        noise = torch.rand((nr, nz), dtype=torch.float64, device=DEV, generator=_rng(seed))
        return r0 + 1e-3 * r0 * torch.exp(-(((R - rc) / 20.0) ** 2)) + 1e-6 * (2 * noise - 1), r0
    radius = 0.25 * min(nz, nr) * rng.uniform(0.97, 1.03)
    zc = nz / 2.0 + rng.uniform(-2, 2)
    if field == "droplet2d":
        dz, dr = Z - zc, R - (nr / 2.0 + rng.uniform(-2, 2))
    else:
        dz, dr = Z - zc, R
    d = torch.sqrt(dz * dz + dr * dr)
    cos_t = dz / d.clamp_min(1e-300)
    Rt = radius * (1 + rng.uniform(0.03, 0.06) * 0.5 * (3 * cos_t * cos_t - 1))
    # `squeeze`: both densities above the flat interface's, as a curved one's are (Laplace and Kelvin)
    return c.get("squeeze", 1.0) * (0.5 * (rl + rv) - 0.5 * (rl - rv) * torch.tanh(d - Rt)), rv


def _flow(nz, nr, seed):
    """A smooth flow of a few hundredths, zero on the axis in u_r."""
    Z, R = _grid(nz, nr)
    ph = np.random.default_rng(int(seed) + 1).uniform(0, 2 * math.pi, 2)
    uz = 0.03 * torch.sin(2 * math.pi * Z / nz + ph[0]) * torch.cos(math.pi * R / nr)
    ur = 0.02 * torch.sin(2 * math.pi * Z / nz + ph[1]) * torch.sin(math.pi * R / nr)
    return uz.contiguous(), ur.contiguous()


def _axial(nz, nr):
    """An axial stream that falls to zero at the outer wall, for the radial wave to run through."""
    uz = (0.02 * torch.cos(0.5 * math.pi * _grid(nz, nr)[1] / nr)).expand(nr, nz).contiguous()
    return uz, torch.zeros_like(uz)


def _start_solve(c):
    return dict(_solve("", "droplet", c["nz"], c["nr"], 0, prec=c["prec"], eos=c["eos"], T=c["T"], tau=c["tau"]), squeeze=1.01)


def _batch_cases(c):
    """The batch's solves: sizes log-uniform between (lo_z, lo_r) and scale times that (same scale on both axes)."""
    rng = np.random.default_rng(c["pick"])
    out = []
    for _ in range(c["n"]):
        s = math.exp(rng.uniform(0.0, math.log(c["scale"])))
        out.append(_solve("", "droplet", int(round(c["lo_z"] * s)), int(round(c["lo_r"] * s)), c["steps"], prec=c["prec"],
                          T=float(rng.uniform(0.8, 0.88)), tau=float(rng.uniform(0.8, 1.0))))
    return out


def _requests(c, seed):
    """Requests of the served workload, all waiting at the start: grids log-uniform, droplets and waves, both EOS."""
    rng = np.random.default_rng(c["pick"])
    out = []
    for i in range(c["n"]):
        nz = int(round(math.exp(rng.uniform(math.log(32), math.log(c["most_z"])))))
        nr = int(round(math.exp(rng.uniform(math.log(32), math.log(c["most_r"])))))
        out.append(dict(id=int(seed) * 100 + i, t_arrive=0.0, kind="droplet" if i % 2 == 0 else "wave",
                        eos=CS if i % 4 < 2 else VDW, nz=nz, nr=nr, steps=int(rng.integers(c["steps"] // 3, c["steps"] + 1))))
    rng = np.random.default_rng(int(seed))
    for r in out:
        r["T_over_Tc"] = float(rng.uniform(0.82, 0.9))
    return out


def _request_density(q):
    """The density field that a request stands for (what the server itself builds)."""
    rv, rl = _coexistence(q["eos"], q["T_over_Tc"])
    nz, nr = q["nz"], q["nr"]
    Z, R = np.meshgrid(np.arange(nz) + 0.5, np.arange(nr) + 0.5)
    if q["kind"] == "droplet":
        dz = Z - nz / 2.0
        d = np.sqrt(dz * dz + R * R)
        cos_t = np.where(d > 0, dz / np.maximum(d, 1e-300), 1.0)
        Rt = 0.25 * min(nz, nr) * (1 + 0.05 * 0.5 * (3 * cos_t * cos_t - 1))
        return 0.5 * (rl + rv) - 0.5 * (rl - rv) * np.tanh(d - Rt), rv
    noise = np.random.default_rng(1000 + q["id"]).uniform(-1e-4, 1e-4, size=nz * nr).reshape(nr, nz)
    return rl * (1 + 0.01 * np.sin(2 * np.pi * Z / nz)) + noise, rl


# ---------------------------------------------------------- prepare and run --

_TOP = {"freeslip": lbm.TOP_FREESLIP, "noslip": lbm.TOP_NOSLIP, "periodic": lbm.TOP_PERIODIC}


def _eos_of(c):
    return lbm.make_eos(lbm.EOS_CS if c["eos"] == CS else lbm.EOS_VDW, c["T"], lam=LAM)


def _solver(c, seed):
    rho, ref = _density(c, seed)
    s = lbm.Solver(c["nz"], c["nr"], c["tau"], eos=_eos_of(c), A=c["A"], precision=c["prec"], top=_TOP[c["top"]],
                   axis=c["axis"], kappa=lbm.KAPPA_LATTICE if c["kappa"] == "lattice" else lbm.KAPPA_THERMO,
                   rho_ref=ref if c["prec"] == 32 else 0.0,
                   forcing=lbm.FORCING_GUO if c["forcing"] == "guo" else lbm.FORCING_EDM,
                   axis_a_term=lbm.AXIS_A_EXPANSION if c["axis_a"] == 2 else lbm.AXIS_A_PRINTED)
    rho, flow = rho.contiguous(), _axial(c["nz"], c["nr"]) if c["field"] == "ring" else ()
    torch.cuda.synchronize()
    lbm.lbm_axi_init_physical_device(s.h, rho, *flow)
    return s, rho, ref


def prepare(case, seed):
    c = case
    if c["kind"] == "solve":
        s, rho, ref = _solver(c, seed)
        return dict(c=c, s=s, ref=ref, out=torch.empty((4, c["nr"], c["nz"]), dtype=torch.float64, device=DEV))
    if c["kind"] == "batch":
        got = [_solver(b, int(seed) * 1000 + i) for i, b in enumerate(_batch_cases(c))]
        solvers = [g[0] for g in got]
        outs = [torch.empty((3, s.nr, s.nz), dtype=torch.float64, device=DEV) for s in solvers]
        return dict(c=c, s=solvers, ref=[g[2] for g in got], out=outs, batch=lbm.Batch(solvers))
    if c["kind"] == "start":
        full = _start_solve(c)
        s, rho, ref = _solver(full, seed)
        return dict(c=c, s=s, ref=ref, rho=rho, u=_flow(c["nz"], c["nr"], seed), out=torch.empty((4, c["nr"], c["nz"]), dtype=torch.float64, device=DEV))
    reqs = _requests(c, seed)
    return dict(c=c, reqs=reqs, ref=[_coexistence(q["eos"], q["T_over_Tc"])[0 if q["kind"] == "droplet" else 1] for q in reqs])


def _kept(c, ref, f):
    """The fields as the program keeps them: doubles of an FP64 solve, floats of an FP32 one."""
    if c["prec"] == 64:
        return {"rho": f[0], "uz": f[1], "ur": f[2], **({"p": f[3]} if len(f) > 3 else {})}
    return {"drho": (f[0] - ref).float(), "uz": f[1].float(), "ur": f[2].float(), **({"p": f[3].float()} if len(f) > 3 else {})}


_GROUP = 32  # solves of a batch whose fields are joined into one output


def run(state):
    c = state["c"]
    if c["kind"] == "solve":
        s, out = state["s"], state["out"]
        s.step(c["steps"])
        lbm.lbm_axi_moments_device(s.h, rho=out[0], u_z=out[1], u_r=out[2], p=out[3])
        return _kept(c, state["ref"], out)
    if c["kind"] == "batch":
        state["batch"].step(c["steps"])
        for s, out in zip(state["s"], state["out"]):
            lbm.lbm_axi_moments_device(s.h, rho=out[0], u_z=out[1], u_r=out[2])
        got = []
        for i in range(0, c["n"], _GROUP):
            fs = [_kept(c, r, o) for r, o in zip(state["ref"][i:i + _GROUP], state["out"][i:i + _GROUP])]
            got.append({k: torch.cat([f[k].reshape(-1) for f in fs]) for k in fs[0]})
        return got
    if c["kind"] == "start":
        s, out = state["s"], state["out"]
        lbm.lbm_axi_init_physical_device(s.h, state["rho"], *state["u"])
        lbm.lbm_axi_moments_device(s.h, rho=out[0], u_z=out[1], u_r=out[2], p=out[3])
        m = min(c["nz"], c["nr"])
        mass = lbm.lbm_axi_mass(s.h)
        dp = lbm.lbm_axi_pressure_jump(s.h, c["nz"] / 2.0, 0.0, 0.12 * m, 0.4 * m)
        return {"f": _kept(c, state["ref"], out), "mass_rw": mass[0], "mass": mass[1], "dp": dp}
    results, _ = srv.serve(state["reqs"], precision=c["prec"], keep_rho=True)
    by = {r.id: r for r in results}
    return [(by[q["id"]].rho - ref).astype(np.float32) for q, ref in zip(state["reqs"], state["ref"])]


def _flops(c):
    """Additions and multiplications of one node's step, counted on the formulas (a division or root as one)."""
    return 360 if c.get("axis", 1) else 240


def work(case):
    c, es = case, case["prec"] // 8
    if c["kind"] == "solve":
        n = c["nz"] * c["nr"]
        return {"bytes": n * (18 * es * c["steps"] + 4 * 8), "flops": n * c["steps"] * _flops(c)}
    if c["kind"] == "batch":
        n = sum(b["nz"] * b["nr"] for b in _batch_cases(c))
        return {"bytes": n * (18 * es * c["steps"] + 3 * 8), "flops": n * c["steps"] * _flops(c)}
    if c["kind"] == "start":
        n = c["nz"] * c["nr"]  # density and velocity in, populations out, four fields out
        return {"bytes": n * (3 * 8 + 9 * es + 4 * 8), "flops": n * 200}
    q = _requests(c, 0)
    return {"bytes": sum(r["nz"] * r["nr"] * (18 * es * r["steps"] + 16) for r in q),
            "flops": sum(r["nz"] * r["nr"] * r["steps"] * _flops(c) for r in q)}


# ------------------------------------------------------ the method in 64 bits --

_CZ = [0, 1, -1, 0, 0, 1, -1, 1, -1]
_CR = [0, 0, 0, 1, -1, 1, -1, -1, 1]
_W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


def _dir(cz, cr):
    return [i for i in range(9) if _CZ[i] == cz and _CR[i] == cr][0]


class _Exact:
    """The update on whole fields; the state is the set of populations as they arrive (before the collision)."""

    def __init__(self, c):
        self.c, self.T = c, _T(c["eos"], c["T"])
        self.per = c["top"] == "periodic"
        self.r = (torch.arange(c["nr"], dtype=torch.float64, device=DEV) + 0.5)[:, None]

    def ext(self, a, n, sa, st):
        if self.per:
            return torch.cat([a[-n:], a, a[:n]])
        return torch.cat([sa * a[:n].flip(0), a, st * a[-n:].flip(0)])

    def deriv(self, a, sa, st):
        """Both derivatives by the isotropic (8, -1)/36 stencil; sa, st: parity at the axis and the top wall."""
        e, n = self.ext(a, 2, sa, st), a.shape[0]

        def at(m, dr, dz):
            return torch.roll(e[2 + m * dr:2 + m * dr + n], -m * dz, 1)

        out = []
        for along in (lambda s, t: (s, t), lambda s, t: (t, s)):  # (dz, dr)
            d = 0.0
            for m, w in ((1, 8.0), (2, -1.0)):
                for t in (-1, 0, 1):
                    z, r = along(1, t)
                    d = d + w * (at(m, r, z) - at(m, -r if along(1, 0)[1] else r, -z if along(1, 0)[0] else z))
            out.append(d / 36.0)
        return out

    def kup(self, psi):
        e, n = self.ext(psi, 1, 1, 1), psi.shape[0]
        s = [0.0, 0.0, 0.0, 0.0]
        for i in range(1, 9):
            v = torch.roll(e[1 + _CR[i]:1 + _CR[i] + n], -_CZ[i], 1)
            for q, x in ((0, v), (2, v * v)):
                s[q] = s[q] + _W[i] * _CZ[i] * x
                s[q + 1] = s[q + 1] + _W[i] * _CR[i] * x
        A = self.c["A"]
        return tuple(6 * (A * s[2 + k] + (1 - 2 * A) * psi * s[k]) for k in (0, 1))

    def force(self, rho):
        c = self.c
        psi = torch.sqrt(rho / 3 - _p(c["eos"], self.T, rho))
        fz, fr = self.kup(psi)
        if c["axis"]:
            pz, pr = self.deriv(psi, 1, 1)
            prr, prz = self.deriv(pr, -1, -1)[1], self.deriv(pz, 1, 1)[1]
            k = torch.full_like(rho, 1 / 9) if c["kappa"] == "lattice" else _dp(c["eos"], self.T, rho) ** 2
            a = c["axis_a"] * c["A"] / self.r * pr
            fz = fz + 3 * k * (psi * prz / self.r + a * pz)
            fr = fr + 3 * k * (psi * (prr - pr / self.r) / self.r + a * pr)
        return fz, fr

    def moments(self, g):
        rho = sum(g)
        jz = sum(_CZ[i] * g[i] for i in range(9) if _CZ[i])
        jr = sum(_CR[i] * g[i] for i in range(9) if _CR[i])
        fz, fr = self.force(rho)
        return rho, jz, jr, fz, fr, (jz + 0.5 * fz) / rho, (jr + 0.5 * fr) / rho

    @staticmethod
    def feq(rho, uz, ur):
        sq = uz * uz + ur * ur
        out = []
        for i in range(9):
            cu = _CZ[i] * uz + _CR[i] * ur
            out.append(_W[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * sq))
        return out

    def start(self, rho, u=(0.0, 0.0)):
        fz, fr = self.force(rho)
        return self.feq(rho, u[0] - 0.5 * fz / rho, u[1] - 0.5 * fr / rho)

    def step(self, g):
        c = self.c
        om = 1.0 / c["tau"]
        rho, jz, jr, fz, fr, uz, ur = self.moments(g)
        u0z, u0r = jz / rho, jr / rho
        if c["forcing"] == "guo":
            eq = self.feq(rho, uz, ur)
            S = []
            for i in range(9):
                cu, cF = _CZ[i] * uz + _CR[i] * ur, _CZ[i] * fz + _CR[i] * fr
                S.append(_W[i] * (1 - 0.5 * om) * (3 * (cF - uz * fz - ur * fr) + 9 * cu * cF))
        else:
            eq, e1 = self.feq(rho, u0z, u0r), self.feq(rho, u0z + fz / rho, u0r + fr / rho)
            S = [b - a for a, b in zip(eq, e1)]
        f = [g[i] + om * (eq[i] - g[i]) + S[i] for i in range(9)]
        if c["axis"]:
            top = -1 if c["top"] == "noslip" else 1
            duz_dr = self.deriv(uz, 1, top)[1]
            dur_dz, dur_dr = self.deriv(ur, -1, -1)
            mu = rho * (c["tau"] - 0.5) / 3
            Hz = (mu * (duz_dr + dur_dz) - rho * ur * uz) / self.r
            Hr = (2 * mu * (dur_dr - ur / self.r) - rho * ur * ur) / self.r
            m0 = -rho * ur / self.r
            f = [f[i] + _W[i] * (m0 + 3 * (_CZ[i] * Hz + _CR[i] * Hr)) for i in range(9)]
        new = []
        for i in range(9):
            cz, cr = _CZ[i], _CR[i]
            a = torch.roll(f[i], cz, 1)
            if cr:
                a = torch.roll(a, cr, 0)
                if not self.per:
                    if cr > 0:
                        a[0] = torch.roll(f[_dir(cz, -1)][0], cz)
                    elif c["top"] == "noslip":
                        a[-1] = f[_dir(-cz, 1)][-1]
                    else:
                        a[-1] = torch.roll(f[_dir(cz, 1)][-1], cz)
            new.append(a)
        return new

    def fields(self, g):
        rho, _, _, _, _, uz, ur = self.moments(g)
        return rho, uz, ur, _p(self.c["eos"], self.T, rho)


def _exact_fields(c, rho, steps, u=(0.0, 0.0)):
    m = _Exact(c)
    g = m.start(rho, u)
    for _ in range(steps):
        g = m.step(g)
    return m.fields(g)


def _exact_kept(c, ref, f):
    first = {"rho": f[0]} if c["prec"] == 64 else {"drho": f[0] - ref}
    return {**first, "uz": f[1], "ur": f[2], **({"p": f[3]} if len(f) > 3 else {})}


def exact(case, seed):
    c = case
    if c["kind"] == "solve":
        rho, ref = _density(c, seed)
        return _exact_kept(c, ref, _exact_fields(c, rho, c["steps"], _axial(c["nz"], c["nr"]) if c["field"] == "ring" else (0.0, 0.0)))
    if c["kind"] == "batch":  # the first group only: every solve would take minutes
        fs = []
        for i, b in enumerate(_batch_cases(c)[:_GROUP]):
            rho, ref = _density(b, int(seed) * 1000 + i)
            fs.append(_exact_kept(b, ref, _exact_fields(b, rho, c["steps"])[:3]))
        rest = -(-c["n"] // _GROUP) - 1
        return [{k: torch.cat([f[k].reshape(-1) for f in fs]) for k in fs[0]}] + [None] * rest
    if c["kind"] == "start":
        full = _start_solve(c)
        rho, ref = _density(full, seed)
        f = _exact_fields(full, rho, 0, _flow(c["nz"], c["nr"], seed))
        m = min(c["nz"], c["nr"])
        Z, R = _grid(c["nz"], c["nr"])
        d = torch.sqrt((Z - c["nz"] / 2.0) ** 2 + R * R)
        dp = f[3][d < 0.12 * m].mean() - f[3][d > 0.4 * m].mean()
        return {"f": _exact_kept(full, ref, f), "mass_rw": float((R * f[0]).sum()), "mass": float(f[0].sum()), "dp": float(dp)}
    out = []
    for q in _requests(c, seed):
        rho, ref = _request_density(q)
        full = _solve("", q["kind"], q["nz"], q["nr"], q["steps"], eos=q["eos"], T=q["T_over_Tc"], tau=srv.TAU)
        out.append(_exact_fields(full, torch.from_numpy(rho).to(DEV), q["steps"])[0] - ref)
    return out
