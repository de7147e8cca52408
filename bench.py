#!/usr/bin/env python3
"""Throughput of the axisymmetric multiphase D2Q9 update on one GB300.

Workload (default): the FP32 propagating density wave on a 4096 (z) x 2048 (r)
lattice -- Carnahan-Starling EOS (a = 1, b = 4, R = 1) at T = 0.9 T_c on the
liquid branch (rho0 = coexistence liquid density), A = -0.152, tau = 0.6,
rho = rho0 (1 + 0.01 sin(2 pi z / nz)) + U(-1e-4, 1e-4) (PCG64 seed 20151201),
u = 0, free-slip top, specular axis, periodic z.  One step = one time step of
the whole lattice, which the fused kernel does in one launch (gather, moments,
psi, forces, EDM, axisymmetric source, collision).  Metric: MLUPS (million
lattice-node updates per second).

`python bench.py --gpus N --steps K --warmup W` prints one JSON line.  Under
torchrun each rank runs an independent replica (the solves share nothing), so
scaling is weak and value = all nodes updated / max rank time.
`--impl reference` times the FP64 CPU oracle on a bounded window of the same
workload instead.
"""
import argparse
import glob
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

NZ, NR, TAU, A, T_OVER_TC = 4096, 2048, 0.6, -0.152, 0.9
# Algorithmic bytes per node and time step, FP32.  The fused kernel (the default path) reads and
# writes the 9 populations: 72 B, its roofline figure.  The two-kernel form of the step reads 9
# populations and writes rho, j_z, j_r, psi (52 B), then reads 9 populations and the 4 fields and
# writes 9 populations (88 B): 140 B, reported beside it as the equivalent two-kernel traffic.
BYTES_STEP = 140
BYTES_FUSED = 72
BYTES_B = 88
WORKLOAD = "density wave 4096x2048, CS T=0.9Tc, tau=0.6, A=-0.152, FP32 deviation storage"


def _args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-blocks", dest="blocks", action="store_false",
                    help="wave: leave out the bounded batched and served blocks of the default line")
    ap.add_argument("--workload", default="wave", choices=["wave", "batched", "served"],
                    help="wave: the 4096x2048 density wave (headline); batched: 256 uneven droplets in one "
                         "launch per step vs one solve at a time; served: Poisson request stream with "
                         "continuous batching vs a one-at-a-time server")
    ap.add_argument("--requests", type=int, default=48, help="served: requests per arrival rate")
    ap.add_argument("--budget-mb", type=int, default=4096, help="served: HBM admission budget")
    ap.add_argument("--grid", default="%dx%d" % (NZ, NR),
                    help="wave: nz x nr of the wave (the default is the headline workload; other sizes are "
                         "for profiling)")
    ap.add_argument("--path", default="fused", choices=["fused", "split"],
                    help="wave: the single-pass kernel (default) or the two-kernel path")
    args = ap.parse_args()
    _set_grid(args.grid)
    return args


def _set_grid(spec):
    global NZ, NR, WORKLOAD
    nz, nr = (int(x) for x in spec.lower().split("x"))
    if (nz, nr) != (NZ, NR):
        NZ, NR = nz, nr
        WORKLOAD = "density wave %dx%d, CS T=0.9Tc, tau=0.6, A=-0.152, FP32 deviation storage" % (NZ, NR)


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def _peaks():
    """Measured HBM copy bandwidth (GB/s) from MEASURED_PEAKS.json, else the fallback."""
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            data = json.load(fh)

        def find(d):
            if isinstance(d, dict):
                for k, v in d.items():
                    if isinstance(v, (int, float)) and "hbm" in k.lower() and "gb" in k.lower():
                        return float(v)
                for v in d.values():
                    r = find(v)
                    if r:
                        return r
            return None

        v = find(data)
        if v:
            return v, "measured"
    except (OSError, ValueError):
        pass
    return 6800.0, "fallback"


def _source_hash():
    h = hashlib.sha256()
    for fn in sorted(glob.glob(os.path.join(ROOT, "paper_1512_01977_gb300", "csrc", "*"))):
        with open(fn, "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


# What the kernels of a step's main launch do (the names of lbm.lbm_axi_step_kernels).
_KERNELS = {"k_step_warp": "one-pass gather+psi+forces+EDM+source+collide, one warp per strip",
            "k_tile": "one-pass gather+psi+forces+EDM+source+collide over tiles held in shared memory",
            "k_step": "one-pass gather+psi+forces+EDM+source+collide by CTAs marching fixed row chunks",
            "k_phase_l": "gather+psi, forces+u, source+EDM+collide, one launch each",
            "k_density": "forces+EDM+source+collide, after k_density"}


def _step_form(kernels):
    """(roofline label, launches per step, algorithmic bytes per node of what is timed) of a step of these kernels: the
    whole step, whose populations are read and written once, or kernel (b) of the split path."""
    split = kernels[0] == "k_density"
    name = "k_update" if split else " + ".join(kernels)
    return "%s (%s)" % (name, _KERNELS[kernels[0]]), len(kernels), BYTES_B if split else BYTES_FUSED


def _ncu_traffic(kernels):
    """Per-launch DRAM bytes of k_step_warp on the default grid from the committed ncu
    summary, or None for another kernel or grid and when the kernel sources changed since."""
    if kernels != ["k_step_warp"] or (NZ, NR) != (4096, 2048):
        return None
    path = os.path.join(ROOT, "profiles", "k_step_warp_fp32_wave4096x2048.md")
    try:
        vals = {}
        with open(path) as fh:
            for line in fh:
                if ":" in line and line.strip().startswith("- "):
                    k, v = line.strip()[2:].split(":", 1)
                    vals[k.strip()] = v.strip().strip("`")
        if vals.get("source_sha") == _source_hash():
            return int(float(vals["dram_bytes_per_launch"]))
    except (OSError, KeyError, ValueError):
        pass
    return None


class ClockSampler:
    """SM clocks, power and clock-event (throttle) reasons of the bench's GPU,
    read (never set) through NVML every `period` seconds from a background
    thread; nvidia-smi polling is the fallback when NVML cannot be loaded.
    Samples are tagged with the phase the caller marks (e.g. the timed region)."""

    NAMES = {0x4: "sw_power_cap", 0x8: "hw_slowdown", 0x20: "sw_thermal_slowdown", 0x40: "hw_thermal_slowdown",
             0x80: "hw_power_brake_slowdown"}

    def __init__(self, device_index, period=0.002):
        import threading

        self.period = period
        self.samples = []  # (phase, sm_mhz, sm_max_mhz, power_w, reasons bitmask)
        self.phase = "idle"
        self._stop = threading.Event()
        self._thread = None
        self._nvml = None
        self._dev = None
        self.source = None
        self._open_nvml(device_index)

    def _open_nvml(self, device_index):
        import ctypes as C

        try:
            import torch

            nv = C.CDLL("libnvidia-ml.so.1")
            if nv.nvmlInit_v2() != 0:
                return
            dev = C.c_void_p()
            props = torch.cuda.get_device_properties(device_index)
            ok = False
            uid = str(getattr(props, "uuid", "") or "")
            for cand in (uid, "GPU-" + uid):
                if uid and nv.nvmlDeviceGetHandleByUUID(cand.encode(), C.byref(dev)) == 0:
                    ok = True
                    break
            if not ok and hasattr(props, "pci_bus_id"):
                bus = "%08x:%02x:%02x.0" % (getattr(props, "pci_domain_id", 0), props.pci_bus_id,
                                            getattr(props, "pci_device_id", 0))
                ok = nv.nvmlDeviceGetHandleByPciBusId_v2(bus.encode(), C.byref(dev)) == 0
            if ok:
                self._nvml, self._dev, self.source = nv, dev, "nvml"
        except (OSError, AttributeError, ImportError):
            self._nvml = None

    def _read_nvml(self):
        import ctypes as C

        nv, dev = self._nvml, self._dev
        sm, smax, mw, rs = C.c_uint(), C.c_uint(), C.c_uint(), C.c_ulonglong()
        if nv.nvmlDeviceGetClockInfo(dev, 1, C.byref(sm)) != 0:
            return None
        nv.nvmlDeviceGetMaxClockInfo(dev, 1, C.byref(smax))
        nv.nvmlDeviceGetPowerUsage(dev, C.byref(mw))
        fn = getattr(nv, "nvmlDeviceGetCurrentClocksEventReasons", None) or \
            getattr(nv, "nvmlDeviceGetCurrentClocksThrottleReasons")
        fn(dev, C.byref(rs))
        return float(sm.value), float(smax.value), mw.value / 1000.0, int(rs.value)

    def _loop(self):
        while not self._stop.is_set():
            r = self._read_nvml()
            if r is not None:
                self.samples.append((self.phase,) + r)
            self._stop.wait(self.period)

    def __enter__(self):
        import threading

        if self._nvml is not None:
            self._thread = threading.Thread(target=self._loop, daemon=True)
            self._thread.start()
        return self

    def __exit__(self, *exc):
        self._stop.set()
        if self._thread is not None:
            self._thread.join(timeout=5)

    def mark(self, phase):
        self.phase = phase
        if self._nvml is not None:  # one sample at every phase change
            r = self._read_nvml()
            if r is not None:
                self.samples.append((phase,) + r)

    def summary(self, phases):
        rows = [x for x in self.samples if x[0] in phases]
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0, "source": self.source}
        reasons = set()
        for x in rows:
            for bit, name in self.NAMES.items():
                if x[4] & bit:
                    reasons.add(name)
        return {"sm_mhz": statistics.median(x[1] for x in rows), "sm_max_mhz": max(x[2] for x in rows),
                "power_w_max": max(x[3] for x in rows), "reasons": sorted(reasons), "samples": len(rows),
                "source": self.source}


def _wave_fields(nz, nr, rho0):
    from paper_1512_01977_gb300 import inputs as I

    return I.density_wave(nz, nr, rho0, amp=0.01, noise=1e-4, seed=20151201)


def _oracle_rate(nz, nr, rho0, steps, threads):
    """Node updates per second of the FP64 oracle, as it stands, on an nz x nr
    window of the workload (OpenMP timing build; `threads` host threads)."""
    import oracle as O
    from oracle import core

    p = O.make_params(nz, nr, TAU, O.EOS_CS, T_OVER_TC, A=A, top=O.TOP_FREESLIP)
    o = O.Oracle(p, omp=True).init(*_wave_fields(nz, nr, rho0))
    used = core.threads(threads)
    o.step(1)  # first touch of the work arrays
    t0 = time.perf_counter()
    o.step(steps)
    dt = time.perf_counter() - t0
    return nz * nr * steps / dt, used, dt


def _cpu_baseline(rho0):
    """The FP64 oracle timed on this host: all cores and one core, on a
    bounded sample of the workload (the full grid for a number of steps,
    about 10 s of wall time in all)."""
    n_all = os.cpu_count() or 1
    steps_all, steps_one = 20, 5
    r_all, used_all, dt_all = _oracle_rate(NZ, NR, rho0, steps_all, n_all)
    r_one, _, dt_one = _oracle_rate(NZ, NR, rho0, steps_one, 1)
    from oracle import core

    core.threads(n_all)
    return {"value": r_all / 1e6, "unit": "MLUPS", "cores": used_all, "kind": "oracle",
            "sample": "%d steps of the full %dx%d grid, FP64, OpenMP over %d threads (%.1f s)"
                      % (steps_all, NZ, NR, used_all, dt_all),
            "nproc": n_all,
            "one_core": {"value": r_one / 1e6, "unit": "MLUPS", "cores": 1,
                         "sample": "%d steps of the full grid, one thread (%.1f s)" % (steps_one, dt_one)}}


def run_reference(args):
    """Reference arm: the FP64 CPU oracle, as it stands, on all host cores, on
    a window of the workload sized so the K timed steps stay bounded."""
    ws, rank, _ = _dist()
    if rank != 0:
        return
    import oracle as O

    # each step a sample: the full grid for K <= 20, smaller windows (same
    # aspect, same recipe) for longer runs, so the run stays within ~a minute
    scale = min(1.0, 20.0 / max(1, args.steps))
    nz = max(64, int(NZ * scale ** 0.5) // 32 * 32)
    nr = max(32, int(NR * scale ** 0.5) // 32 * 32)
    p = O.make_params(nz, nr, TAU, O.EOS_CS, T_OVER_TC, A=A, top=O.TOP_FREESLIP)
    rho0 = O.eos.maxwell_densities(p)[1]
    n_all = os.cpu_count() or 1
    from oracle import core

    o = O.Oracle(p, omp=True).init(*_wave_fields(nz, nr, rho0))
    used = core.threads(n_all)
    o.step(max(1, args.warmup))
    t0 = time.perf_counter()
    o.step(args.steps)
    dt = time.perf_counter() - t0
    v = nz * nr * args.steps / dt / 1e6
    sample = ("%dx%d window of the workload (same EOS, tau, A, wave recipe), FP64, OpenMP over %d threads"
              % (nz, nr, used))
    print(json.dumps({
        "impl": "reference", "metric": "MLUPS", "value": v, "unit": "MLUPS", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1e3 / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD + " (oracle window %dx%d)" % (nz, nr), "nz": nz, "nr": nr},
        "cpu_baseline": {"value": v, "unit": "MLUPS", "cores": used, "kind": "oracle", "sample": sample},
        "e2e": {"value": v, "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


def run_ours(args):
    import ctypes as C

    import numpy as np
    import torch

    import __graft_entry__
    from paper_1512_01977_gb300 import lbm

    from paper_1512_01977_gb300 import replicas

    ws, rank, local = _dist()
    torch.cuda.set_device(local)
    rep = replicas.Replicas(device=torch.device("cuda", local))
    __graft_entry__.build()

    eos = lbm.make_eos(lbm.EOS_CS, T_OVER_TC)
    rho0 = lbm.lbm_eos_coexistence(eos)[1]
    fields = _wave_fields(NZ, NR, rho0)
    n = NZ * NR
    # pinned host copies of the inputs and outputs (the e2e leg copies through them)
    pin = lambda: torch.empty(n, dtype=torch.float64, pin_memory=True).numpy()
    h_in = [pin() for _ in range(3)]
    for dst, src in zip(h_in, fields):
        dst[:] = src.reshape(-1)
    h_out = [pin() for _ in range(4)]

    stream = torch.cuda.Stream()
    s = lbm.Solver(NZ, NR, TAU, eos=eos, A=A, precision=32, rho_ref=rho0, stream=stream.cuda_stream)
    if args.path == "split":
        lbm.lbm_axi_set_tuning(s.h, lbm.PATH_SPLIT, 0)
    s.init(*h_in)
    lbm.lbm_axi_step(s.h, args.warmup)

    def barrier():
        rep.barrier()

    # ---- device-timed throughput: K steps, inputs resident in HBM
    props = torch.cuda.get_device_properties(local)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    clk = ClockSampler(local)
    with clk:
        barrier()
        clk.mark("timed")
        e0.record(stream)
        lbm.lbm_axi_step_async(s.h, args.steps)
        e1.record(stream)
        e1.synchronize()
        clk.mark("after")
        lbm.lbm_axi_sync(s.h)
        barrier()
        # a clock window: the same step loop for at least 0.5 s after the timed
        # region (not part of any figure), so that the clock record holds enough
        # samples even when the timed region lasts a few milliseconds
        clk.mark("window")
        w0 = time.perf_counter()
        n_window = 0
        while time.perf_counter() - w0 < 0.5:
            lbm.lbm_axi_step(s.h, 200)
            n_window += 200
        clk.mark("done")
    ms = e0.elapsed_time(e1)
    ms_max = rep.max(ms)
    value = replicas.aggregate_rate(n * args.steps, ws, ms_max * 1e-3) / 1e6  # MLUPS

    # ---- per-kernel device time (CUDA events around each launch, same stream)
    path, rows_per_cta = lbm.lbm_axi_get_tuning(s.h)
    kr = max(20, min(args.steps, 1000))
    ms_a, ms_b = lbm.lbm_axi_time_kernels(s.h, kr)
    t_a, t_b = ms_a / kr * 1e-3, ms_b / kr * 1e-3
    t_iso = t_b  # one launch bracketed by its own events
    t_step = ms * 1e-3 / args.steps
    if path == lbm.PATH_FUSED:
        # the timed region ran the step's kernels alone: their average duration per step
        # over that region is the region's time per step
        t_a, t_b = 0.0, t_step
    kernels = lbm.lbm_axi_step_kernels(s.h)
    label, per_step, bytes_main = _step_form(kernels)
    peak, peak_kind = _peaks()
    ach_b = bytes_main * n / t_b / 1e9
    traffic = _ncu_traffic(kernels)

    # ---- end to end through the C ABI: pinned host -> init -> K steps -> moments -> pinned host
    barrier()
    w0 = time.perf_counter()
    lbm.lbm_axi_init(s.h, NZ, NR, *h_in)
    lbm.lbm_axi_step(s.h, args.steps)
    ptr = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))
    rc = lbm.lib().lbm_axi_moments(s.h, *[ptr(a) for a in h_out])
    if rc != 0:
        raise lbm.LbmError(rc, "lbm_axi_moments")
    barrier()
    wall = time.perf_counter() - w0
    e2e = replicas.aggregate_rate(n * args.steps, ws, rep.max(wall)) / 1e6
    mass_rw, _ = s.mass()
    s.close()

    pop_mb = int(round(9 * n * 4 / 1e6))
    extra = {}
    if ws == 1 and args.blocks:
        # the batched and served workloads, bounded, on the same GPU after the headline
        extra["batched"] = _batched_block(steps=1000, warmup=3)
        extra["served"] = _served_block(rates=(100,), requests=24, budget_mb=4096)
    if rank == 0:
        cpu = None
        if ws == 1 and not args.no_cpu_baseline:
            cpu = _cpu_baseline(rho0)
        timed = clk.summary({"timed", "after"})
        window = clk.summary({"window"})
        clocks = dict(timed if timed["samples"] >= 3 else window)
        clocks.update({"samples_timed_region": timed["samples"], "samples_window": window["samples"],
                       "window": "%d more steps of the same loop right after the timed region" % n_window,
                       "reasons_window": window["reasons"], "sm_mhz_window": window["sm_mhz"]})
        out = {
            "metric": "MLUPS", "value": value, "unit": "MLUPS", "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_max / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": WORKLOAD, "nz": NZ, "nr": NR, "nodes": n, "replicas": ws,
                       "l2": ("no flush: inputs larger than L2 (2 x %d MB FP32 population buffers)" % pop_mb)
                       if 2 * pop_mb > 129 else "inputs smaller than L2 (%d MB): not an HBM measurement" % (2 * pop_mb),
                       "parallelism": "replicas only (independent solves per GPU)",
                       "device": props.name},
            "roofline": {"bound": "hbm",
                         "kernel": label,
                         "achieved": ach_b, "peak": peak, "unit": "GB/s", "frac": ach_b / peak,
                         "peak_source": peak_kind, "traffic": traffic,
                         "algorithmic_bytes_per_node": bytes_main,
                         "traffic_bytes_per_node": traffic / n if traffic else None,
                         "avg_launch_us": t_b * 1e6 / (per_step if path == lbm.PATH_FUSED else 1),
                         "avg_launch_source": "timed region / launches" if path == lbm.PATH_FUSED
                         else "CUDA events around each launch",
                         "isolated_launch_us": t_iso * 1e6,
                         "launches_per_step": per_step,
                         "frac_of_nominal_7900_gbs": ach_b / 7900.0,
                         "two_kernel_equivalent": {
                             "bytes_per_node": BYTES_STEP,
                             "frac": BYTES_STEP * n / t_step / 1e9 / peak,
                             "note": "the traffic the two-kernel form of the step would need at this step time"},
                         "rows_per_cta": rows_per_cta},
            "e2e": {"value": e2e, "unit": "MLUPS", "steps": args.steps, "h2d_bytes_per_step": 3 * 8 * n / args.steps,
                    "d2h_bytes_per_step": 4 * 8 * n / args.steps,
                    "note": "one solve: init from pinned host fields, K steps, moments back to pinned host; "
                            "the copies are fixed per run, so the rate rises with K"},
            "gpu_launches": per_step * args.steps,
            "clocks": clocks,
            "mass_rweighted": mass_rw,
        }
        out.update(extra)
        if cpu is not None:
            out["cpu_baseline"] = cpu
        print(json.dumps(out))
    rep.close()


def _batched_block(steps, warmup, trials=3):
    """256 independent droplets (sizes log-uniform 64x32 .. 512x256, R = 0.25 of
    the shorter side, T/Tc ~ U[0.5, 0.85], tau ~ U[0.6, 1.0], CS, FP32 with
    deviations about rho_v, started at rest), `steps` steps each: one batched
    launch per step (autotuned) against the same solves stepped one at a time.
    Only solves that finish every step are credited, in both arms."""
    import torch

    from paper_1512_01977_gb300 import inputs as I
    from paper_1512_01977_gb300 import lbm

    specs = I.batch_droplets(n=256, seed=4)

    def make():
        out = []
        for sp in specs:
            eos = lbm.make_eos(lbm.EOS_CS, sp["T_over_Tc"])
            rv, rl = lbm.lbm_eos_coexistence(eos)
            s = lbm.Solver(sp["nz"], sp["nr"], sp["tau"], eos=eos, A=A, precision=32, rho_ref=rv)
            s.init(*I.droplet(sp["nz"], sp["nr"], sp["R"], rl, rv), physical=True)  # at rest
            out.append(s)
        return out

    nodes = sum(sp["nz"] * sp["nr"] for sp in specs)
    # one at a time: each solve's own CUDA-graph step loop
    solvers = make()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    ok_seq = []
    for s in solvers:
        try:
            s.step(steps)
            ok_seq.append(True)
        except lbm.LbmError:
            ok_seq.append(False)
    torch.cuda.synchronize()
    t_seq = time.perf_counter() - t0
    for s in solvers:
        s.close()
    # batched
    solvers = make()
    b = lbm.Batch(solvers)
    tuning = b.autotune(trials=trials)
    b.step(warmup)
    torch.cuda.synchronize()
    w0 = time.perf_counter()
    b.step_async(steps)
    b.sync()
    t_batch = time.perf_counter() - w0
    status = b.status()
    b.close()
    for s in solvers:
        s.close()
    nodes_ok = sum(sp["nz"] * sp["nr"] for sp, st in zip(specs, status) if st == lbm.OK)
    nodes_ok_seq = sum(sp["nz"] * sp["nr"] for sp, ok in zip(specs, ok_seq) if ok)
    value = nodes_ok * steps / t_batch / 1e6
    seq = nodes_ok_seq * steps / t_seq / 1e6
    return {"value": value, "unit": "MLUPS", "steps": steps, "warmup": warmup, "wall_s": t_batch,
            "workload": "256 droplets, log-uniform 64x32..512x256, CS, T/Tc 0.5..0.85, tau 0.6..1.0, "
                        "FP32, started at rest; one launch per step (CUDA graph)",
            "solves": 256, "nodes": nodes, "nodes_completed": nodes_ok, "tuning_strip_grid": list(tuning),
            "failed": sum(1 for x in status if x != lbm.OK),
            "credit": "node-steps of solves that finished every step",
            "one_at_a_time": {"value": seq, "unit": "MLUPS", "wall_s": t_seq, "failed": ok_seq.count(False)},
            "speedup_vs_one_at_a_time": value / seq if seq > 0 else None,
            "timing": "host wall clock around the step loop, synchronised on both sides"}


def _served_block(rates, requests, budget_mb):
    """Poisson request streams: continuous batching vs one request at a time;
    p50 / p99 latency and MLUPS per rate."""
    from paper_1512_01977_gb300 import inputs as I
    from paper_1512_01977_gb300 import serve

    rows = []
    for rate in rates:
        reqs = I.request_stream(rate, requests, seed=5)
        _, st = serve.serve(reqs, budget_bytes=budget_mb << 20)
        _, sq = serve.serve_sequential(reqs)
        rows.append({"rate_per_s": rate, "batched": st, "one_at_a_time": sq})
    return {"workload": "served Poisson stream, droplets + waves, CS/vdW, T/Tc 0.5..0.9, grids 32x32..1024x512, "
                        "1k..20k steps", "requests_per_rate": requests, "budget_mb": budget_mb, "rates": rows}


def run_batched(args):
    import torch

    import __graft_entry__

    ws, rank, local = _dist()
    torch.cuda.set_device(local)
    __graft_entry__.build()
    blk = _batched_block(args.steps, args.warmup)
    print(json.dumps({
        "metric": "MLUPS", "value": blk["value"], "unit": "MLUPS", "n_gpus": 1, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": blk["wall_s"] * 1e3 / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": blk["workload"], "solves": 256, "nodes": blk["nodes"],
                   "nodes_completed": blk["nodes_completed"], "tuning_strip_grid": blk["tuning_strip_grid"],
                   "credit": blk["credit"]},
        "one_at_a_time": blk["one_at_a_time"], "speedup_vs_one_at_a_time": blk["speedup_vs_one_at_a_time"],
        "failed": blk["failed"], "gpu_launches": args.steps,
    }))


def run_served(args):
    import torch

    import __graft_entry__

    ws, rank, local = _dist()
    torch.cuda.set_device(local)
    __graft_entry__.build()
    blk = _served_block((10, 30, 100, 300, 1000), args.requests, args.budget_mb)
    best = max(r["batched"]["mlups"] for r in blk["rates"])
    print(json.dumps({
        "metric": "MLUPS", "value": best, "unit": "MLUPS", "n_gpus": 1, "steps": None, "warmup": 0,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": blk["workload"], "requests_per_rate": args.requests, "budget_mb": args.budget_mb},
        "rates": blk["rates"],
    }))


def main():
    args = _args()
    if args.impl == "reference":
        run_reference(args)
    elif args.workload == "batched":
        run_batched(args)
    elif args.workload == "served":
        run_served(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
