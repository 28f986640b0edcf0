"""Benchmark of the eMG V-cycle on the 128 x 64 cylinder O-grid at p = 4 (one GB300).

A step is one FAS V-cycle p = 4 -> 0 -> 4 (every hot-path kernel: residuals, exact
block assembly, batched LU, PRK stages, transfers, p = 0 Jacobian, Arnoldi, phi_1).
`value` is the V-cycle throughput of the mixed form (PRK blocks in FP32; residual,
Arnoldi and phi_1 in FP64) in GDoF/s: K = 5 N_4 E degrees of freedom per cycle over the
time per cycle, inputs resident in HBM.  The plain FP64 form is measured beside it.  The
line also carries the DG residual throughput, the wall time to a 1e-10 drop of ||R(rho)||
for both forms, the end-to-end rate through the C ABI with host buffers, the roofline of
the dominant kernel and the CPU oracle timed on a bounded sample.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl emg|reference]
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

WORKLOADS = {
    # the 128 x 64 cylinder O-grid at p = 4 is the timed configuration; the smaller ones
    # serve profiling captures that must stay small
    "cyl128x64_p4": dict(name="cyl128x64_p4", n_theta=128, n_r=64, p_max=4, mach=0.3),
    "cyl64x32_p4": dict(name="cyl64x32_p4", n_theta=64, n_r=32, p_max=4, mach=0.3),
    "cyl32x16_p2": dict(name="cyl32x16_p2", n_theta=32, n_r=16, p_max=2, mach=0.3),
    # small spheres for profiling captures of the 3-D kernels
    "sph6x8x8x8_p4": dict(name="sph6x8x8x8_p4", kind="sphere", n=8, n_r=8, p_max=4, mach=0.3),
    "sph6x8x8x12_p3": dict(name="sph6x8x8x12_p3", kind="sphere", n=8, n_r=12, p_max=3, mach=0.3),
}


def make_mesh(W):
    from workloads import cubed_sphere_shell, ogrid
    if W.get("kind") == "sphere":
        return cubed_sphere_shell(W["n"], W["n_r"])
    return ogrid(W["n_theta"], W["n_r"])
METRIC = "time to 1e-10 residual drop & DG residual GDoF/s: mixed vs FP64, 1 GB300"
# DRAM bytes (read + write) of one k_volume launch at p = 4 on the 128 x 64 O-grid, from an ncu
# capture of this kernel (dram__bytes_read.sum + dram__bytes_write.sum); None once the kernel
# changes until it is captured again.
VOLUME_P4_TRAFFIC = {"cyl128x64_p4": 142.427e6}
PREC_NAMES = {0: "fp64", 1: "fp32_blocks", 2: "bf16_blocks"}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="emg", choices=["emg", "reference"])
    ap.add_argument("--workload", default="cyl128x64_p4", choices=sorted(WORKLOADS))
    ap.add_argument("--prec", default="all", choices=["all", "both", "fp64", "mixed", "bf16"],
                    help="all: the mixed (FP32 blocks) form timed, with the FP64 and BF16-block forms beside it")
    ap.add_argument("--start-seeds", type=int, default=3,
                    help="extra solves of the first form from the free stream perturbed by 1e-13 (relative, "
                         "seeded normal draws): the spread of the cycle count to 1e-10, which rounding decides")
    ap.add_argument("--krylov-f32", type=int, default=-1, choices=[-1, 0, 1],
                    help="Arnoldi process of the EXP1 step in float32 (emg_params.krylov_f32; -1: float32 "
                         "with the float32 block forms)")
    ap.add_argument("--block-kernels", type=int, default=0, choices=[0, 1, 2, 3],
                    help="float32 block kernels: 0 the built-in choice per level, 1 tensor cores, 2 SIMT")
    ap.add_argument("--no-solve", action="store_true", help="skip the time-to-1e-10 solves")
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU oracle baseline")
    ap.add_argument("--serve", action="store_true",
                    help="run the seeded stream of served cylinder solves through the request loop instead")
    ap.add_argument("--serve-requests", type=int, default=64)
    ap.add_argument("--max-active", type=int, default=8)
    ap.add_argument("--stall-cycles", type=int, default=100,
                    help="served solves that set no new residual minimum for this many cycles end early")
    return ap.parse_args()


def max_over_ranks(x, device="cuda"):
    """The largest of every rank's x (the slowest rank sets a replica run's time); x itself
    when no process group is running."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def clocks_dir():
    """Where the raw nvidia-smi samples go (their summary is in the JSON line)."""
    import tempfile
    return os.environ.get("EMG_CLOCKS_DIR") or tempfile.gettempdir()


def dist_info():
    return (int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")),
            int(os.environ.get("LOCAL_RANK", "0")))


def oracle_sample(W, steps, warmup):
    """The oracle's V-cycle (FP64 numpy) on a bounded sample of the workload: the same
    O-grid family and degree at 16 x 8 elements.  Returns (GDoF/s, seconds, E)."""
    from oracle import emg as oemg
    from oracle.dg import DG
    from workloads import cubed_sphere_shell, ogrid
    sample = cubed_sphere_shell(2, 1) if W.get("kind") == "sphere" else ogrid(16, 8)
    dg = DG(sample, W["p_max"], mach=W["mach"])
    u = dg.freestream_state()
    opts = oemg.Options()
    n = 1
    for _ in range(warmup):
        u, _ = oemg.vcycle(dg, u, n, opts)
        n += 1
    t = time.perf_counter()
    for _ in range(steps):
        u, _ = oemg.vcycle(dg, u, n, opts)
        n += 1
    el = time.perf_counter() - t
    K = 5 * dg.N(W["p_max"]) * dg.E
    return K * steps / el / 1e9, el, dg.E


def _one_thread():
    """Pool initializer: one BLAS/OpenMP thread per worker process (one core each)."""
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ[k] = "1"


def _oracle_job(a):
    return oracle_sample(*a)


def oracle_cores(W, steps, warmup, cores):
    """The oracle sample on `cores` host cores at once: one worker process per core (spawned,
    never forked after CUDA), each on its own copy of the sample; the aggregate rate is the
    sum of the workers' rates over their timed loops.  Returns (GDoF/s, wall s, E)."""
    import multiprocessing as mp
    t0 = time.perf_counter()
    with mp.get_context("spawn").Pool(cores, initializer=_one_thread) as pool:
        res = pool.map(_oracle_job, [(W, steps, warmup)] * cores)
    return sum(r[0] for r in res), time.perf_counter() - t0, res[0][2]


def cpu_baseline(W, steps, warmup):
    """The oracle on one core and on every host core (os.cpu_count())."""
    ncores = os.cpu_count() or 1
    v1, el1, E = oracle_cores(W, steps, warmup, 1)
    vall, elall, _ = oracle_cores(W, steps, warmup, ncores)
    sample = (f"{steps} oracle V-cycles (after {warmup} untimed) of the 16x8 O-grid at p={W['p_max']} "
              f"({E} elements) per core")
    return {"value": vall, "unit": "GDoF/s", "cores": ncores, "kind": "oracle", "sample": sample,
            "single_core": {"value": v1, "cores": 1, "wall_s": round(el1, 2)}, "wall_s": round(elall, 2)}


class Clocks:
    """nvidia-smi sampling during the timed region."""

    def __init__(self, idx, path):
        self.path = path
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.f = open(path, "w")
            self.p = subprocess.Popen(["nvidia-smi", f"--id={idx}", f"--query-gpu={q}", "--format=csv,noheader,nounits",
                                       "-lms", "100"], stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.p = None

    def stop(self):
        if self.p is None:
            return None
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except Exception:
            self.p.kill()
        self.f.close()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        try:
            return json.load(open(path)), "measured"
        except Exception:
            pass
    return {}, "fallback"


def run_reference(args, rank, world):
    """The reference arm: the CPU oracle, as it stands, on every host core (one spawned worker
    per core, each on its own copy of the bounded sample; rank 0 only)."""
    if rank != 0:
        return
    W = WORKLOADS[args.workload]
    ncores = os.cpu_count() or 1
    v, el, E = oracle_cores(W, args.steps, args.warmup, ncores)
    sample = (f"{args.steps} oracle V-cycles (after {args.warmup} untimed) of the 16x8 O-grid at p={W['p_max']} "
              f"({E} elements) per core, {ncores} cores")
    line = {
        "impl": "reference", "metric": METRIC, "value": v, "unit": "GDoF/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * el / max(args.steps, 1),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": W["name"], "sample": sample},
        "cpu_baseline": {"value": v, "unit": "GDoF/s", "cores": ncores, "kind": "oracle", "sample": sample},
        "e2e": {"value": v, "unit": "GDoF/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def state_comparison(a, b, W):
    """Converged states of the two forms: the largest difference relative to the largest
    coefficient, and the same for their parts symmetric under the mirror y -> -y of the O-grid
    (alpha = 0: the steady flow is symmetric; the antisymmetric part is the circulation mode
    of the inviscid cylinder, which the residual fixes only weakly and rounding seeds)."""
    import numpy as np
    nt, nr, p = W["n_theta"], W["n_r"], W["p_max"]
    perm = np.array([l * nt + (nt - 1 - k) % nt for l in range(nr) for k in range(nt)])
    ey = np.array([d - x for d in range(p + 1) for x in range(d, -1, -1)])   # y exponent per mode
    sgn = np.array([1.0, 1.0, -1.0, 1.0, 1.0])[:, None] * ((-1.0) ** ey)[None, :]
    sym = lambda u: 0.5 * (u + u[perm] * sgn[None])          # noqa: E731
    den = np.abs(b).max()
    sa, sb = sym(a), sym(b)
    return {"mixed_vs_fp64_converged_relerr": float(np.abs(a - b).max() / den),
            "mixed_vs_fp64_symmetric_part_relerr": float(np.abs(sa - sb).max() / den),
            "antisymmetric_part_rel": {"fp32_blocks": float(np.abs(a - sa).max() / den),
                                       "fp64": float(np.abs(b - sb).max() / den)}}


def kernel_rooflines(prof_cycle, work, peaks, hbm_gbs, form):
    """Achieved rate of each kernel class (algorithmic work of one cycle / its measured time
    per cycle) against the roof that bounds it."""
    out = {}
    alu64, alu32 = peaks["fp64_tflops"], peaks["fp32_tflops"]
    roofs = {"residual_volume": ("alu", alu64), "residual_face_flux": ("alu", alu64),
             "diag_block_assembly": ("alu", alu64 if form == 0 else alu32),
             "block_lu": ("alu", alu64 if form == 0 else alu32),
             "prk_stage_solve": ("hbm", hbm_gbs), "arnoldi": ("hbm", hbm_gbs)}
    for k, (bound, peak) in roofs.items():
        if k not in prof_cycle or k not in work:
            continue
        ms = prof_cycle[k]["ms_per_cycle"]
        if ms <= 0:
            continue
        if bound == "alu":
            ach = work[k][0] / (ms * 1e-3) / 1e12
            out[k] = {"bound": "alu", "achieved": ach, "peak": peak, "unit": "TFLOP/s", "frac": ach / peak,
                      "ms_per_cycle": ms}
        else:
            ach = work[k][1] / (ms * 1e-3) / 1e9
            out[k] = {"bound": "hbm", "achieved": ach, "peak": peak, "unit": "GB/s", "frac": ach / peak,
                      "ms_per_cycle": ms}
    return out


def unit_roofline(ops, seconds, peaks, hbm_gbs):
    """The unit that needs longest for these operations, its rate and the fraction of its peak."""
    from paper_1807_01151_gb300 import perfmodel
    t = perfmodel.unit_times(ops, peaks, hbm_gbs)
    unit = max(t, key=t.get)
    frac = t[unit] / seconds
    peak, name = {"int": (perfmodel.INT_MAD_TOPS, "T integer multiply-adds/s"), "f64": (peaks["fp64_tflops"], "TFLOP/s"),
                  "f32": (peaks["fp32_tflops"], "TFLOP/s"), "hbm": (hbm_gbs, "GB/s")}[unit]
    return {"bound": "hbm" if unit == "hbm" else "alu", "pipe": unit, "achieved": frac * peak, "peak": peak, "unit": name,
            "frac": frac}


def unit_rooflines(prof_cycle, work, peaks, hbm_gbs):
    """unit_roofline of every kernel class of a cycle (perfmodel.kernel_work)."""
    return {k: dict(unit_roofline(work[k], v["ms_per_cycle"] * 1e-3, peaks, hbm_gbs), ms_per_cycle=v["ms_per_cycle"])
            for k, v in prof_cycle.items() if k in work and v["ms_per_cycle"] > 0}


def measure(pkg, torch, mesh, W, prec, args, world, local, rank, with_clocks, peaks, hbm_gbs):
    """Time K V-cycles of one form; return a dict of results (and the solver closed)."""
    import numpy as np
    from paper_1807_01151_gb300 import perfmodel
    stream = torch.cuda.Stream()
    # set-up (mesh, geometry, basis, quadrature tables, Gauss-Jordan tuner), reported apart
    torch.cuda.synchronize()
    t_setup = time.perf_counter()
    s = pkg.Solver(mesh, p_max=W["p_max"], mach=W["mach"], prec=prec, stream=stream.cuda_stream,
                   block_kernels=args.block_kernels, krylov_f32=args.krylov_f32)
    torch.cuda.synchronize()
    t_setup = time.perf_counter() - t_setup
    E, N = s.E, s.n_modes(W["p_max"])
    K = 5 * N * E
    F = int((mesh.face_bc.size + (mesh.face_bc >= 0).sum()) // 2)   # interior faces counted twice
    dim = mesh.dim
    s.set_state(None)
    for _ in range(max(args.warmup, 3)):
        s.vcycle(info=False)
    torch.cuda.synchronize()

    def barrier():
        if world > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()

    outdir = clocks_dir()
    clocks = Clocks(local, os.path.join(outdir, f"clocks_rank{rank}_{PREC_NAMES[prec]}.csv")) if with_clocks else None
    # timed region: the product path (captured graphs replayed), profiler off
    l0 = s.launch_count
    barrier()
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for _ in range(args.steps):
        s.vcycle(info=False)
    ev1.record(stream)
    barrier()
    ms = ev0.elapsed_time(ev1)
    launches = s.launch_count - l0
    clk = clocks.stop() if clocks else None
    ms = max_over_ranks(ms)
    out = {"value": world * K * args.steps / (ms * 1e-3) / 1e9, "ms_per_step": ms / args.steps,
           "gpu_launches": launches, "graph_kernels": s.graph_kernels, "clocks": clk, "K": K, "E": E}
    # a separate pass with the event profiler (kernel by kernel) for the split per kernel class
    nprof = max(3, min(args.steps, 5))
    s.profile(True)
    for _ in range(nprof):
        s.vcycle(info=False)
    prof = s.profile_read()
    s.profile(False)
    prof_cycle = {k: {"ms_per_cycle": v[0] / nprof, "launches_per_cycle": v[1] / nprof}
                  for k, v in prof.items() if v[1]}
    out["kernels"] = prof_cycle
    out["kernels_total_ms_per_cycle"] = sum(v["ms_per_cycle"] for v in prof_cycle.values())
    # residual throughput (p_max residual, device buffers, back-to-back)
    u = torch.empty((E, 5, N), dtype=torch.float64, device="cuda")
    R = torch.empty_like(u)
    s.get_state(u)
    torch.cuda.synchronize()
    for _ in range(10):
        s.residual(W["p_max"], u, R)
    nres = 200
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(nres):
        s.residual(W["p_max"], u, R)
    e1.record(stream)
    torch.cuda.synchronize()
    res_ms = e0.elapsed_time(e1) / nres
    # the same loop with the event profiler: per-launch time of each residual kernel at p_max
    s.profile(True)
    for _ in range(nres):
        s.residual(W["p_max"], u, R)
    rprof = s.profile_read()
    s.profile(False)
    vol_launch_ms = rprof["residual_volume"][0] / rprof["residual_volume"][1]
    out["residual_gdofs"] = K / (res_ms * 1e-3) / 1e9
    out["residual_ms"] = res_ms
    # end to end through the C ABI with host buffers: H2D state, V-cycle, D2H state + info
    host = torch.empty((E, 5, N), dtype=torch.float64, pin_memory=True).numpy()
    s.get_state(host)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        s.set_state(host)
        s.vcycle(info=True)
        s.get_state(host)
    e2e_s = time.perf_counter() - t0
    out["setup_s"] = t_setup
    out["e2e"] = {"value": world * K * args.steps / e2e_s / 1e9, "unit": "GDoF/s",
                  "h2d_bytes_per_step": K * 8, "d2h_bytes_per_step": K * 8 + 64}
    # time to a 1e-10 drop from the free stream; then on to a 1e-12 drop (not timed), where the
    # states of the two forms are compared as well
    if not args.no_solve:
        s.set_state(None)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        rep = s.solve_steady(drop=1e-10, max_cycles=5000, raise_on_fail=False)
        out["time_to_1e-10"] = {"seconds": time.perf_counter() - t0, "cycles": rep["cycles"],
                                "converged": rep["converged"],
                                "drop": rep["res_final"] / rep["res0"] if rep["res0"] else None}
        out["state"] = s.get_state()
        if with_clocks and args.start_seeds > 0:
            # the cycle count to 1e-10 depends on rounding (the weakly unstable antisymmetric mode
            # of the cylinder is seeded by it): the same solve from starts 1e-13 apart
            s.set_state(None)
            u0 = s.get_state()
            cyc, sec = [rep["cycles"]], [out["time_to_1e-10"]["seconds"]]
            for seed in range(1, args.start_seeds + 1):
                rng = np.random.default_rng(seed)
                s.set_state(np.ascontiguousarray(u0 * (1.0 + 1e-13 * rng.standard_normal(u0.shape))))
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                r2 = s.solve_steady(drop=1e-10, max_cycles=5000, raise_on_fail=False)
                cyc.append(r2["cycles"] if r2["converged"] else None)
                sec.append(time.perf_counter() - t0 if r2["converged"] else None)
            ok = [x for x in sec if x is not None]
            out["start_spread"] = {"starts": "free stream, then the free stream times (1 + 1e-13 z), z seeded normal",
                                   "cycles": cyc, "seconds": [None if x is None else round(x, 3) for x in sec],
                                   "median_s": float(np.median(ok)) if ok else None}
    # roofline of the residual's largest kernel, k_volume at p_max, per launch (the operations of its
    # formulation / live launch time), and of every kernel class per cycle
    top = perfmodel.kernel_work(dim, W["p_max"], E, F, form=prec)
    below = perfmodel.kernel_work(dim, W["p_max"] - 1, E, F, form=prec) if W["p_max"] > 0 else None
    launches_top = 2 if below is None else 1 + 2 * 4   # residuals of that level in a cycle
    ops = {u: (n - (below["residual_volume"][u] if below else 0.0)) / launches_top
           for u, n in top["residual_volume"].items()}
    out["roofline"] = dict(unit_roofline(ops, vol_launch_ms * 1e-3, peaks, hbm_gbs),
                           kernel=f"k_volume<{dim},{W['p_max']}> (DG residual, volume + face projection)",
                           traffic=VOLUME_P4_TRAFFIC.get(W["name"]),
                           peak_source=peaks["fp64_source"], probe_tflops=peaks["fp64_probe_tflops"],
                           operations_per_launch=ops, ms_per_launch=vol_launch_ms,
                           note="unit that needs longest for the kernel's own operations (perfmodel.kernel_work)")
    out["rooflines"] = unit_rooflines(prof_cycle, top, peaks, hbm_gbs)
    s.close()
    return out


def run_serve(args, rank, world, local):
    """The served stream: 64 cylinder solves (seed 1807, Poisson arrivals at 4/s, O-grids
    32x16..256x128, p in 1..4, Ma in [0.1, 0.5]) through the library's request loop, mixed
    form.  Replicas only: with N ranks every rank serves its own copy of the stream."""
    import torch
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    from paper_1807_01151_gb300 import serving
    from workloads import ogrid, request_stream
    reqs = request_stream(n=args.serve_requests)
    cache = {}

    def make_mesh(rq):
        key = (rq.n_theta, rq.n_r)
        if key not in cache:
            cache[key] = ogrid(*key)
        return cache[key]

    for rq in reqs:
        make_mesh(rq)
    if world > 1:
        torch.distributed.barrier()
    outdir = clocks_dir()
    clocks = Clocks(local, os.path.join(outdir, f"clocks_rank{rank}_serve.csv"))
    out, summ = serving.serve_stream(reqs, make_mesh, max_active=args.max_active, prec=1,
                                     stall_cycles=args.stall_cycles)
    clk = clocks.stop()
    span = summ["makespan_s"]
    span = max_over_ranks(span)
    if rank == 0:
        line = {
            "metric": "served steady solves to a 1e-10 drop: solves/s, p50/p99 time-to-converge",
            "value": world * summ["converged"] / span, "unit": "solves/s", "n_gpus": world,
            "steps": len(reqs), "warmup": 0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64+f32", "data": "synthetic",
            "config": {"workload": f"served_cylinder_stream_{len(reqs)}", "seed": 1807, "arrivals": "Poisson, 4/s",
                       "grids": "32x16, 64x32, 128x64, 256x128", "p": "1..4", "mach": "U[0.1, 0.5]",
                       "form": "fp32_blocks", "max_active": args.max_active, "stall_cycles": args.stall_cycles,
                       "parallelism": "replicas" if world > 1 else "single GPU"},
            "p50_s": summ["p50_s"], "p99_s": summ["p99_s"], "makespan_s": span,
            "converged": summ["converged"], "requests": summ["requests"], "peak_active": summ["peak_active"],
            "cycles_total": summ["cycles_total"], "clocks": clk,
            "failed": [dict(id=r["id"], status=r["status_name"], cycles=r["cycles"],
                            drop=(r["res_final"] / r["res0"]) if r["res0"] > 0 else None,
                            grid=f"{reqs[k].n_theta}x{reqs[k].n_r}", p=reqs[k].p, mach=round(reqs[k].mach, 3))
                       for k, r in enumerate(out) if r["status"] != 0],
            "per_request": [dict(grid=f"{reqs[k].n_theta}x{reqs[k].n_r}", p=reqs[k].p, mach=round(reqs[k].mach, 3),
                                 status=r["status_name"], cycles=r["cycles"],
                                 ttc_s=round(r["time_to_converge"], 3)) for k, r in enumerate(out)],
        }
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()


def main():
    args = parse()
    if args.serve and args.impl == "emg":
        rank, world, local = dist_info()
        return run_serve(args, rank, world, local)
    W = WORKLOADS[args.workload]
    rank, world, local = dist_info()
    if args.impl == "reference":
        return run_reference(args, rank, world)
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        cpu = cpu_baseline(W, 2, 0)   # spawned workers, before any GPU work
    import torch
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    import paper_1807_01151_gb300 as pkg
    from paper_1807_01151_gb300._lib import probe_peaks
    probe = probe_peaks()
    mp_, mp_src = measured_peaks()
    # ALU roofs from the unit counts and the SM clock (the recipe's maximum clock unless the
    # samples of the timed region are lower); the probe measures the same roofs directly
    clk0 = Clocks(local, os.path.join(clocks_dir(), f"clocks_rank{rank}_probe.csv"))
    probe2 = probe_peaks()
    cs = clk0.stop() or {}
    mhz = float(mp_.get("sm_max_mhz", 2070.0))
    peaks = {
        "fp64_tflops": 2 * 2 * 152 * mhz * 1e6 / 1e12, "fp32_tflops": 128 * 2 * 152 * mhz * 1e6 / 1e12,
        "fp64_source": f"2 FP64 FMA/clk/SM x 2 flop x 152 SMs x {mhz:.0f} MHz (unit counts x maximum SM clock)",
        "fp32_source": f"128 FP32 FMA/clk/SM x 2 flop x 152 SMs x {mhz:.0f} MHz",
        "fp64_probe_tflops": max(probe["fp64_tflops"], probe2["fp64_tflops"]),
        "fp32_probe_tflops": max(probe["fp32_tflops"], probe2["fp32_tflops"]),
        "probe_sm_mhz": probe2["sm_mhz"], "probe_clock_samples": cs,
    }
    hbm_gbs = float(mp_.get("hbm_gbs", 6800.0))
    mesh = make_mesh(W)
    precs = {"all": [1, 0, 2], "both": [1, 0], "mixed": [1], "fp64": [0], "bf16": [2]}[args.prec]
    res = {p: measure(pkg, torch, mesh, W, p, args, world, local, rank, with_clocks=(i == 0), peaks=peaks,
                      hbm_gbs=hbm_gbs)
           for i, p in enumerate(precs)}
    head = res[precs[0]]
    if rank == 0:
        t_key = {}
        for p in precs:
            t = res[p].get("time_to_1e-10")
            if t:
                t_key[f"t_1e-10_{PREC_NAMES[p]}_s"] = round(t["seconds"], 3)
                t_key[f"cycles_1e-10_{PREC_NAMES[p]}"] = t["cycles"]
                t_key[f"converged_{PREC_NAMES[p]}"] = t["converged"]
            t_key[f"setup_{PREC_NAMES[p]}_s"] = round(res[p]["setup_s"], 3)
            if "start_spread" in res[p]:
                t_key[f"start_spread_{PREC_NAMES[p]}"] = res[p]["start_spread"]
        if W.get("kind") != "sphere" and 0 in res and "state" in res[0]:
            if 1 in res and "state" in res[1]:
                t_key.update(state_comparison(res[1]["state"], res[0]["state"], W))
            if 2 in res and "state" in res[2]:
                c2 = state_comparison(res[2]["state"], res[0]["state"], W)
                t_key["bf16_vs_fp64_symmetric_part_relerr"] = c2["mixed_vs_fp64_symmetric_part_relerr"]
                t_key["bf16_vs_fp64_converged_relerr"] = c2["mixed_vs_fp64_converged_relerr"]
        line = {
            "metric": METRIC, "value": head["value"], "unit": "GDoF/s", **t_key,
            "n_gpus": world, "steps": args.steps,
            "warmup": max(args.warmup, 3), "ms_per_step": head["ms_per_step"], "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": {0: "f64", 1: "f64+f32", 2: "f64+bf16"}[precs[0]],
            "data": "synthetic",
            "config": {"workload": W["name"],
                       "mesh": (f"cubed-sphere shell 6x{W['n']}x{W['n']}x{W['n_r']} r in [0.5,20]" if W.get("kind") == "sphere"
                                else f"O-grid {W['n_theta']}x{W['n_r']} r in [0.5,20]"),
                       "p_max": W["p_max"], "elements": head["E"], "dof": head["K"], "mach": W["mach"],
                       "form": PREC_NAMES[precs[0]],
                       "l2": "inputs larger than L2: tables and block factors stream > 1 GB per V-cycle",
                       "timed_path": "captured V-cycle graphs replayed, profiler off",
                       "block_kernels": args.block_kernels, "krylov_f32": args.krylov_f32,
                       "parallelism": "replicas" if world > 1 else "single GPU"},
            "residual_gdofs": head["residual_gdofs"], "residual_ms": head["residual_ms"],
            "time_to_1e-10": head.get("time_to_1e-10"),
            "e2e": head["e2e"], "gpu_launches": head["gpu_launches"], "roofline": head["roofline"],
            "clocks": head["clocks"], "cpu_baseline": cpu,
            "peaks": dict(peaks, hbm_gbs=hbm_gbs, hbm_source=mp_src),
            "rooflines": head["rooflines"], "kernels": head["kernels"],
            "kernels_total_ms_per_cycle": head["kernels_total_ms_per_cycle"],
        }
        for p in precs[1:]:
            r = res[p]
            line[PREC_NAMES[p]] = {k: r[k] for k in ("value", "ms_per_step", "residual_gdofs", "time_to_1e-10",
                                                     "gpu_launches", "rooflines", "kernels") if k in r}
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()
