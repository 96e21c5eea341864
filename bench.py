"""Throughput of the two-phase lattice Boltzmann step on GB300.

Workload (default): D3Q27 drop impact on a textured wall, 384x384x256, a wall
at z = 0 with 8x8x16 pillars at pitch 16 (halfway bounce-back, solid density
rho_v), Peng-Robinson EOS at T/Tc = 0.5 (density ratio 1.1e4), a drop of
radius 60 moving down at U = 0.05 (seeded synthetic init, see
paper_2112_01975_gb300/inputs.py), FP32 storage with the fused FP32 step; the
FP64 path is timed on the same workload and reported under "f64". One bench
step = one lattice time step over all 37.7 M nodes (moments, EOS, Korteweg
force, correction, collision, streaming with bounce-back). Metric: MLUPS
(million lattice-node updates per second), whole job. The population buffers
(2 x 4.08 GB in FP32) exceed the 129 MB L2, so no flush is needed between
steps. ``--workload`` selects another configured workload (the 128^3 drop,
the 256^3 coalescence).

  python bench.py [--gpus N --steps K --warmup W] [--impl reference]

With N > 1 (torchrun), every rank advances its own replica (the method has no
cross-lattice exchange in this workload): weak scaling, max time over ranks.
``--impl reference`` times the FP64 CPU oracle on the host cores instead.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

ALG_BYTES_PER_LU = {  # populations read once and written once per lattice update
    (1, "f64"): 2 * 27 * 8,
    (0, "f64"): 2 * 9 * 8,
    (1, "f32"): 2 * 27 * 4,
    (0, "f32"): 2 * 9 * 4,
    # 16-bit populations plus the 4-byte source density read and written
    (1, "f16s"): 2 * 27 * 2 + 8,
    (0, "f16s"): 2 * 9 * 2 + 8,
    (1, "bf16s"): 2 * 27 * 2 + 8,
    (0, "bf16s"): 2 * 9 * 2 + 8,
}
# FP64 flops per node executed by the D3Q27 collision kernel (k_force_sweep3
# with its collision), counted from the source: force sums of two fields 111
# (per field and with the tile's halo: differences 9, x smoothing of the z
# differences 9, each node's smoothings 18, z sums and rings 20), force
# 11, Phi 3, 1/rho and its factor 3, product-form factors 54, partial products
# 26, collision 135; at relaxation time 1, where the equilibrium and the
# populations drop out, the last three are 33, 12 and 27.
def collide_fp64_flops(tau: float) -> int:
    return 200 if tau == 1.0 else 343


FP64_PEAK_TFLOPS = 1.25   # GB300 nominal FP64 rate (context; the roofline uses the live probe)


def fp64_peak():
    """(TFLOP/s, source) of the FP64 roofline: the library's FMA-chain probe
    on this GPU, run now; the nominal rate only if the probe fails."""
    from paper_2112_01975_gb300.lbm import LBMError, probe_fp64_tflops
    try:
        return probe_fp64_tflops(), "measured: FP64 FMA-chain probe (lbm_probe_fp64_tflops), this run"
    except LBMError:
        return FP64_PEAK_TFLOPS, "nominal FP64 rate of GB300 (recipe table; the probe failed)"


# DRAM bytes (dram__bytes_read.sum + dram__bytes_write.sum) per lattice node
# of one launch of the fused step, from an ncu capture of the named workload
# (scaled to the capture's lattice, as stated), keyed by (workload, storage,
# tile rows, fused-step form); each entry records the SHA-256 prefix of the fused kernel's
# source it was taken on, and is not used once that source has changed.
MEASURED_TRAFFIC = {
    # k_step_f32_wstma, 32 x 8 tiles, chunk 247 (one 247-plane and one
    # 9-plane chunk per column, as at full size), on the impact scaled to
    # 192x192x256: 1116.2 + 964.1 MB for 9,437,184 nodes
    # (profiles/k_step_f32_wstma_d3q27_impact_192x192x256.md)
    ("d3q27_impact_384x384x256_pr_tr0.5", "f32", 8, 4): {
        "bytes_per_node": 220.43, "src_sha": "76cdd479947f5188"},
    # k_step_shifted_tmtma (FP16-shifted, Tensor Memory with TMA-staged
    # planes), 32 x 8 tiles, chunk 240, on the same scaled impact: 583.4 +
    # 504.3 MB for 9,437,184 nodes
    # (profiles/k_step_shifted_tmtma_d3q27_impact_192x192x256.md)
    ("d3q27_impact_384x384x256_pr_tr0.5", "f16s", 8, 5): {
        "bytes_per_node": 115.26, "src_sha": "76cdd479947f5188"},
}
FUSED_SRC = os.path.join(ROOT, "paper_2112_01975_gb300", "csrc", "lbm_fused_f32_body.cuh")


def fused_src_sha() -> str:
    import hashlib
    with open(FUSED_SRC, "rb") as fh:
        return hashlib.sha256(fh.read()).hexdigest()[:16]


def measured_traffic(name: str, storage: str, rows: int, variant: int, nodes: int):
    """ncu DRAM bytes of one launch scaled to `nodes`, or None."""
    v = MEASURED_TRAFFIC.get((name, storage, rows, variant))
    if v is None or v["src_sha"] != fused_src_sha():
        return None
    return v["bytes_per_node"] * nodes


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=400)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="d3q27_impact_384x384x256_pr_tr0.5")
    ap.add_argument("--shape", default="",
                    help="nx,ny,nz: run the workload scaled to this lattice (profiling captures)")
    ap.add_argument("--storage", default="f32", choices=["f64", "f32", "f16s", "bf16s"])
    ap.add_argument("--chunk", type=int, default=0, help="planes per CTA of the FP32 step")
    ap.add_argument("--tile", type=int, default=0, choices=[0, 7, 8],
                    help="D3Q27 FP32 tile height (0: picked by the autotuner, or 8 with --chunk)")
    ap.add_argument("--variant", type=int, default=-1, choices=[-1, 0, 1, 2, 3, 4, 5],
                    help="fused-step form: 0 plain, 1 warp-specialised, 2 Tensor Memory, 3 "
                         "warp-specialised with Tensor Memory, 4 the same with TMA-staged planes, "
                         "5 Tensor Memory with TMA-staged planes (shifted storage) "
                         "(-1: picked by the autotuner, or plain with --chunk)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-f64", action="store_true", help="skip the FP64 side measurement")
    ap.add_argument("--eos64", action="store_true",
                    help="reduced storage with the EOS and force sums in FP64 (LBM_FLAG_EOS_F64)")
    ap.add_argument("--no-serve", action="store_true",
                    help="skip the serving sweep reported under \"serve\"")
    ap.add_argument("--mode", default="step", choices=["step", "serve", "validate"],
                    help="serve: the parameter-sweep server against one-at-a-time FP64; "
                         "validate: the coexistence/Laplace, coalescence and impact runs "
                         "at their configured lengths")
    ap.add_argument("--validate", default="", help="validate mode: comma list of cfg2,cfg3,cfg4")
    ap.add_argument("--validate-storages", default="f64,f32,f16s,bf16s",
                    help="validate mode: storages of the coalescence run")
    ap.add_argument("--requests", type=int, default=48)
    ap.add_argument("--request-steps", type=int, default=500)
    return ap.parse_args()


def dist_setup(n_gpus):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


class ClockSampler:
    """nvidia-smi clocks and throttle reasons: one `nvidia-smi -lms 100`
    process, started (and seen to answer) before the timed region; the rows
    that arrive while the region runs are kept."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.rows = []          # (arrival time, fields)
        self.proc = None
        self._t = None
        self.t0 = self.t1 = 0.0

    def _read(self):
        for line in self.proc.stdout:
            line = line.strip()
            if line:
                self.rows.append((time.monotonic(), [c.strip() for c in line.split(",")]))

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.FIELDS,
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self._t = threading.Thread(target=self._read, daemon=True)
            self._t.start()
            deadline = time.monotonic() + 5.0
            while not self.rows and time.monotonic() < deadline and self.proc.poll() is None:
                time.sleep(0.02)
        except Exception:
            self.proc = None
        self.t0 = time.monotonic()
        return self

    def __exit__(self, *a):
        self.t1 = time.monotonic()
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            self._t.join(timeout=5)

    def summary(self):
        if not self.rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        rows = [r for t, r in self.rows if self.t0 <= t <= self.t1]
        if not rows:   # a region shorter than the 100 ms period: the last row before its end
            rows = [r for t, r in self.rows if t <= self.t1][-1:] or [self.rows[0][1]]
        sm = [float(r[1]) for r in rows if len(r) > 2 and r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if len(r) > 2 and r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in rows for k in range(4)
                          if len(r) > 5 + k and r[5 + k].lower().startswith("active")})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(rows)}


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def host_cpu() -> dict:
    """The host's CPU model (lscpu, else the platform) and core count."""
    import platform
    model = platform.machine()
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.startswith("Model name:"):
                model = line.split(":", 1)[1].strip()
                break
    except Exception:
        pass
    return {"cpu": model, "nproc": os.cpu_count()}


def sample_shape(w, kind: str):
    """Lattice of the CPU oracle's bounded sample of workload w: the
    all-host-cores and one-thread baselines ("cpu") and the reference arm,
    whose every step is one lattice update of it ("reference")."""
    if w.lattice == 0:
        return (64, 64, 1)
    if w.mask_seed is not None:   # the impact keeps its pillars and gap: a 1/4 or 1/6 box
        return (96, 96, 64) if kind == "cpu" else (48, 48, 48)
    return (48, 48, 48) if kind == "cpu" else (32, 32, 32)


def oracle_for(w, shape, openmp: bool = False):
    """The FP64 oracle on workload w scaled to shape, initialised."""
    from oracle.lbm import OracleLBM
    rho, u0, mask = w.fields(shape)
    nx, ny, nz = shape
    o = OracleLBM(w.lattice, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, w.tau, mask=mask, a=w.a,
                  b=w.b, rho_w=1.0 if w.rho_w is None else w.rho_w, openmp=openmp)
    o.init(rho, u0)
    return o


def oracle_sample_mlups(w, target_s: float = 12.0, openmp: bool = False):
    """FP64 oracle throughput on the workload scaled down (sample_shape): one
    host thread, or (openmp) the -fopenmp build of the same source on all cores."""
    shape = sample_shape(w, "cpu")
    o = oracle_for(w, shape, openmp=openmp)
    o.step(1)
    steps, t0 = 0, time.perf_counter()
    while time.perf_counter() - t0 < target_s:
        o.step(1)
        steps += 1
    dt = time.perf_counter() - t0
    nodes = shape[0] * shape[1] * shape[2]
    return nodes * steps / dt / 1e6, (f"the workload scaled to {shape[0]}x{shape[1]}x{shape[2]} "
                                      f"(drop radius and centres x {shape[0]}/{w.nx}), {steps} "
                                      f"steps, {dt:.1f} s")


def run_reference(args, w, world, rank):
    """The CPU oracle as it stands, one host thread, each step one lattice
    update of the workload scaled down (sample_shape)."""
    if rank != 0:
        return
    shape = sample_shape(w, "reference")
    o = oracle_for(w, shape)
    for _ in range(args.warmup):
        o.step(1)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        o.step(1)
    dt = time.perf_counter() - t0
    nodes = shape[0] * shape[1] * shape[2]
    mlups = nodes * args.steps / dt / 1e6
    sample = (f"{w.name} scaled to {shape[0]}x{shape[1]}x{shape[2]} (drop radius and centres x "
              f"{shape[0]}/{w.nx}), one lattice update per step")
    print(json.dumps({
        "impl": "reference", "metric": "MLUPS", "value": mlups, "unit": "MLUPS",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": dt / args.steps * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": w.name, "lattice": "D3Q27" if w.lattice else "D2Q9",
                   "nodes": w.nodes, "storage": "f64"},
        "cpu_baseline": {"value": mlups, "unit": "MLUPS", "cores": 1, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": mlups, "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


def reduce_max(x: float, dist, device) -> float:
    """Largest x over all ranks (x itself without a process group)."""
    if dist is None:
        return x
    import torch
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_mlups(nodes: int, steps: int, world: int, max_ms: float) -> float:
    """Whole-job MLUPS: every rank advances its own replica of `nodes` nodes
    `steps` times; the job takes as long as the slowest rank."""
    return nodes * steps * world / (max_ms * 1e-3) / 1e6


def timed_steps(g, stream, steps, dist, local):
    """Time exactly `steps` lattice steps (graph replays) with CUDA events on
    the handle's stream, barrier + synchronize on both sides."""
    import torch

    def barrier():
        torch.cuda.synchronize()
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    barrier()
    l0 = g.launches
    e0.record(stream)
    g.step(steps)
    e1.record(stream)
    e1.synchronize()
    l1 = g.launches
    barrier()
    g.sync()
    ms = reduce_max(e0.elapsed_time(e1), dist, "cuda")
    return ms, l1 - l0


def serve_sweep(count: int, request_steps: int, seed: int = 5) -> dict:
    """Sweep of Poisson-arriving drop solves (rate 50/s): the continuous-
    batching server (each request FP32 or FP16-shifted, drawn per request)
    against the same requests solved one at a time in FP64. Each request's
    host set-up (EOS values from a table built once per arm, the initial
    density field) runs after its arrival and counts in its latency."""
    from paper_2112_01975_gb300 import eos_tables, serve
    reqs = serve.sweep_requests(count=count, rate=50.0, seed=seed, steps=request_steps)
    t = time.perf_counter()
    trs = [r.t_over_tc for r in reqs]
    table = eos_tables.SetupTable(0, min(trs), max(trs))
    t_table = time.perf_counter() - t
    srv = serve.Server(hbm_budget=64 << 30, tick_steps=50)
    fast = serve.summarize(srv.run(reqs, realtime=True, table=table))
    slow = serve.summarize(serve.run_sequential_f64(reqs, realtime=True, table=table))
    return {
        "metric": "sweep solves/s, p50/p99 latency", "unit": "solves/s",
        "value": fast["solves_per_s"], "higher_is_better": True,
        "server_batched_f32_f16s": fast, "sequential_fp64": slow,
        "speedup_solves_per_s": fast["solves_per_s"] / slow["solves_per_s"],
        "p99_ratio": slow["p99_s"] / fast["p99_s"],
        "config": {"workload": "sweep of static/oscillating drops, D2Q9 64..512^2 and D3Q27 "
                               "64..192^3, T/Tc U[0.5, 0.95], radius U[0.15, 0.35] n, "
                               "Poisson arrivals 50/s, storage FP32 or FP16-shifted "
                               "with probability 1/2, interface width 5, rest start",
                   "requests": count, "steps_per_request": request_steps,
                   "lattice_updates": sum(r.nodes * r.steps for r in reqs),
                   "tick_steps": 50, "hbm_budget_gib": 64,
                   "peak_resident": srv.peak_resident, "batches_built": srv.batches_built,
                   "latency": "arrival to result on the host, set-up included",
                   "setup_table_s": t_table}}


def run_serve(args):
    import __graft_entry__
    __graft_entry__.build()
    import torch
    torch.cuda.set_device(0)
    out = serve_sweep(args.requests, args.request_steps)
    out["mode"] = "serve"
    out["data"] = "synthetic"
    print(json.dumps(out), flush=True)


def _validate_cfg2(L, storage, tr, steps):
    """D3Q27 128^3, PR at T/Tc: a flat slab (liquid 32 <= x < 96) for the
    coexistence densities against Maxwell and the tension from the discrete
    pressure tensor, and a drop of radius 24 for the Laplace law
    Delta P = 2 sigma / R_e (3D), R_e the equimolar radius."""
    from paper_2112_01975_gb300 import eos_tables, inputs
    a = eos_tables.stable_a(1, tr)
    rv, rl, ps = eos_tables.coexistence(1, tr, a)
    kap = eos_tables.kappa_for_width(1, tr, a, width=5.0)
    P = eos_tables.pressure(1, tr, a)
    n = 128
    st = {"f64": L.F64, "f32": L.F32}[storage]
    g = L.LBM(1, n, n, n, 1, tr, kap, 1.0, a=a, storage=st)
    g.init(inputs.slab(n, n, n, 32, 96, rv, rl))
    t0 = time.perf_counter()
    g.step(steps)
    g.sync()
    t_slab = time.perf_counter() - t0
    rho = g.moments()[0].reshape(n, n, n)
    line = rho[n // 2, n // 2]
    Pt = g.pressure_tensor().reshape(6, n, n, n)[:, n // 2, n // 2]
    sigma_flat = float(np.sum(Pt[0] - Pt[1])) / 2.0
    g.close()
    g = L.LBM(1, n, n, n, 1, tr, kap, 1.0, a=a, storage=st)
    g.init(inputs.drop(n, n, n, 24.0, rv, rl))
    g.step(steps)
    rho = g.moments()[0].reshape(n, n, n)
    r_in, r_out = float(rho[n // 2, n // 2, n // 2]), float(rho[0, 0, 0])
    vol = (float(rho.sum()) - r_out * n ** 3) / (r_in - r_out)
    R_e = (3.0 * vol / (4.0 * np.pi)) ** (1.0 / 3.0)
    sigma_lap = float(P(r_in) - P(r_out)) * R_e / 2.0
    g.close()
    return {"T/Tc": tr, "storage": storage, "steps": steps, "rho_v": float(line[0]),
            "rho_l": float(line[64]), "rho_v_maxwell": rv, "rho_l_maxwell": rl,
            "rho_v_err": float(line[0]) / rv - 1.0, "rho_l_err": float(line[64]) / rl - 1.0,
            "sigma_flat_pressure_tensor": sigma_flat, "sigma_laplace": sigma_lap,
            "R_e": R_e, "laplace_vs_flat": sigma_lap / sigma_flat - 1.0,
            "mlups_slab": n ** 3 * steps / t_slab / 1e6}


def _validate_cfg3(L, torch, storage, steps, every=1000):
    """Two PR drops of radius 40 touching at the centre of a periodic 256^3
    box, T/Tc 0.45, tau 0.725: mass drift, far-field vapour and drop-centre
    liquid densities, and the neck radius (liquid area of the mid-plane
    between the drops, r = sqrt(A / pi)) every `every` steps."""
    from paper_2112_01975_gb300 import eos_tables, inputs
    tr, n, R = 0.45, 256, 40.0
    a = eos_tables.stable_a(1, tr)
    rv, rl, _ = eos_tables.coexistence(1, tr, a)
    kap = eos_tables.kappa_for_width(1, tr, a, width=5.0)
    flags = L.FLAG_EOS_F64 if storage.endswith("e64") else 0
    st = {"f64": L.F64, "f32": L.F32, "f16s": L.F16S, "bf16s": L.BF16S}[storage.replace("e64", "")]
    centres = [(n // 2 - R, n // 2, n // 2), (n // 2 + R, n // 2, n // 2)]
    rho0 = inputs.add_noise(inputs.drops(n, n, n, centres, R, rv, rl, width=5.0), 1e-4, 3)
    g = L.LBM(1, n, n, n, 1, tr, kap, 0.725, a=a, storage=st, flags=flags)
    g.init(rho0)
    m0, _ = g.reduce()
    rho_t = torch.empty(n ** 3, dtype=torch.float64, device="cuda")
    mid = 0.5 * (rl + rv)
    neck, t0 = [], time.perf_counter()
    for s in range(every, steps + 1, every):
        g.step(every)
        g.moments((rho_t, None, None))
        area = int((rho_t.view(n, n, n)[:, :, n // 2] > mid).sum())
        neck.append((s, float(np.sqrt(area / np.pi))))
    g.sync()
    dt = time.perf_counter() - t0
    m1, _ = g.reduce()
    r = rho_t.view(n, n, n)
    liquid = r[r > mid]
    vapour = r[r < mid]
    out = {"storage": storage, "steps": steps, "mass_drift": m1 / m0 - 1.0,
           "rho_v_far": float(r[0, 0, 0]), "rho_l_median": float(liquid.median()),
           "rho_v_median": float(vapour.median()), "rho_l_maxwell": rl, "rho_v_maxwell": rv,
           "neck_radius": neck, "mlups_incl_readback": n ** 3 * steps / dt / 1e6}
    g.close()
    return out


def _validate_cfg4(L, steps, every=2000):
    """The impact workload (inputs.IMPACT_D3Q27_384: a drop of radius 60 at
    U = 0.115, We = 100, onto 8x8x16 pillars on a two-plane wall,
    384x384x256, PR T/Tc 0.5, tau 0.725, FP32): mass drift, the liquid area
    just above the pillar tops and the height of the liquid's centre of mass
    over time, and the last step reached."""
    from paper_2112_01975_gb300 import inputs
    w = inputs.IMPACT_D3Q27_384
    nx, ny, nz = w.nx, w.ny, w.nz
    rv, rl = w.rho_v, w.rho_l
    rho0, u0, mask = w.fields()
    g = L.LBM(1, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, w.tau, mask=mask, a=w.a, b=w.b,
              rho_w=w.rho_w, storage=L.F32)
    g.init(rho0, u0)
    m0, _ = g.reduce()
    zt = w.wall + w.pillar[1]
    wet, t0, failed = [], time.perf_counter(), None
    for s in range(every, steps + 1, every):
        try:
            g.step(every)
            rho = g.moments()[0].reshape(nz, ny, nx)
        except L.LBMError as exc:
            failed = f"step <= {s}: {exc}"
            break
        liq = rho > 0.5 * (rl + rv)
        zc = float((np.arange(nz)[:, None, None] * liq).sum() / max(liq.sum(), 1))
        wet.append((s, float(np.sqrt(np.count_nonzero(liq[zt]) / np.pi)), zc))
    dt = time.perf_counter() - t0
    out = {"steps": steps, "U": w.u_down, "tau": w.tau, "wall_planes": w.wall,
           "step_wetted_radius_above_pillars_liquid_z": wet, "failed": failed}
    if failed is None:
        m1, _ = g.reduce()
        out["mass_drift"] = m1 / m0 - 1.0
        out["mlups_incl_readback"] = nx * ny * nz * steps / dt / 1e6
    g.close()
    return out


def run_validate(args):
    import __graft_entry__
    __graft_entry__.build()
    import torch
    from paper_2112_01975_gb300 import lbm as L
    torch.cuda.set_device(0)
    res = {"mode": "validate", "data": "synthetic", "cfg2": [], "cfg3": [], "cfg4": None}
    only = set(args.validate.split(",")) if args.validate else {"cfg2", "cfg3", "cfg4"}
    for tr in (0.9, 0.7) if "cfg2" in only else ():
        for st in ("f64", "f32"):
            res["cfg2"].append(_validate_cfg2(L, st, tr, 20000))
            print(json.dumps(res["cfg2"][-1]), file=sys.stderr, flush=True)
    for st in args.validate_storages.split(",") if "cfg3" in only else ():
        res["cfg3"].append(_validate_cfg3(L, torch, st, 10000))
        print(json.dumps(res["cfg3"][-1]), file=sys.stderr, flush=True)
    ref = res["cfg3"][0] if res["cfg3"] and res["cfg3"][0]["storage"] == "f64" else None
    for r in (res["cfg3"][1:] if ref else []):
        for k in ("rho_v_far", "rho_l_median", "rho_v_median"):
            r[k + "_vs_f64"] = r[k] / ref[k] - 1.0
    if "cfg4" in only:
        res["cfg4"] = _validate_cfg4(L, 20000, every=1000)
    print(json.dumps(res), flush=True)


def main():
    args = parse()
    if args.mode == "serve":
        run_serve(args)
        return
    if args.mode == "validate":
        run_validate(args)
        return
    from paper_2112_01975_gb300 import inputs
    w = inputs.WORKLOADS[args.workload]
    world, rank, local = dist_setup(args.gpus)
    if args.impl == "reference":
        run_reference(args, w, world, rank)
        return

    import __graft_entry__
    __graft_entry__.build()
    import ctypes
    import torch
    from paper_2112_01975_gb300.lbm import F32, F64, LBM, _lib

    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    stream = torch.cuda.Stream()
    from paper_2112_01975_gb300.lbm import BF16S, F16S
    storage = {"f64": F64, "f32": F32, "f16s": F16S, "bf16s": BF16S}[args.storage]
    shape = tuple(int(v) for v in args.shape.split(",")) if args.shape else (w.nx, w.ny, w.nz)
    nx, ny, nz = shape
    nodes = nx * ny * nz
    rho0, u0, mask = w.fields(shape)
    D = 3 if w.lattice else 2

    from paper_2112_01975_gb300.lbm import FLAG_EOS_F64

    def make(st):
        return LBM(w.lattice, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, w.tau, mask=mask, a=w.a,
                   b=w.b, rho_w=w.rho_w, stream=stream, storage=st,
                   flags=FLAG_EOS_F64 if args.eos64 and st != F64 else 0)

    g = make(storage)
    g.init(rho0, u0)
    chunk = 0
    if storage != F64:
        chunk = args.chunk or g.autotune()
        g.set_chunk(chunk)
        if args.tile and storage == F32 and w.lattice == 1:
            g.set_tile(args.tile)
        if args.variant >= 0:
            g.set_fused_variant(args.variant)
    g.step(args.warmup)
    g.sync()
    with ClockSampler(local) as clocks:
        ms, launches = timed_steps(g, stream, args.steps, dist, local)
    mlups = job_mlups(nodes, args.steps, world, ms)

    # The dominant kernel's average launch duration over the timed region:
    # the replayed graph launches one fused kernel per step (FP32 and
    # shifted storage), so it is the timed region's length over its
    # launches. Plain launches with events between kernels give a second
    # figure (and the FP64 path's split into its two kernels).
    n_t = max(5, min(50, args.steps // 4))
    ms_macro, ms_collide = g.time_kernels(n_t)
    peak, peak_kind = measured_peaks()
    alg = ALG_BYTES_PER_LU[(w.lattice, args.storage)] * nodes
    per_step = launches / args.steps if args.steps else 1
    tile = g.tile()
    variant = g.fused_variant if storage != F64 else 0
    if storage != F64:
        ms_launch = ms / max(launches, 1)
        achieved = alg / (ms_launch * 1e-3) / 1e9
        traffic = measured_traffic(w.name, args.storage, tile[1], variant, nodes) if per_step == 1 else None
        roofline = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                    "frac": achieved / peak, "traffic": traffic,
                    "frac_of_nominal_7900_gbs": achieved / 7900.0,
                    "kernel": {0: "k_step_f32 (fused step)",
                               1: "k_step_f32_ws (fused step, warp-specialised)",
                               2: "k_step_f32_tm (fused step, Tensor Memory staging)",
                               3: "k_step_f32_wstm (fused step, warp-specialised, Tensor Memory "
                                  "staging)",
                               4: "k_step_f32_wstma (fused step, warp-specialised, Tensor Memory "
                                  "staging, TMA-staged planes)"}[variant]
                    if storage == F32 else
                    {0: "k_step_shifted", 2: "k_step_shifted_tm", 3: "k_step_shifted_wstm",
                     4: "k_step_shifted_wstma", 5: "k_step_shifted_tmtma (Tensor Memory, TMA-staged planes)"}
                    .get(variant, "k_step_shifted"),
                    "peak_source": peak_kind + " hbm_gbs (burst copy)",
                    "alg_bytes_per_launch": alg, "ms_per_launch": ms_launch,
                    "ms_per_launch_source": "CUDA events over the timed graph replays / launches",
                    "ms_per_launch_plain": ms_collide,
                    "chunk": chunk, "tile": f"{tile[0]}x{tile[1]}"}
    else:
        achieved = alg / (ms_collide * 1e-3) / 1e9
        tflops = collide_fp64_flops(w.tau) * nodes / (ms_collide * 1e-3) / 1e12
        p64, p64_src = fp64_peak()
        roofline = {"bound": "alu", "achieved": tflops, "peak": p64,
                    "unit": "TFLOP/s", "frac": tflops / p64,
                    "traffic": None,
                    "kernel": "k_force_sweep3 (FP64 force sweep and collision)",
                    "peak_source": p64_src, "nominal_peak": FP64_PEAK_TFLOPS,
                    "flops_per_node": collide_fp64_flops(w.tau),
                    "ms_per_launch": ms_collide, "ms_moments_kernel": ms_macro,
                    "hbm_achieved_gbs": achieved, "hbm_frac": achieved / peak}

    # end to end through the C ABI with pinned host buffers: the initial
    # density (and velocity) in, K steps, the density and velocity out
    pin_rho0 = torch.from_numpy(rho0).pin_memory()
    pin_u0 = torch.from_numpy(u0).pin_memory() if u0 is not None else None
    out_rho = torch.empty(nodes, dtype=torch.float64).pin_memory()
    out_u = torch.empty(D * nodes, dtype=torch.float64).pin_memory()
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    t0 = time.perf_counter()
    g.init(pin_rho0.numpy(), None if pin_u0 is None else pin_u0.numpy())
    g.step(args.steps)
    g._check(_lib.lbm_moments(g._h, ctypes.c_void_p(out_rho.data_ptr()),
                              ctypes.c_void_p(out_u.data_ptr()), None, 0))
    t_e2e = reduce_max(time.perf_counter() - t0, dist, "cuda")
    e2e_mlups = job_mlups(nodes, args.steps, world, t_e2e * 1e3)
    h2d = 8 * nodes * (1 + (D if u0 is not None else 0))

    # the FP64 path on the same workload, reported beside the headline
    f64 = None
    if storage == F32 and not args.no_f64:
        g.close()
        del g
        h = make(F64)
        h.init(rho0, u0)
        h.step(5)
        k64 = max(20, args.steps // 10)
        ms64, _ = timed_steps(h, stream, k64, dist, local)
        m64, c64 = h.time_kernels(10)
        p64, p64_src = fp64_peak()
        t64 = collide_fp64_flops(w.tau) * nodes / (c64 * 1e-3) / 1e12
        f64 = {"value": nodes * k64 * world / (ms64 * 1e-3) / 1e6, "unit": "MLUPS",
               "steps": k64, "ms_per_step": ms64 / k64,
               "roofline": {"bound": "alu", "kernel": "k_force_sweep3 (FP64 force sweep and collision)",
                            "achieved": t64, "peak": p64, "unit": "TFLOP/s", "frac": t64 / p64,
                            "peak_source": p64_src, "nominal_peak": FP64_PEAK_TFLOPS,
                            "ms_per_launch": c64, "ms_moments_kernel": m64}}
        h.close()

    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return
    serve_line = None
    if world == 1 and not args.no_serve:
        if f64 is None:
            g.close()
        torch.cuda.empty_cache()
        serve_line = serve_sweep(args.requests, args.request_steps)
    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        v, sample = oracle_sample_mlups(w)
        cpu = {"value": v, "unit": "MLUPS", "cores": 1, "kind": "oracle", "sample": sample,
               "host": host_cpu()}
        try:   # the same oracle built with -fopenmp, all host cores
            va, sa = oracle_sample_mlups(w, target_s=6.0, openmp=True)
            cores = int(os.environ.get("OMP_NUM_THREADS", os.cpu_count() or 1))
            cpu["all_cores"] = {"value": va, "unit": "MLUPS", "cores": cores,
                                "kind": "oracle, -fopenmp build", "sample": sa}
        except Exception as exc:   # no OpenMP in the host compiler
            cpu["all_cores"] = {"unavailable": str(exc)[:200]}
    line = {
        "metric": "MLUPS", "value": mlups, "unit": "MLUPS", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": args.storage + ("+eos64" if args.eos64 else ""),
        "data": "synthetic",
        "config": {"workload": w.name if not args.shape else f"{w.name} scaled to {args.shape}",
                   "lattice": "D3Q27" if w.lattice else "D2Q9", "shape": [nx, ny, nz],
                   "nodes": nodes, "storage": args.storage,
                   "eos": "Peng-Robinson" if w.eos == 1 else "vdW",
                   "solid_nodes": int(mask.sum()) if mask is not None else 0,
                   "l2": "inputs larger than L2 (2 x %.0f MB populations)" % (
                       (27 if w.lattice else 9) * {"f64": 8, "f32": 4}.get(args.storage, 2)
                       * nodes / 1e6),
                   "parallelism": f"replicas x{world}"},
        "roofline": roofline,
        "cpu_baseline": cpu,
        "e2e": {"value": e2e_mlups, "unit": "MLUPS",
                "h2d_bytes_per_step": h2d / args.steps,
                "d2h_bytes_per_step": 8 * (1 + D) * nodes / args.steps},
        "gpu_launches": launches,
        "clocks": clocks.summary(),
        "f64": f64,
        "serve": serve_line,
    }
    print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
