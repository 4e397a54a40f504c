#!/usr/bin/env python
"""Throughput of the D2Q9 bounce-back solver with per-step forces on one GB300.

One bench step is one lattice time step of the whole hot path: the fused
collide-stream kernel over the grid (bounce-back, inlet/outlet, DRTT partials)
plus the link kernel (momentum exchange A, A', B, DRTT and stress integration),
forces of every scheme recorded on the device.  Steps are taken four at a time
(one pass of the multi-step kernel): the roofline entry is that kernel's in the
timed region, roofline_single_step the single-step kernel's, timed launch by
launch outside it.  Default workload: 4096 x 2048 NACA0012, chord
256 at 4 degrees, Re 1000, FP32 storage.  The population arrays (2 x 302 MB)
exceed the 129 MB L2, so no flush is needed between steps.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Prints one JSON line (rank 0).  Under torchrun each rank runs an independent
replica of the workload (weak scaling, no collective on the data path).
"""
import argparse
import hashlib
import json
import os
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

BYTES_PER_UPDATE = {"f64": 144, "f32": 72, "f32dev": 72, "f16dev": 36}
FALLBACK_HBM_GBS = 6800.0


def args_():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=50000)
    p.add_argument("--warmup", type=int, default=200)
    p.add_argument("--impl", default="ours", choices=["ours", "reference"])
    p.add_argument("--no-variants", action="store_true")
    p.add_argument("--cpu-seconds", type=float, default=15.0)
    p.add_argument("--ref-seconds", type=float, default=None,
                   help="time budget of the reference (oracle) arm; default from steps+warmup")
    p.add_argument("--profile", action="store_true",
                   help="only create the solver and run warm-up + K steps (for ncu captures)")
    p.add_argument("--workload", default=None, help="workload name (profile mode)")
    p.add_argument("--storage", default=None, help="f64|f32|f32dev|f16dev (profile mode)")
    p.add_argument("--kernel", default="direct", choices=["direct", "staged"],
                   help="collide-stream kernel: direct loads or staged bulk copies")
    p.add_argument("--batch", type=int, default=0,
                   help="profile mode: a batch of the first N domains of the 256-domain "
                        "NACA00xx recipe instead of one workload")
    p.add_argument("--batch-launch", default=None,
                   help="profile mode: 'shape,ctas_per_sm' for the batch instead of the tuner")
    p.add_argument("--adjoint", type=int, default=0,
                   help="profile mode: run lbm_adjoint over this many steps (window: the last half) "
                        "instead of stepping")
    p.add_argument("--shrink", type=int, default=1,
                   help="profile mode: the workload's geometry shrunk by this integer factor")
    return p.parse_args()


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def reduce_max(value, device=None):
    """Max of a per-rank value over all ranks (the job's time is its slowest rank)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(value)
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


# Sources each profiled kernel is compiled from: a committed DRAM-traffic
# figure is used only while these files are unchanged.
KERNEL_SOURCES = {
    "collide_stream": ["lbm_step.cu", "lbm_collide.cuh", "lbm_device.cuh", "lbm_internal.cuh"],
    "collide_stream_f16dev": ["lbm_step.cu", "lbm_collide.cuh", "lbm_device.cuh",
                              "lbm_internal.cuh"],
    "march": ["lbm_march.cu", "lbm_march.cuh", "lbm_tma.cuh", "lbm_collide.cuh", "lbm_device.cuh",
              "lbm_internal.cuh"],
    "link_force": ["lbm_link.cu", "lbm_device.cuh", "lbm_internal.cuh"],
}
PASS_STEPS = 4  # steps of one pass of the multi-step kernel


def kernel_source_hash(kernel="collide_stream"):
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2210_10377_gb300", "csrc")
    for f in KERNEL_SOURCES[kernel]:
        with open(os.path.join(csrc, f), "rb") as fh:
            h.update(f.encode() + fh.read())
    return h.hexdigest()[:16]


def ncu_traffic(kernel, workload):
    """DRAM bytes per launch from a committed ncu summary, if it was taken on
    the current kernel sources; else None."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(path) as f:
            d = json.load(f)
        e = d[kernel][workload]
        if e.get("source_hash") != kernel_source_hash(kernel):
            return None
        return float(e["bytes_per_launch"])
    except Exception:
        return None


class Clocks:
    """nvidia-smi samples during the timed region."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.file = None

    def start(self):
        try:
            self.file = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.QUERY,
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=self.file, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
            return
        # the first sample lands before the timed region starts
        self._wait_rows(1, 5.0)

    def _rows(self):
        try:
            with open(self.file.name) as f:
                return sum(1 for line in f if line.count(",") >= 8)
        except Exception:
            return 0

    def _wait_rows(self, n, limit):
        t0 = time.time()
        while self.proc is not None and self.proc.poll() is None and self._rows() < n and time.time() - t0 < limit:
            time.sleep(0.02)

    def stop(self):
        if self.proc is None:
            return None
        # at least one sample after the timed region, however short it was
        self._wait_rows(self._rows() + 1, 2.0)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.file.flush()
        rows = []
        with open(self.file.name) as f:
            for line in f:
                parts = [x.strip() for x in line.split(",")]
                if len(parts) >= 9:
                    rows.append(parts)
        os.unlink(self.file.name)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({n for r in rows for n, v in zip(names, r[5:9]) if v == "Active"})
        return {"sm_mhz": float(np.median(sm)) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(rows)}


def naca_mask_device(w):
    from paper_2210_10377_gb300 import binding
    return binding.naca_mask(w.nx, w.ny, w.chord, w.thickness, w.alpha_deg, w.xc, w.yc)


def time_steps(torch, lat, steps):
    """Device time of `steps` steps: CUDA events on the handle's stream around
    the queued steps (lbm_step_async), then the wait and the status check."""
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(lat.stream)
    lat.step_async(steps)
    e1.record(lat.stream)
    lat.sync()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1)


# Stored FP64 oracle force series of the full-size workloads' first steps
# (written by tests/golden/make_prefix_series.py from the oracle alone):
# columns t, then F_x F_y of A, B, DRTT, A', SI.
PREFIX_SERIES = {
    "naca0012_4096x2048_c256_a4_re1000_f32":
        "naca0012_4096x2048_c256_a4_re1000_oracle_prefix5000.txt",
    "naca0012_8192x4096_c512_a6_re2000_f16dev":
        "naca0012_8192x4096_c512_a6_re2000_oracle_prefix1000.txt",
}
COEFF_SCHEMES = ("A", "B", "DRTT", "A_RTT", "SI")


def load_prefix(workload):
    """(t[n], F[5][2][n]) of the stored oracle series of a workload."""
    rows = np.loadtxt(os.path.join(ROOT, "tests", "golden", PREFIX_SERIES[workload]))
    t = rows[:, 0].astype(int)
    return t, rows[:, 1:].reshape(len(t), 5, 2).transpose(1, 2, 0)


def coeff_errors(lat, w, t, oracle_f, upto=None):
    """Drag and lift coefficients of every scheme (the library's
    lbm_coefficients) against the stored oracle series, at the stored steps
    below `upto` (default: all steps whose DRTT is complete).  Per step the
    error is relative to S(t) = max over compared steps s >= min(t, n/2) of
    max(|C_d(s)|, |C_l(s)|) of the oracle (the back half is judged against its
    largest coefficient; the force of the impulsive start sets the scale only
    for itself and its decay); the mean is over the back half of the compared
    steps, relative to max(|mean C_d|, |mean C_l|)."""
    upto = lat.steps_done - 1 if upto is None else upto
    keep = t < upto
    tk = t[keep]
    if tk.size < 2:
        return {"steps_compared": int(tk.size)}
    norm = 2.0 / (w.rho0 * w.u_in ** 2 * w.chord)
    out = {"steps_compared": int(tk.size), "last_step": int(tk[-1])}
    h = tk.size // 2
    for j, s in enumerate(COEFF_SCHEMES):
        cd, cl, _ = lat.coefficients(s, w.chord, w.u_in, 0, int(tk[-1]) + 1)
        g = np.stack([cd[tk], cl[tk]])
        o = norm * oracle_f[j][:, keep]
        mag = np.abs(o).max(axis=0)
        env = np.maximum.accumulate(mag[::-1])[::-1]
        env[h:] = env[h]
        per_step = float((np.abs(g - o).max(axis=0) / env).max())
        mo, mg = o[:, h:].mean(axis=1), g[:, h:].mean(axis=1)
        out[s] = {"per_step": per_step, "mean": float(np.abs(mg - mo).max() / np.abs(mo).max())}
    return out


def prefix_accuracy(binding, w, storage, device):
    """A run over the whole stored prefix of a workload: coefficient errors
    of every scheme (see coeff_errors)."""
    t, o = load_prefix(w.name)
    lat = binding.Lattice(naca_mask_device(w), w.tau, w.u_in, storage=storage, device=device)
    lat.step(int(t[-1]) + 2)
    out = {"workload": w.name, "storage": storage, "oracle_steps": "0..%d every %d" % (t[-1], t[1] - t[0])}
    out.update(coeff_errors(lat, w, t, o))
    lat.close()
    return out


def kernel_roofline(torch, lat, w, storage, steps, peak):
    lat.set_kernel_timing(True)
    lat.kernel_times(reset=True)
    lat.step(steps)
    kt = lat.kernel_times(reset=True)
    lat.set_kernel_timing(False)
    ms, n = kt["collide_stream"]
    avg_s = ms / n / 1e3
    algo = BYTES_PER_UPDATE[storage] * w.nodes
    achieved = algo / avg_s / 1e9
    return {"achieved": achieved, "peak": peak, "frac": achieved / peak,
            "avg_launch_us": avg_s * 1e6, "algorithmic_bytes": algo,
            "link_kernel_us": kt["link_force"][0] / kt["link_force"][1] * 1e3}


def pass_roofline(w, storage, ms, steps, launches, peak):
    """The multi-step kernel in a timed region of `steps` steps (None if it did
    not serve them: single steps launch two kernels each, a pass three).  The
    time of a pass is the region's, its link kernels running beside the next
    pass; its bytes are one read and one write of the state for four steps."""
    if launches >= steps or steps < PASS_STEPS:
        return None
    avg_s = ms / 1e3 * PASS_STEPS / steps
    algo = BYTES_PER_UPDATE[storage] * w.nodes
    achieved = algo / avg_s / 1e9
    return {"bound": "issue", "achieved": round(achieved, 1), "peak": peak, "unit": "GB/s",
            "frac": round(achieved / peak, 4), "traffic": ncu_traffic("march", w.name),
            "kernel": "k_march<%s>" % storage, "steps_per_launch": PASS_STEPS,
            "avg_launch_us": round(avg_s * 1e6, 2), "algorithmic_bytes_per_launch": algo}


def variant(torch, binding, w, storage, steps, peak, device):
    mask = naca_mask_device(w)
    lat = binding.Lattice(mask, w.tau, w.u_in, storage=storage, device=device)
    lat.step(20)
    ms = time_steps(torch, lat, steps)
    rl = kernel_roofline(torch, lat, w, storage, min(steps, 500), peak)
    lat.close()
    mlups = w.nodes * steps / (ms / 1e3) / 1e6
    return {"workload": w.name if storage == w.storage else w.name + "_as_" + storage,
            "storage": storage, "MLUPS": round(mlups, 1), "steps": steps,
            "ms_per_step": ms / steps, "bytes_per_update": BYTES_PER_UPDATE[storage],
            "collide_stream_GBps": round(rl["achieved"], 1),
            "frac_of_measured_hbm": round(rl["frac"], 4)}


def adjoint_variant(torch, binding, w, storage, steps, window, device):
    """Wall time of lbm_adjoint (forward with checkpoints, recompute, backward,
    gradients read back) against the forward steps alone, same start state."""
    mask = naca_mask_device(w)
    base = binding.Lattice(mask, w.tau, w.u_in, storage=storage, device=device)
    f0 = base.populations()
    base.close()
    out = {"workload": w.name if storage == w.storage else w.name + "_as_" + storage,
           "storage": storage, "steps": steps, "window": window,
           "checkpoint_every": "auto: the last L states kept in device memory (L from 60 % of the "
                               "memory torch can provide), the first steps - L checkpointed every "
                               "ceil(sqrt(steps - L)) steps"}
    for rep in range(2):  # the first pass warms allocator and graphs
        lat = binding.Lattice(mask, w.tau, w.u_in, storage=storage, device=device)
        lat.set_populations(f0)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        lat.step(steps)
        lat.force_series("B", steps - window, window)
        torch.cuda.synchronize()
        fwd = time.perf_counter() - t0
        lat.close()
        adj = {}
        for where in ("device", "host"):
            lat = binding.Lattice(mask, w.tau, w.u_in, storage=storage, device=device)
            lat.set_populations(f0)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            J, dtau, du, df0 = lat.adjoint(steps, window, 1.0, 0.0, want_df0=True,
                                           df0_device=where == "device")
            torch.cuda.synchronize()
            adj[where] = time.perf_counter() - t0
            lat.close()
            del df0
    out.update({"forward_ms": round(fwd * 1e3, 2), "adjoint_ms": round(adj["device"] * 1e3, 2),
                "adjoint_over_forward": round(adj["device"] / fwd, 2),
                "adjoint_MLUPS": round(w.nodes * steps / adj["device"] / 1e6, 1),
                "adjoint_ms_df0_to_host": round(adj["host"] * 1e3, 2),
                "J": J, "dJ_dtau": dtau,
                "includes": "forward keeping states and checkpoints, recompute of the checkpointed "
                            "segments, backward sweep, dJ/dtau and dJ/du_in[ny] read back, "
                            "dJ/df0[9][ny][nx] in FP64 "
                            "as a CUDA tensor (adjoint_ms) or copied to a host array "
                            "(adjoint_ms_df0_to_host)"})
    return out


def oracle_sample(w, seconds, mask=None):
    """The FP64 CPU oracle on the same workload, stepped until `seconds` pass."""
    import oracle
    if mask is None:
        mask = oracle.naca_mask(w.nx, w.ny, w.chord, w.thickness, w.alpha_deg, w.xc, w.yc)
    sim = oracle.Sim(mask, w.tau, w.u_in)
    sim.step(1)
    steps = 0
    t0 = time.perf_counter()
    while True:
        sim.step(1)
        steps += 1
        el = time.perf_counter() - t0
        if el >= seconds:
            break
    return w.nodes * steps / el / 1e6, steps, el


def oracle_band(w, rows):
    """A band of `rows` rows of the workload as its own channel domain with
    periodic y: a bounded sample of the workload for the oracle.  A band of at
    least half the height is centred on the mid-line and holds the whole
    airfoil; a narrower one takes the top rows, which are all fluid (a thin
    band through the airfoil would be a channel blocked by it)."""
    import oracle
    mask = oracle.naca_mask(w.nx, w.ny, w.chord, w.thickness, w.alpha_deg, w.xc, w.yc)
    rows = max(3, min(w.ny, int(rows)))
    y0 = (w.ny - rows) // 2 if 2 * rows >= w.ny else w.ny - rows
    return mask[y0:y0 + rows].copy(), y0


def run_reference(a):
    """The oracle arm: K timed steps after W warm-up steps, each step the FP64
    oracle advancing a band of rows of the workload, the band sized so that the
    whole run takes about `budget` seconds."""
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    import oracle
    from paper_2210_10377_gb300 import inputs
    w = inputs.LARGE_F32
    cores = oracle.set_threads(os.cpu_count() or 1)
    budget = a.ref_seconds if a.ref_seconds else min(120.0, max(10.0, 0.002 * (a.steps + a.warmup)))
    # calibrate the oracle's cost per node update on a 16-row band
    cal, _ = oracle_band(w, 16)
    sim = oracle.Sim(cal, w.tau, w.u_in)
    sim.step(1)
    t0 = time.perf_counter()
    sim.step(10)
    per_node = (time.perf_counter() - t0) / (10 * cal.size)
    del sim
    rows = budget / max(1, a.steps + a.warmup) / (per_node * w.nx)
    band, y0 = oracle_band(w, rows)
    sim = oracle.Sim(band, w.tau, w.u_in)
    for _ in range(a.warmup):
        sim.step(1)
    t0 = time.perf_counter()
    for _ in range(a.steps):
        sim.step(1)
    el = time.perf_counter() - t0
    mlups = band.size * a.steps / el / 1e6
    line = {"metric": "MLUPS", "value": round(mlups, 3), "unit": "MLUPS", "impl": "reference",
            "n_gpus": a.gpus, "steps": a.steps, "warmup": a.warmup, "ms_per_step": el / a.steps * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic",
            "config": {"workload": w.name, "nx": w.nx, "ny": w.ny, "chord": w.chord,
                       "alpha_deg": w.alpha_deg, "re": w.re, "tau": w.tau},
            "cpu_baseline": {"value": round(mlups, 3), "unit": "MLUPS", "cores": cores,
                             "kind": "oracle",
                             "sample": "FP64 oracle, node loops on %d host threads; each step advances the %dx%d band "
                                       "(rows %d-%d, %d solid nodes) of the workload as a channel "
                                       "of its own; %d steps after %d warm-up steps"
                                       % (cores, w.nx, band.shape[0], y0, y0 + band.shape[0] - 1,
                                          int(band.sum()), a.steps, a.warmup)},
            "e2e": {"value": round(mlups, 3), "unit": "MLUPS", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def run_ours(a):
    import torch

    from paper_2210_10377_gb300 import binding, inputs
    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    binding.lib()
    w = inputs.LARGE_F32
    storage = w.storage
    peak, peak_kind = measured_peaks()

    # -- device throughput: inputs resident, K steps between barriers.  The
    # force series is grown and every captured step graph built before the
    # warm-up (lbm_prepare), so the timed steps only launch.
    mask = naca_mask_device(w)
    lat = binding.Lattice(mask, w.tau, w.u_in, storage=storage, device=local)
    lat.prepare(a.warmup + a.steps + 2000)
    lat.step(a.warmup)
    clocks = Clocks(local)
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    clocks.start()
    launches0 = lat.launch_count
    ms = time_steps(torch, lat, a.steps)
    launches = lat.launch_count - launches0
    clk = clocks.stop()
    if world > 1:
        ms = reduce_max(ms, device="cuda")
        torch.distributed.barrier()
    value = world * w.nodes * a.steps / (ms / 1e3) / 1e6
    coeff = None
    if rank == 0:
        t_o, f_o = load_prefix(w.name)
        coeff = {"timed_run": coeff_errors(lat, w, t_o, f_o)}
    rl = kernel_roofline(torch, lat, w, storage, min(a.steps, 2000), peak)
    lat.close()
    if rank == 0:
        coeff["prefix"] = [prefix_accuracy(binding, w, storage, local)]
        if not a.no_variants:
            coeff["prefix"] += [prefix_accuracy(binding, w, "f32", local),
                                prefix_accuracy(binding, inputs.PRECISION, "f32dev", local),
                                prefix_accuracy(binding, inputs.PRECISION, "f16dev", local)]
        coeff["definition"] = ("C = 2F/(rho0 u_in^2 chord), every scheme, against the stored FP64 "
                               "oracle series; per_step: max over the compared steps of |dC| / S(t), "
                               "S(t) = max over compared steps s >= min(t, n/2) of max(|C_d(s)|, "
                               "|C_l(s)|); mean: "
                               "back half of the compared steps, |d mean| / max(|mean C_d|, |mean C_l|)")

    # -- end to end through the public API from pinned host buffers
    pm = torch.empty((w.ny, w.nx), dtype=torch.uint8, pin_memory=True)
    pm.numpy()[:] = mask
    schemes = ("A", "B", "DRTT", "A_RTT", "SI")
    fx = torch.empty((len(schemes), a.steps), dtype=torch.float64, pin_memory=True)
    fy = torch.empty((len(schemes), a.steps), dtype=torch.float64, pin_memory=True)
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    lat2 = binding.Lattice(pm.numpy(), w.tau, w.u_in, storage=storage, device=local)
    lat2.step(a.steps)
    for k, s in enumerate(schemes):
        gx, gy = lat2.force_series(s)
        fx.numpy()[k] = gx
        fy.numpy()[k] = gy
    lat2.close()
    torch.cuda.synchronize()
    e2e_s = time.perf_counter() - t0
    if world > 1:
        e2e_s = reduce_max(e2e_s, device="cuda")
    e2e = {"value": round(world * w.nodes * a.steps / e2e_s / 1e6, 1), "unit": "MLUPS",
           "h2d_bytes_per_step": round((w.nodes + 8) / a.steps, 3),
           "d2h_bytes_per_step": round(len(schemes) * 2 * 8, 3),
           "includes": "lbm_create from a pinned host mask (device set-up: mask, links, inlet rows, "
                       "initial state), lbm_step(K), every step's force of all five schemes read back "
                       "(the step's result), lbm_destroy"}

    variants = adjoint = batch = cyl = None
    if not a.no_variants and rank == 0:
        variants = [variant(torch, binding, w, "f64", 1000, peak, local),
                    variant(torch, binding, w, "f32dev", 4000, peak, local),
                    variant(torch, binding, w, "f16dev", 4000, peak, local),
                    variant(torch, binding, inputs.PRECISION, "f16dev", 2000, peak, local),
                    variant(torch, binding, inputs.PRECISION, "f32dev", 1000, peak, local)]
        adjoint = [adjoint_variant(torch, binding, inputs.DIFF, inputs.DIFF.storage, 4000, 1000, local),
                   adjoint_variant(torch, binding, w, w.storage, 1000, 500, local)]
        batch = [batch_variant(torch, binding, inputs, 256, "f32dev", 2000, peak, local),
                 batch_variant(torch, binding, inputs, 256, "f16dev", 2000, peak, local)]
        from paper_2210_10377_gb300 import cylinder
        t0 = time.perf_counter()
        cyl = cylinder.cd_study(device=local)
        cyl["wall_s"] = round(time.perf_counter() - t0, 2)
        t0 = time.perf_counter()
        cyl["cd_vs_re"] = cylinder.cd_vs_re(device=local)
        cyl["cd_vs_re"]["wall_s"] = round(time.perf_counter() - t0, 2)

    cpu = None
    if rank == 0 and world == 1:
        import oracle
        cores = os.cpu_count() or 1
        oracle.set_threads(1)
        m1, s1, e1 = oracle_sample(w, a.cpu_seconds / 2, mask)
        used = oracle.set_threads(cores)
        mlups, steps, el = oracle_sample(w, a.cpu_seconds / 2, mask)
        oracle.set_threads(1)
        cpu = {"value": round(mlups, 3), "unit": "MLUPS", "cores": used, "kind": "oracle",
               "single_thread": round(m1, 3),
               "sample": "FP64 oracle with its node loops on %d host threads (force, flux and momentum "
                         "sums on one, in their fixed order), %d steps of the full %dx%d grid after one "
                         "warm-up step (%.1f s); one thread: %d steps, %.1f s"
                         % (used, steps, w.nx, w.ny, el, s1, e1)}

    if rank == 0:
        single = {"bound": "hbm", "achieved": round(rl["achieved"], 1), "peak": peak,
                  "unit": "GB/s", "frac": round(rl["frac"], 4), "traffic": ncu_traffic("collide_stream", w.name),
                  "kernel": "k_collide_stream<%s>" % storage, "steps_per_launch": 1, "peak_source": peak_kind,
                  "avg_launch_us": round(rl["avg_launch_us"], 2),
                  "algorithmic_bytes_per_launch": rl["algorithmic_bytes"],
                  "link_kernel_us": round(rl["link_kernel_us"], 2)}
        timed = pass_roofline(w, storage, ms, a.steps, launches, peak)
        if timed:
            timed["peak_source"] = peak_kind
        line = {
            "metric": "MLUPS", "value": round(value, 1), "unit": "MLUPS", "n_gpus": world,
            "steps": a.steps, "warmup": a.warmup, "ms_per_step": ms / a.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": w.name, "nx": w.nx, "ny": w.ny, "chord": w.chord,
                       "thickness": w.thickness, "alpha_deg": w.alpha_deg, "re": w.re,
                       "tau": w.tau, "u_in": w.u_in, "storage": storage,
                       "forces_per_step": ["MEA_A", "MEA_B", "DRTT", "MEA_A_RTT"],
                       "l2": "inputs larger than L2 (3 rotating x %.0f MB population buffers)"
                             % (9 * 4 * w.nodes / 1e6),
                       "parallelism": "replicas%d" % world},
            "roofline": timed or single,
            "roofline_single_step": dict(single, in_timed_region=timed is None),
            "cpu_baseline": cpu,
            "coeff_error": coeff,
            "e2e": e2e,
            "gpu_launches": int(launches),
            "clocks": clk,
            "variants": variants,
            "adjoint": adjoint,
            "batch": batch,
            "cylinder": cyl,
        }
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


def batch_domains(binding, inputs, n):
    ws = inputs.batch_instances(256)[:n]
    return ws, [{"mask": binding.naca_mask(w.nx, w.ny, w.chord, w.thickness, w.alpha_deg, w.xc, w.yc),
                 "tau": w.tau, "u_in": w.u_in} for w in ws]


def batch_variant(torch, binding, inputs, n, storage, steps, peak, device):
    """The batching workload: n NACA00xx domains of uneven size in one batch,
    launch configuration from the tuner, `steps` steps timed with events."""
    ws, doms = batch_domains(binding, inputs, n)
    b = binding.Batch(doms, storage=storage, device=device)
    b.step(20)
    shape, k, tuned_ms = b.autotune(trials=5)
    b.step(32)
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(b.stream)
    b.step(steps)
    e1.record(b.stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / steps
    flags, _ = b.status()
    algo = BYTES_PER_UPDATE[storage] * b.nodes
    out = {"workload": "naca00xx_batch%d_seed%d" % (n, inputs.SEED), "storage": storage, "domains": n,
           "nodes": b.nodes, "steps": steps, "MLUPS": round(b.nodes / ms / 1e3, 1),
           "ms_per_step": round(ms, 4),
           "launch": {"tile": list(b.shape(shape)), "ctas_per_sm": k,
                      "form": "persistent" if k > 0 else "one CTA per tile"},
           "collide_stream_us": round(tuned_ms * 1e3, 1),
           "collide_stream_GBps": round(algo / (tuned_ms / 1e3) / 1e9, 1),
           "frac_of_measured_hbm": round(algo / (tuned_ms / 1e3) / 1e9 / peak, 4),
           "unstable_domains": int(flags.sum())}
    b.close()
    return out


def run_profile(a):
    """Warm-up + K steps of one workload and nothing else (the command that the
    committed ncu summaries were taken on)."""
    import torch

    from paper_2210_10377_gb300 import binding, inputs
    if a.batch:
        torch.cuda.set_device(0)
        ws, doms = batch_domains(binding, inputs, a.batch)
        b = binding.Batch(doms, storage=a.storage or "f32")
        if a.batch_launch:
            b.set_launch(*[int(v) for v in a.batch_launch.split(",")])
        else:
            b.autotune(trials=2)
        b.step(a.warmup)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        b.step(a.steps)
        torch.cuda.synchronize()
        el = time.perf_counter() - t0
        print(json.dumps({"workload": "naca00xx_batch%d" % a.batch, "nodes": b.nodes,
                          "launch": b.launch(), "steps": a.steps,
                          "MLUPS": round(b.nodes * a.steps / el / 1e6, 1)}), flush=True)
        b.close()
        return 0
    w = inputs.WORKLOADS[a.workload] if a.workload else inputs.LARGE_F32
    if a.shrink > 1:
        w = inputs.scaled(w, a.shrink)
    storage = a.storage or w.storage
    torch.cuda.set_device(0)
    lat = binding.Lattice(naca_mask_device(w), w.tau, w.u_in, storage=storage, kernel=a.kernel)
    if a.adjoint:
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        J, dtau, _, _ = lat.adjoint(a.adjoint, max(1, a.adjoint // 2), 1.0, 0.0, want_df0=False)
        torch.cuda.synchronize()
        print(json.dumps({"workload": w.name, "storage": storage, "adjoint_steps": a.adjoint,
                          "ms": round((time.perf_counter() - t0) * 1e3, 2), "J": J, "dJ_dtau": dtau}), flush=True)
        lat.close()
        return 0
    lat.step(a.warmup)
    ms = time_steps(torch, lat, a.steps)
    print(json.dumps({"workload": w.name, "storage": storage, "kernel": a.kernel, "steps": a.steps,
                      "MLUPS": round(w.nodes * a.steps / (ms / 1e3) / 1e6, 1),
                      "force_B": lat.force("B")}), flush=True)
    lat.close()
    return 0


def main():
    a = args_()
    if a.profile:
        return run_profile(a)
    if a.impl == "reference":
        return run_reference(a)
    return run_ours(a)


if __name__ == "__main__":
    sys.exit(main())
