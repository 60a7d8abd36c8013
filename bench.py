#!/usr/bin/env python3
"""Benchmark of the collision-aware local-global loop on GB300.

One step = one full solve of the three-finger gripper workload: reset to the
rest shape, then 200 outer iterations (collision check, spring update, local
step, RHS gather, PCG global solve) of 193,920 tets with a rigid sphere, in
MIXED precision.  The metric is tet-element iterations per second
(n_tets * n_iters / time).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl casim|reference]

``--impl reference`` times the FP64 CPU oracle (a bounded sample: one outer
iteration of the same workload per step) on the host cores.  With several GPUs
each rank runs an independent replica of the workload (a single mesh does not
shard); the value is the work of all ranks over the slowest rank's time.
"""
from __future__ import annotations

import argparse
import math
import hashlib
import json
import os
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

# The CPU legs (the FP64 oracle) may use every host core: numpy's BLAS and
# LAPACK read these before they load.
NPROC = os.cpu_count() or 1
for _v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
    os.environ.setdefault(_v, str(NPROC))

METRIC = "tet-element iterations/sec at 200k tets"
UNIT = "tet-iterations/s"
WORKLOAD = ("gripper3_plate_sphere: three 60x12x12-voxel pneumatic fingers (8 chambers each) "
            "below a 40x40x4-voxel plate, rigid sphere r=3cm, 193,920 tets, 200 outer iterations")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="casim", choices=["casim", "reference"])
    ap.add_argument("--iters", type=int, default=200, help="outer iterations per step")
    ap.add_argument("--only-plain", action="store_true",
                    help="time the single-robot workload only (no batched, adjoint or CPU legs; for profiling)")
    ap.add_argument("--only-batched", type=int, default=0, metavar="N",
                    help="run 2 warm-up and then N iterations of the 256-robot batch, print one line and exit "
                         "(for profiling)")
    return ap.parse_args()


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


# --------------------------------------------------------------------- clocks
class ClockSampler:
    """Samples nvidia-smi clocks and throttle reasons while running."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.rows = []
        self.proc = None
        self.th = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.th = threading.Thread(target=self._read, daemon=True)
        self.th.start()

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 9:
                self.rows.append(parts)

    def stop(self):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
        if self.th is not None:
            self.th.join(timeout=5)

    def summary(self):
        def num(x):
            try:
                return float(x)
            except ValueError:
                return None

        sm = [num(r[1]) for r in self.rows if num(r[1]) is not None]
        mx = [num(r[2]) for r in self.rows if num(r[2]) is not None]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = set()
        for r in self.rows:
            for k, nm in enumerate(names):
                if r[5 + k].lower().startswith("active"):
                    reasons.add(nm)
        sm_sorted = sorted(sm)
        med = sm_sorted[len(sm_sorted) // 2] if sm_sorted else None
        return {"sm_mhz": med, "sm_max_mhz": max(mx) if mx else None, "reasons": sorted(reasons),
                "samples": len(self.rows)}


# ------------------------------------------------------------------- roofline
def pcg_bytes_per_launch(n_free: int, nnz_row: float, k_pcg: float) -> float:
    """Algorithmic DRAM bytes of one PCG launch (FP32 vectors, 12 B per 3-vector,
    4 B per scalar, 8 B per off-diagonal entry): the initial residual pass
    (52 + 8 nnz), the first SpMV pass (40 + 8 nnz) and per iteration
    148 + 8 nnz bytes per free vertex (x, r, p, s, u, w each read and written
    once, the diagonal read once, the matrix row read once)."""
    return n_free * ((52 + 8 * nnz_row) + (40 + 8 * nnz_row) + k_pcg * (148 + 8 * nnz_row))


def offdiag_nnz_per_free_row(m) -> float:
    import numpy as np

    fixed = m.fixed.astype(bool)
    t = m.tets.astype(np.int64)
    pairs = []
    for a in range(4):
        for b in range(4):
            if a != b:
                pairs.append(np.stack([t[:, a], t[:, b]], axis=1))
    e = np.unique(np.concatenate(pairs), axis=0)
    e = e[~fixed[e[:, 0]] & ~fixed[e[:, 1]]]
    return e.shape[0] / max(1, int((~fixed).sum()))


def kernel_source_hash() -> str:
    """Hash of the PCG kernels' source: team.cu, cg.cuh, common.cuh and the lines of
    kernels.h that concern the PCG (its constants and launchers)."""
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2203_02054_gb300", "csrc")
    for f in ("team.cu", "cg.cuh", "common.cuh"):
        with open(os.path.join(csrc, f), "rb") as fh:
            h.update(fh.read())
    with open(os.path.join(csrc, "kernels.h")) as fh:
        h.update("".join(line for line in fh if "TEAM_" in line or "team" in line).encode())
    return h.hexdigest()[:16]


def recorded_traffic(kernel: str):
    """DRAM bytes per launch from the committed ncu summary, if it was taken
    from the current kernel source (else None)."""
    p = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(p) as fh:
            rec = json.load(fh).get(kernel)
    except (OSError, ValueError):
        return None
    if not rec or rec.get("source_hash") != kernel_source_hash():
        return None
    return rec.get("bytes_per_launch")


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    except (OSError, ValueError, KeyError):
        return 6800.0, "fallback"


def aggregate(ms_local: float, units_local: float, pg=None, device=None):
    """Whole-job throughput: the work of all ranks over the slowest rank's
    time (max over ranks of the timed milliseconds)."""
    import torch

    t = torch.tensor([ms_local, units_local], dtype=torch.float64, device=device)
    if pg is not None:
        mx = t[:1].clone()
        pg.all_reduce(mx, op=pg.ReduceOp.MAX)
        tot = t[1:].clone()
        pg.all_reduce(tot, op=pg.ReduceOp.SUM)
        ms, units = float(mx.item()), float(tot.item())
    else:
        ms, units = float(t[0].item()), float(t[1].item())
    return units / (ms / 1e3), ms


# ------------------------------------------------------------------ oracle arm
CONTACT_SAMPLE = ("one outer iteration of the 193,920-tet gripper from a seeded contact-bearing state "
                  "(rest + uniform noise of +-0.3 voxel edges on free vertices, seed 2203, FP32-rounded): "
                  "brute-force exact collision check, spring creation by ray casts, local step, "
                  "sparse LU global solve; FP64 numpy/scipy")


def contact_state(m):
    from paper_2203_02054_gb300 import synth
    import numpy as np

    return synth.perturbed_positions(m, 0.3, seed=2203, dtype=np.float32)


def oracle_sample(m, prep=None, X0=None):
    """One outer iteration of the FP64 oracle from X0 (default: the rest
    shape) with no prior springs; returns (wall seconds, tet-iterations,
    process CPU seconds, the iteration record)."""
    import numpy as np

    from oracle import loop, springs

    prep = prep or loop.prepare(m.rest, m.tets, m.group, m.fixed)
    st = springs.SpringState.empty(prep.query.shape[0])
    X = np.array(m.rest if X0 is None else X0)
    c0 = time.process_time()
    t0 = time.perf_counter()
    _x, _s, rec, _p, _o = loop.iterate(prep, X, st, m.alpha, m.spheres, m.w_knots, m.k_spring, m.eps, m.collision)
    return time.perf_counter() - t0, m.n_tets, time.process_time() - c0, rec


def cpu_model() -> str:
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.split(":")[0].strip() == "Model name":
                return line.split(":", 1)[1].strip()
    except (OSError, subprocess.SubprocessError):
        pass
    import platform

    return platform.processor() or platform.machine()


def cpu_baseline_record(value, wall, cpu, sample, extra=None):
    """cores = the host threads the oracle actually kept busy (process CPU
    time over wall time, rounded up), next to the cores it was allowed."""
    busy = cpu / wall if wall > 0 else 1.0
    rec = {"value": value, "unit": UNIT, "cores": max(1, int(math.ceil(busy - 0.05))), "kind": "oracle",
           "sample": sample, "cores_allowed": NPROC, "cpu_busy_ratio": busy, "cpu_model": cpu_model(),
           "blas_threads": os.environ.get("OPENBLAS_NUM_THREADS")}
    if extra:
        rec.update(extra)
    return rec


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    from paper_2203_02054_gb300 import synth
    from oracle import loop

    m = synth.config3_gripper()
    prep = loop.prepare(m.rest, m.tets, m.group, m.fixed)
    X0 = contact_state(m)
    for _ in range(args.warmup):
        oracle_sample(m, prep, X0)
    tot_t = tot_c = 0.0
    tot_u = 0
    rec = None
    for _ in range(args.steps):
        t, u, c, rec = oracle_sample(m, prep, X0)
        tot_t += t
        tot_c += c
        tot_u += u
    value = tot_u / tot_t
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * tot_t / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": {"workload": WORKLOAD, "n_tets": m.n_tets,
                                        "sample": "1 contact-bearing outer iteration per step"},
        "cpu_baseline": cpu_baseline_record(value, tot_t, tot_c, CONTACT_SAMPLE,
                                            {"self_pairs": rec.n_self_pairs, "springs": rec.n_springs}),
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    return 0


# ------------------------------------------------- batched and adjoint forms
def _event_ms(stream, fn):
    import torch

    a = torch.cuda.Event(enable_timing=True)
    b = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    a.record(stream)
    fn()
    b.record(stream)
    torch.cuda.synchronize()
    return a.elapsed_time(b)


def bench_batched(stream, plain_value, n_iters=100, n_seq=16):
    """256 independent fingers (12.1M tets) in one simulation, 100 iterations
    per step, against the same robots solved one after another (a seeded
    subset of ``n_seq`` robots, scaled by tets)."""
    import numpy as np

    from paper_2203_02054_gb300 import casim, synth

    batch = synth.config4_batch(n_iters=n_iters)
    n_t = sum(m.n_tets for m in batch)
    sim = casim.Sim(batch, stream=stream.cuda_stream, stats=0, tuned=True)
    kern = sim.stats().pcg_kernel
    step = lambda: (casim.casim_reset(sim.h), casim.casim_step(sim.h, n_iters))
    casim.casim_reset(sim.h)
    casim.casim_step(sim.h, 5)
    casim.casim_sync(sim.h)
    ms = _event_ms(stream, step)
    status = casim.casim_sync(sim.h)
    st = casim.casim_get_stats(sim.h)
    tuned = sim.tuned_from
    sim.close()
    rng = np.random.default_rng(1004)
    sub = sorted(rng.choice(len(batch), n_seq, replace=False).tolist())
    seq_ms = 0.0
    seq_t = 0
    for r in sub:
        one = casim.Sim(batch[r], stream=stream.cuda_stream, stats=0)
        f = lambda: (casim.casim_reset(one.h), casim.casim_step(one.h, n_iters))
        casim.casim_step(one.h, 2)
        casim.casim_sync(one.h)
        seq_ms += _event_ms(stream, f)
        seq_t += batch[r].n_tets
        one.close()
    value = n_t * n_iters / (ms / 1e3)
    seq_value = seq_t * n_iters / (seq_ms / 1e3)
    return {"workload": "256 pneumatic fingers (20k x 4k x 4k voxels, k~U{1..4}, 4-10 chambers), "
                        "12,119,040 tets, self-collision per robot", "n_robots": len(batch), "n_tets": n_t,
            "n_iters": n_iters, "value": value, "unit": UNIT, "ms_per_step": ms, "device_status": status,
            "pcg_kernel": kern, "tuned": tuned,
            "k_pcg_max_mean": st.total_pcg_iters / max(1, st.iterations) / len(batch),
            "sequential": {"robots": n_seq, "value": seq_value, "how": "each robot alone, same GPU, scaled by tets"},
            "vs_sequential": value / seq_value, "vs_plain": value / plain_value}


def bench_adjoint(stream, n_iters=100, every=10):
    """Adjoint workload: 983,040-tet finger (160x32x32, 16 chambers), loss on
    64 tip vertices, checkpointed forward + reverse pass through 100
    iterations, against the plain forward of the same iterations."""
    import numpy as np

    from paper_2203_02054_gb300 import casim, synth

    m = synth.config5_adjoint(n_iters=n_iters)
    sim = casim.Sim(m, stream=stream.cuda_stream, stats=0)
    casim.casim_step(sim.h, 2)
    casim.casim_sync(sim.h)
    fwd_ms = _event_ms(stream, lambda: (casim.casim_reset(sim.h), casim.casim_step(sim.h, n_iters)))
    ck_ms = _event_ms(stream, lambda: (casim.casim_reset(sim.h), casim.casim_forward_ckpt(sim.h, n_iters, every)))
    X = sim.positions()
    gX = np.zeros_like(X)
    gX[m.tip_verts] = 2.0 * (X[m.tip_verts] - m.tip_targets)
    t0 = time.perf_counter()
    grad = casim.casim_backward(sim.h, gX, m.n_groups)
    bwd_ms = 1e3 * (time.perf_counter() - t0)
    sim.close()
    plain = m.n_tets * n_iters / (fwd_ms / 1e3)
    value = m.n_tets * n_iters / ((ck_ms + bwd_ms) / 1e3)
    return {"workload": "finger 160x32x32 voxels, 16 chambers, 983,040 tets; loss on 64 tip vertices; "
                        "checkpoint every 10", "n_tets": m.n_tets, "n_iters": n_iters, "value": value,
            "unit": UNIT + " (forward + backward)", "forward_ms": ck_ms, "backward_ms": bwd_ms,
            "plain_forward_value": plain, "vs_plain_forward": value / plain,
            "grad_finite": bool(np.all(np.isfinite(grad))), "grad_norm": float(np.linalg.norm(grad))}


def bench_anderson(stream, n_iters=200, mem=5):
    """Anderson acceleration (memory 5, energy safeguard) against the plain
    loop on the 51,840-tet finger: Eq. 8 energy per iteration, iterations to
    come within 1e-2 / 1e-3 of the lower of the two runs' final energies, and
    time per iteration (both timed around synchronous calls: the accelerated
    loop synchronises every iteration)."""
    import numpy as np

    from paper_2203_02054_gb300 import casim, synth

    m = synth.config2_finger()
    res = {"workload": "finger 60x12x12 voxels, 8 chambers, 51,840 tets, self collision, %d iterations" % n_iters,
           "n_tets": m.n_tets, "n_iters": n_iters, "memory": mem}
    energies = {}
    for mm in (0, mem):
        sim = casim.Sim(m, stream=stream.cuda_stream)
        casim.casim_step(sim.h, 2)
        casim.casim_sync(sim.h)
        casim.casim_reset(sim.h)
        casim.casim_set_actuation(sim.h, m.alpha)
        casim.casim_sync(sim.h)
        t0 = time.perf_counter()
        if mm == 0:
            casim.casim_step(sim.h, n_iters)
            acc = 0
        else:
            _recs, acc = casim.casim_step_anderson(sim.h, n_iters, mm)
        casim.casim_sync(sim.h)
        dt = time.perf_counter() - t0
        E = np.array([h["energy"] for h in sim.history(cap=4096)][-n_iters:])
        energies[mm] = E
        key = "plain" if mm == 0 else "anderson"
        res[key] = {"ms_per_iter": 1e3 * dt / n_iters, "accepted": acc, "final_energy": float(E[-1])}
        sim.close()
    e_min = min(float(energies[0].min()), float(energies[mem].min()))
    for tol in (1e-2, 1e-3):
        for mm, key in ((0, "plain"), (mem, "anderson")):
            hit = np.nonzero(energies[mm] <= e_min * (1.0 + tol))[0]
            res[key]["iters_to_%g" % tol] = int(hit[0]) + 1 if hit.size else None
    return res


def bench_broad_phase(stream):
    """The two broad phases on the finger (51,840 tets, 100 iterations) and
    the gripper (193,920 tets, 200 iterations): CUDA-event phase split of the
    collision check and spring update per outer iteration, and the whole
    loop's time per outer iteration (graph replay), for the per-iteration
    spatial hash (0) and the AABB trees refitted every iteration (1)."""
    from paper_2203_02054_gb300 import casim, synth

    out = {}
    for name, m in (("finger_51840", synth.config2_finger()), ("gripper_193920", synth.config3_gripper())):
        rec = {}
        for broad in (0, 1):
            sim = casim.Sim(m, stream=stream.cuda_stream, stats=0, broad_phase=broad)
            casim.casim_step(sim.h, 3)
            casim.casim_sync(sim.h)
            ms = _event_ms(stream, lambda: (casim.casim_reset(sim.h), casim.casim_step(sim.h, m.n_iters)))
            sim.close()
            prof = casim.Sim(m, stream=stream.cuda_stream, stats=2, broad_phase=broad)
            prof.step(m.n_iters)
            prof.sync()
            ph = casim.casim_get_phase_times(prof.h) / m.n_iters
            prof.close()
            rec["hash" if broad == 0 else "aabb_tree"] = {
                "ms_per_iter": ms / m.n_iters, "collision_ms_per_iter": float(ph[0]),
                "springs_ms_per_iter": float(ph[1])}
        out[name] = rec
    return out


# -------------------------------------------------------------------- GPU arm
def run_only_batched(n_iters: int) -> int:
    import torch

    from paper_2203_02054_gb300 import casim, synth

    torch.cuda.set_device(0)
    stream = torch.cuda.current_stream(0)
    batch = synth.config4_batch(n_iters=n_iters)
    sim = casim.Sim(batch, stream=stream.cuda_stream, stats=0, tuned=True)
    casim.casim_step(sim.h, 2)
    casim.casim_sync(sim.h)
    st0 = casim.casim_get_stats(sim.h)
    ms = _event_ms(stream, lambda: casim.casim_step(sim.h, n_iters))
    status = casim.casim_sync(sim.h)
    st1 = casim.casim_get_stats(sim.h)
    hist = sim.history(cap=4096)[-n_iters:]
    n_t = sum(m.n_tets for m in batch)
    k_max = sum(h["pcg_iters"] for h in hist) / max(1, len(hist))   # per launch: the slowest robot
    k_mean = (st1.total_pcg_iters - st0.total_pcg_iters) / max(1, n_iters) / len(batch)
    print(json.dumps({"workload": "256-robot batch, %d tets" % n_t, "n_iters": n_iters, "ms": ms,
                      "ms_per_iter": ms / max(1, n_iters), "pcg_kernel": sim.stats().pcg_kernel,
                      "k_pcg_max_per_launch": k_max, "k_pcg_mean_per_robot": k_mean,
                      "device_status": status}))
    sim.close()
    return 0


def main():
    args = parse()
    if args.only_batched > 0:
        return run_only_batched(args.only_batched)
    if args.impl == "reference":
        return run_reference(args)
    rank, world, local = dist_env()
    import numpy as np
    import torch

    from paper_2203_02054_gb300 import casim, synth

    torch.cuda.set_device(local)
    pg = None
    if world > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl")
        pg = dist
    stream = torch.cuda.current_stream()
    m = synth.config3_gripper(n_iters=args.iters)
    n_iters = args.iters
    # the autotuner's cached winners for this GPU and workload shape, if any
    # (paper_2203_02054_gb300/tuned.json): what a user of casim.Sim(tuned=True) runs
    sim = casim.Sim(m, stream=stream.cuda_stream, stats=0, tuned=True)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")

    def one_step():
        casim.casim_reset(sim.h)
        casim.casim_step(sim.h, n_iters)

    for _ in range(max(args.warmup, 0)):
        one_step()
    st = casim.casim_sync(sim.h)
    if st != 0:
        print("warning: device status %d after warm-up" % st, file=sys.stderr)

    def barrier():
        if pg is not None:
            pg.barrier()
        torch.cuda.synchronize()

    sampler = ClockSampler(torch.cuda.current_device()) if rank == 0 else None
    barrier()
    if sampler:
        sampler.start()
    evs = []
    for _ in range(args.steps):
        flush.zero_()                     # L2 flush between timed steps (not timed)
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        one_step()
        b.record(stream)
        evs.append((a, b))
    barrier()
    if sampler:
        sampler.stop()
    status = casim.casim_sync(sim.h)
    ms = sum(a.elapsed_time(b) for a, b in evs)
    units = float(m.n_tets) * n_iters * args.steps * world
    value, ms_max = aggregate(ms, float(m.n_tets) * n_iters * args.steps, pg, "cuda")
    stats = casim.casim_get_stats(sim.h)
    # query vertices + 3 of the faces' hash + narrow phase + spring update + ray casts + local step + RHS gather + PCG; the
    # team PCG (kernel 5) finalizes the iteration itself, the others need 1 launch more
    kernels_per_iter = 10 if stats.pcg_kernel == 5 else 11
    gpu_launches = kernels_per_iter * n_iters * args.steps
    hist = casim.casim_get_history(sim.h, n_iters)

    # ---- end-to-end through the public API with host buffers ----
    rest = np.ascontiguousarray(m.rest)
    alpha = np.ascontiguousarray(m.alpha)
    out = np.empty_like(rest)
    barrier()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        casim.casim_reset(sim.h)
        casim.casim_set_positions(sim.h, rest)
        casim.casim_set_actuation(sim.h, alpha)
        casim.casim_step(sim.h, n_iters)
        casim.casim_get_positions(sim.h, m.n_verts)
    barrier()
    e2e_s = time.perf_counter() - t0
    e2e_value, _ = aggregate(1e3 * e2e_s, float(m.n_tets) * n_iters * args.steps, pg, "cuda")
    del out

    line = None
    if rank == 0:
        # ---- roofline of the dominant kernel: eager pass with phase events ----
        prof = casim.Sim(m, stream=stream.cuda_stream, stats=2, tuned=True)
        prof.step(n_iters)
        prof.sync()
        ph = casim.casim_get_phase_times(prof.h)
        pst = casim.casim_get_stats(prof.h)
        prof.close()
        k_pcg = pst.total_pcg_iters / max(1, pst.iterations)
        pcg_ms = ph[4] / n_iters
        nnz = offdiag_nnz_per_free_row(m)
        n_free = int((m.fixed == 0).sum())
        bpl = pcg_bytes_per_launch(n_free, nnz, k_pcg)
        peak, peak_kind = load_peaks()
        achieved = bpl / (pcg_ms / 1e3) / 1e9
        clocks = sampler.summary() if sampler else None
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_max / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64-reductions", "data": "synthetic",
            "config": {"workload": WORKLOAD, "n_tets": m.n_tets, "n_verts": m.n_verts, "n_iters": n_iters,
                       "precision": "MIXED (FP32 vectors/targets, FP64 dots, exact predicates)",
                       "l2": "flushed between timed steps (256 MiB write); one step's working set fits L2",
                       "parallelism": "replicas" if world > 1 else "single-gpu",
                       "tuned": sim.tuned_from, "device_status": status},
            "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": 8 * 3 * m.n_verts + 8 * m.n_groups,
                    "d2h_bytes_per_step": 8 * 3 * m.n_verts},
            "gpu_launches": gpu_launches,
            "roofline": {"bound": "hbm", "kernel": {1: "k_pcg (streaming)", 2: "k_pcg_rr (register-resident)",
                                                    3: "k_pcg_cluster", 4: "k_pcg_seg (segmented)",
                                                    5: "k_pcg_team (vectors on chip, two-level preconditioner)"}
                         .get(stats.pcg_kernel, "k_pcg"),
                         "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                         "peak_kind": peak_kind, "traffic": recorded_traffic("k_pcg"),
                         "bytes_per_launch": bpl, "ms_per_launch": pcg_ms, "k_pcg_mean": k_pcg,
                         "phase_ms_per_iter": {"collision": ph[0] / n_iters, "springs": ph[1] / n_iters,
                                               "local": ph[2] / n_iters, "rhs": ph[3] / n_iters,
                                               "pcg": ph[4] / n_iters}},
            "clocks": clocks,
            "solver": {"k_pcg_mean_timed": stats.total_pcg_iters / max(1, stats.iterations),
                       "device_status_bits": stats.status_bits,
                       "pairs_truncated": bool(stats.status_bits & 16),
                       "last_step": {"max_self_pairs": max(h["n_self_pairs"] for h in hist),
                                     "max_obstacle_pairs": max(h["n_obstacle_pairs"] for h in hist),
                                     "iters_with_obstacle_contact": sum(1 for h in hist if h["n_obstacle_pairs"]),
                                     "max_springs": max(h["n_springs"] for h in hist),
                                     "final_springs": hist[-1]["n_springs"]}},
        }
        if args.only_plain:
            print(json.dumps(line))
            sim.close()
            return 0
        line["batched"] = bench_batched(stream, value)
        line["adjoint"] = bench_adjoint(stream)
        try:
            line["broad_phase"] = bench_broad_phase(stream)
        except Exception as e:  # a failure here must not cost the main line
            line["broad_phase"] = {"error": "%s: %s" % (type(e).__name__, e)}
        try:
            line["anderson"] = bench_anderson(stream)
        except Exception as e:  # a failure here must not cost the main line
            line["anderson"] = {"error": "%s: %s" % (type(e).__name__, e)}
        # ---- CPU baseline: the oracle on bounded samples of the same workload ----
        from oracle import loop as oloop

        prep = oloop.prepare(m.rest, m.tets, m.group, m.fixed)
        t_c, u_c, c_c, rec_c = oracle_sample(m, prep, contact_state(m))
        t_r, u_r, c_r, _rec_r = oracle_sample(m, prep)
        line["cpu_baseline"] = cpu_baseline_record(
            u_c / t_c, t_c, c_c, CONTACT_SAMPLE,
            {"self_pairs": rec_c.n_self_pairs, "springs": rec_c.n_springs,
             "from_rest": {"value": u_r / t_r, "unit": UNIT, "cpu_busy_ratio": c_r / t_r,
                           "sample": "one outer iteration from the rest shape (no contacts)"}})
        print(json.dumps(line))
    sim.close()
    if pg is not None:
        pg.barrier()
        pg.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
