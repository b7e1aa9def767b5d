#!/usr/bin/env python
"""Benchmark of the explicit MMFD step on one GB300 (or N replicas under torchrun).

Workload (default): tgv2d_4096 -- 4096x4096 periodic He-Luo NSE, D2Q9, two-level MMFD,
Taylor-Green vortex (Re 100), FP32 storage.  One bench step = one MMFD time step over the
whole grid (16.8M lattice-node updates).  The level buffers (201 MB each) exceed the 129 MB
L2, so no L2 flush is needed between steps.

Prints one JSON line (rank 0).  --impl reference times the FP64 CPU oracle instead.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import re
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "MLUPS and % of HBM roofline per MMFD step; served p50/p99 latency vs plain FP32"
UNIT = "MLUPS"
SMI_QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def max_over_ranks(x: float, device: str = "cpu") -> float:
    """Maximum of x over the ranks of the default process group (x itself without one)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_mlups(ranks: int, nodes_per_rank: int, steps: int, seconds: float) -> float:
    """Whole-job throughput: every rank advances its own grid `steps` times in `seconds`
    (the slowest rank's time), so the job updates ranks x nodes x steps lattice nodes."""
    return ranks * nodes_per_rank * steps / seconds / 1e6


L2_BYTES = 129e6           # GB300 L2 capacity: workloads whose levels fit are reported as L2-resident
NOMINAL_HBM_GBS = 7900.0   # GB300 HBM3e, nominal (the measured copy bandwidth is the denominator of frac)


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


# The sources that determine the step kernels a solver may run under each kernel name it reports (the
# family's name: FP32 levels of the NSE families, FP64 levels and NCDE solves run kernels of their own in
# class form), and their launches.  The traffic figure of a committed profile is used only while
# these files and everything they include are unchanged.
COMMON_SOURCES = ["tune.cpp", "tma_host.cpp", "params.cpp"]   # work-item heights, tensor-map boxes, which form applies
KERNEL_SOURCES = {
    "k_march2d": ["k_march2d.cu", "k_march2d_nse.cu", "k_march_ncde.cu"],
    "k_march2d_tb": ["k_march2d_tb.cu"],
    "k_march2d_nse_s": ["k_march_lean.cu", "k_march2d_nse.cu"],
    "k_march2d_nse_g": ["k_march_lean.cu"],
    "k_march2d_tb_nse": ["k_march2d_tb_nse.cu", "k_march2d_nse.cu"],
    "k_march2d_src": ["k_march2d_src.cu"],
    "k_march3d": ["k_march3d.cu", "k_march3d_nse.cu", "k_march_ncde.cu"],
    "k_march3d_nse_s": ["k_march_lean.cu", "k_march3d_nse.cu"],
    "k_march3d_nse_g": ["k_march_lean.cu"],
    "k_march3d_src": ["k_march3d_src.cu"],
    "k_direct": ["k_direct.cu", "k_cluster.cu"],
    "k_direct_src": ["k_direct_src.cu"],
    # one theta-scheme step: the first pass and the fused sweeps, or the right-hand side and single sweeps,
    # issued by solver.cpp; the traffic entry also records the sweep count it was taken at
    "k_march2d_theta": ["k_march2d_theta.cu", "k_march2d_src.cu", "k_march2d.cu", "solver.cpp"],
}
CSRC = os.path.join(ROOT, "paper_2505_17057_gb300", "csrc")


def kernel_sources(kernel: str):
    """The source files of a kernel name, with everything they include (sorted; all files for an unknown name)."""
    todo = list(COMMON_SOURCES) + KERNEL_SOURCES.get(kernel, [f for f in os.listdir(CSRC)])
    seen = set()
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        with open(os.path.join(CSRC, f)) as fh:
            for inc in re.findall(r'^\s*#\s*include\s+"([^"]+)"', fh.read(), flags=re.M):
                if os.path.exists(os.path.join(CSRC, inc)):
                    todo.append(inc)
    return sorted(seen)


def kernel_source_sha(kernel: str) -> str:
    h = hashlib.sha256()
    for f in kernel_sources(kernel):
        with open(os.path.join(CSRC, f), "rb") as fh:
            h.update(f.encode() + fh.read())
    return h.hexdigest()[:16]


def traffic_from_profile(kernel: str, workload: str, depth: int = 1, sweeps: int = 0, storage: str = "fp32"):
    """DRAM bytes per launch from the committed ncu summary, if it was taken on this source, with
    this storage, at this temporal depth and (theta-scheme) with this many Jacobi sweeps per step.
    Keys are "workload:kernel" for FP32 storage and "workload:kernel:storage" otherwise."""
    p = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(p):
        return None
    with open(p) as fh:
        d = json.load(fh)
    e = d.get(f"{workload}:{kernel}" + ("" if storage == "fp32" else f":{storage}"))
    if not e or e.get("source_sha") != kernel_source_sha(kernel) or e.get("temporal_depth", 1) != depth:
        return None
    if e.get("sweeps", 0) != sweeps:
        return None
    return e.get("dram_bytes_per_launch")


def e2e_two_streams(mmfd, desc_kw, s0, fields, host_ptrs, back_ptrs, steps, nodes):
    """The end-to-end job (upload the level from page-locked host memory, advance it one step,
    read the stepped level back into page-locked host memory) on two solvers, each on its own
    stream and driven by its own host thread, so that one job's upload overlaps the other's
    read-back over the host link (the read-back call is synchronous).  Returns the aggregate MLUPS
    of both and the per-job bytes."""
    import threading
    import torch
    s1 = mmfd.Solver(mmfd.make_desc(**desc_kw), stream=torch.cuda.Stream())
    try:
        s1.set_fields(fields)
        back1 = [torch.empty(tuple(f.shape), dtype=torch.float32).pin_memory() for f in fields]
        jobs = [(s0, back_ptrs), (s1, [b.data_ptr() for b in back1])]

        def job(sv, back):
            mmfd.mmfd_set_fields(sv.h, 0, host_ptrs, mmfd.MMFD_HOST, mmfd.MMFD_DT_F32)
            sv.step(1)
            mmfd.mmfd_fields(sv.h, 0, back, mmfd.MMFD_HOST, mmfd.MMFD_DT_F32)

        for sv, back in jobs:   # warm both solvers (first-launch set-up happens here, one thread)
            job(sv, back)
        torch.cuda.synchronize()

        errors = []

        def worker(sv, back):
            try:
                for _ in range(steps):
                    job(sv, back)
            except Exception as e:   # reported after the join: a failed job voids the figure
                errors.append(e)

        threads = [threading.Thread(target=worker, args=j) for j in jobs]
        t0 = time.perf_counter()
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        secs = time.perf_counter() - t0
        if errors:
            raise errors[0]
    finally:
        s1.close()
    return {"value": 2 * steps * nodes / secs / 1e6, "unit": UNIT, "jobs": 2 * steps,
            "how": "two solvers on two streams, one host thread each; every job uploads the level, "
                   "steps it once and reads the stepped level back (FP32, page-locked host memory)"}


CLOCK_WINDOW_S = 1.0   # untimed launches after a timed region, so that the clock record sees the load


def l2_note(device_bytes: float, levels: int):
    """The config's statement about L2 and the roofline's bound: levels larger than the L2 are
    streamed from HBM each step (no flush needed); levels that fit are L2-resident, reported in
    MLUPS only."""
    if device_bytes > L2_BYTES:
        return f"inputs larger than L2 ({device_bytes / levels / 1e6:.0f} MB per level), no flush", "hbm"
    return (f"L2-resident ({device_bytes / 1e6:.0f} MB of levels in the {L2_BYTES / 1e6:.0f} MB L2): "
            "MLUPS only, the HBM roofline does not bound it", "l2-resident")


def clock_window_calls(ms_per_call: float) -> int:
    """Calls of the timed region's launch group that fill about CLOCK_WINDOW_S."""
    return max(1, int(CLOCK_WINDOW_S * 1e3 / max(ms_per_call, 1e-3)))


def clock_window(step_fn, ms_per_call):
    """Keep the GPU on the timed region's launches for about CLOCK_WINDOW_S after it (untimed),
    so that the clock samples, taken every 200 ms, see this load even when the timed region is
    shorter than one sampling interval."""
    import torch
    step_fn(clock_window_calls(ms_per_call))
    torch.cuda.synchronize()


class ClockSampler:
    def __init__(self, device_index: int):
        self.fh = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.proc = None
        self.dev = device_index

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.dev}", f"--query-gpu={SMI_QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.fh, stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None
            return
        # wait (at most 3 s) for the first sample, so that sampling is live when the timed region
        # starts
        t0 = time.perf_counter()
        while time.perf_counter() - t0 < 3.0 and os.path.getsize(self.fh.name) == 0:
            time.sleep(0.02)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.fh.flush()
        self.fh.seek(0)
        sms, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.fh.read().strip().splitlines():
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sms.append(float(parts[1]))
                mx = float(parts[2])
            except ValueError:
                continue
            for name, val in zip(names, parts[5:9]):
                if val.lower() == "active":
                    reasons.add(name)
        os.unlink(self.fh.name)
        return {"sm_mhz": statistics.median(sms) if sms else None, "sm_max_mhz": mx,
                "samples": len(sms), "reasons": sorted(reasons)}


class OracleTimer:
    """The FP64 CPU oracle (as it stands) on the bench workload: whole steps of the full grid on
    every host core, and a node-range sample of one step on one core."""

    def __init__(self, workload: str):
        from oracle import oracle as orc
        from oracle import params as P
        from paper_2505_17057_gb300 import configs
        self.orc = orc
        self.cores = os.cpu_count() or 1
        orc.set_threads(self.cores)
        if not workload.startswith("tgv2d"):
            raise ValueError(workload)
        n = int(workload.split("_")[1])
        desc, fields, _ = configs.tgv2d_4096(n=n)
        self.prob = P.problem_nse("D2Q9", 2, [n, n], 1.0, [1.0, 1.0], desc["a"], desc["abar"])
        self.n = n
        self.fields = fields
        self.stepper = None
        self.sampler = None

    def full_step(self) -> float:
        """Seconds for one whole oracle step of the n x n grid on every core (the level advances)."""
        if self.stepper is None:
            self.stepper = self.orc.LevelStepper(self.prob, self.fields)
        self.orc.set_threads(self.cores)
        t0 = time.perf_counter()
        self.stepper.step(1)
        return time.perf_counter() - t0

    def one_thread(self, seconds: float):
        """(MLUPS, sample) of the oracle on one core over a node-range sample of about `seconds`."""
        if self.sampler is None:
            self.sampler = self.orc.NodeSampler(self.prob, self.fields)
        self.orc.set_threads(1)
        try:
            n = self.n
            self.sampler.run(0, n)                       # warm caches
            t0 = time.perf_counter()
            self.sampler.run(0, 4 * n)
            t = max(time.perf_counter() - t0, 1e-6)
            rows = max(4, min(n, int(4 * seconds / t)))
            t0 = time.perf_counter()
            self.sampler.run((n // 3) * n, rows * n)
            t = time.perf_counter() - t0
        finally:
            self.orc.set_threads(self.cores)
        return rows * n / t / 1e6, (f"rows {n // 3}..{n // 3 + rows - 1} ({rows * n} nodes) of one MMFD step of the "
                                    f"{n}x{n} grid, direct form, 1 thread")

    def measure(self, steps: int = 3):
        """(MLUPS, sample) over `steps` whole steps on every core, after one warm-up step."""
        self.full_step()
        t = sum(self.full_step() for _ in range(steps))
        return steps * self.n * self.n / t / 1e6, (f"{steps} whole MMFD steps of the {self.n}x{self.n} grid, "
                                                    f"direct form, {self.cores} OpenMP threads")


def serving_bench(count, seed, mmfd, stream, budget_gb=40.0, slots=64, steps_per_tick=16):
    """Config 5: a seeded Poisson stream of mixed CDE/NCDE/NSE solves.

    plain: each request alone through the single-solve API (create, upload, step, read back),
    first-come first-served, under the same open-loop arrivals as the server (measured).
    served: the continuous-batching server, real time, open-loop arrivals.
    Arrival rate: 0.8 x the plain path's capacity.
    """
    import numpy as np
    from paper_2505_17057_gb300 import serving

    reqs = serving.make_stream(count, seed=seed, storage_mix=True)
    total_lu = float(sum(r.nodes * r.steps for r in reqs))
    # plain per-solve FP32
    service, plain_out = [], []
    for r in reqs:
        d = dict(r.desc)
        d["storage"] = "fp32"
        t0 = time.perf_counter()
        s = mmfd.Solver(mmfd.make_desc(**d), stream=stream)
        s.set_fields(r.fields)
        s.step(r.steps)
        out = s.fields(0)
        s.close()
        service.append(time.perf_counter() - t0)
        plain_out.append(out)
    capacity = count / sum(service)
    arrivals = serving.poisson_arrivals(count, 0.8 * capacity, seed=seed)

    def plain_open_loop():
        # the plain path under the same open-loop arrivals as the server: requests are taken in
        # arrival order, one at a time, each as soon as it has arrived and the previous one is done
        finish = np.zeros(count)
        t0 = time.perf_counter()
        for k, r in enumerate(reqs):
            wait = arrivals[k] - (time.perf_counter() - t0)
            if wait > 0:
                time.sleep(wait)
            d = dict(r.desc)
            d["storage"] = "fp32"
            s = mmfd.Solver(mmfd.make_desc(**d), stream=stream)
            s.set_fields(r.fields)
            s.step(r.steps)
            s.fields(0)
            s.close()
            finish[k] = time.perf_counter() - t0
        return finish - arrivals, float(finish.max() - arrivals[0])

    plain_lat, plain_makespan = plain_open_loop()

    def served(storage_mode):
        srv = mmfd.Server(int(budget_gb * (1 << 30)), max_slots=slots, steps_per_tick=steps_per_tick,
                          use_graphs=True, stream=stream)
        descs = []
        for r in reqs:
            d = dict(r.desc)
            if storage_mode == "fp32":
                d["storage"] = "fp32"
            descs.append(mmfd.make_desc(**d))
        finish = np.zeros(count)
        outs = [None] * count
        pending = {}
        i, done = 0, 0
        t0 = time.perf_counter()
        while done < count:
            now = time.perf_counter() - t0
            while i < count and arrivals[i] <= now:
                pending[srv.submit(descs[i], reqs[i].fields, reqs[i].steps)] = i
                i += 1
            progressed = False
            for t in list(pending):
                rc, res = srv.poll(t)
                if rc == mmfd.MMFD_OK:
                    k = pending.pop(t)
                    outs[k] = srv.result(t)
                    finish[k] = time.perf_counter() - t0
                    srv.release(t)
                    done += 1
                    progressed = True
            if not pending and i < count:
                wait = arrivals[i] - (time.perf_counter() - t0)
                if wait > 0:
                    time.sleep(min(wait, 0.001))
            elif not progressed:
                time.sleep(0.0001)
        st = srv.stats()
        srv.close()
        lat = finish - arrivals
        makespan = float(finish.max() - arrivals[0])
        return lat, makespan, outs, st

    def summary(lat, makespan):
        lat_ms = np.asarray(lat) * 1e3
        return {"p50_ms": float(np.percentile(lat_ms, 50)), "p99_ms": float(np.percentile(lat_ms, 99)),
                "mlups": total_lu / makespan / 1e6, "makespan_s": makespan}

    def burst(storage_mode):
        # saturated: every request is queued at t = 0; aggregate MLUPS = total updates / makespan
        srv = mmfd.Server(int(budget_gb * (1 << 30)), max_slots=slots, steps_per_tick=steps_per_tick,
                          use_graphs=True, stream=stream)
        t0 = time.perf_counter()
        tickets = []
        for r in reqs:
            d = dict(r.desc)
            if storage_mode == "fp32":
                d["storage"] = "fp32"
            tickets.append(srv.submit(mmfd.make_desc(**d), r.fields, r.steps))
        pending = set(tickets)
        while pending:
            for t in list(pending):
                rc, _ = srv.poll(t)
                if rc == mmfd.MMFD_OK:
                    srv.release(t)
                    pending.discard(t)
        mk = time.perf_counter() - t0
        srv.close()
        return total_lu / mk / 1e6

    lat32, mk32, out32, st32 = served("fp32")
    latmix, mkmix, outmix, stmix = served("mixed")
    # deviation per field relative to the request's initial field scale: a decaying flow ends far
    # below its initial magnitude (the low-Re vortices of small grids reach 1e-29 after 5000
    # steps), where a ratio to the final field's own maximum measures only the rounding floor
    def dev(outs):
        return max(max(float(np.abs(a - b).max() / max(1e-30, np.abs(f0).max())) for a, b, f0 in zip(o, p, r.fields))
                   for o, p, r in zip(outs, plain_out, reqs))
    err32 = dev(out32)
    errmix = dev(outmix)
    res = {"requests": count, "seed": seed, "arrival_rate_per_s": 0.8 * capacity, "total_lattice_updates": total_lu,
           "plain_fp32": summary(plain_lat, plain_makespan),
           "served_fp32": {**summary(lat32, mk32), "max_dev_vs_plain": err32,
                           "ticks": st32["ticks"], "launches": st32["launches"], "graph_replays": st32["graph_replays"]},
           "served_mixed_fp32_bf16": {**summary(latmix, mkmix), "max_dev_vs_plain_fp32": errmix},
           "budget_gb": budget_gb, "max_slots": slots, "steps_per_tick": steps_per_tick,
           "deviation": "max over requests and fields of max|served - plain| / max|initial field|"}
    res["served_fp32_vs_plain_mlups"] = res["served_fp32"]["mlups"] / res["plain_fp32"]["mlups"]
    # saturated throughput (capacity): plain = sum of service times; served = burst makespan
    res["capacity_mlups"] = {"plain_fp32": total_lu / sum(service) / 1e6, "served_fp32": burst("fp32"),
                             "served_mixed_fp32_bf16": burst("mixed")}
    res["capacity_served_fp32_vs_plain"] = res["capacity_mlups"]["served_fp32"] / res["capacity_mlups"]["plain_fp32"]
    return res


def accuracy_block():
    """Errors at each configuration's stated step count, next to the stated tolerances: FP32
    storage within 1e-5 relative max-norm of the FP64 run; BF16-offset storage at most 2x the FP64
    run's error against the exact solution where one exists (the Taylor-Green decay), else its
    deviation from FP64 as measured.  FP64 against the FP64 oracle (1e-12) is asserted by the test
    suite, not here.  The 3D NSE runs on 256^3 (its FP64 reference is bound by FP64 arithmetic)."""
    from paper_2505_17057_gb300 import accuracy as A
    tol32 = 1e-5
    blk = {"fp32_tol": tol32, "bf16_rule": "<= 2x the FP64 error against the exact solution"}
    c1 = A.cde2d_64()
    blk["cde2d_64"] = {"steps": 200, "fp64_gre_vs_exact_pde": {k: c1[k]["gre"] for k in ("D2Q5", "D2Q9")},
                       "note": "FP64 only; FP64 against the oracle to 1e-12 in the tests"}
    c2 = A.ncde2d(1024, 10000)
    blk["ncde2d_1024"] = {"steps": 10000, "reference": "FP64 GPU run",
                          "fp32_maxrel_vs_fp64": c2["fp32"]["max_rel_vs_fp64"],
                          "fp32_met": c2["fp32"]["max_rel_vs_fp64"] <= tol32,
                          "bf16_sr_maxrel_vs_fp64": c2["bf16_sr"]["max_rel_vs_fp64"],
                          "bf16_note": "no closed form: deviation from FP64 as measured"}
    c3 = A.tgv(4096, 100.0, 5000)
    g64 = c3["fp64"]["gre_u"]
    blk["tgv2d_4096"] = {"steps": 5000, "re": 100, "reference": "FP64 GPU run; analytic Taylor-Green decay",
                         "fp32_maxrel_vs_fp64": c3["fp32"]["max_rel_vs_fp64"],
                         "fp32_met": c3["fp32"]["max_rel_vs_fp64"] <= tol32,
                         "fp64_gre_u_vs_exact": g64, "fp32_gre_u_vs_exact": c3["fp32"]["gre_u"],
                         "bf16_gre_u_vs_exact": c3["bf16"]["gre_u"], "bf16_sr_gre_u_vs_exact": c3["bf16_sr"]["gre_u"],
                         "bf16_met": min(c3["bf16"]["gre_u"], c3["bf16_sr"]["gre_u"]) <= 2 * g64}
    for kind, n in (("cde3d", 512), ("nse3d", 256)):
        c4 = A.three_d(kind, n, 1000)
        blk[f"{kind}_{n}"] = {"steps": 1000, "reference": "FP64 GPU run",
                              "fp32_maxrel_vs_fp64": c4["fp32"]["max_rel_vs_fp64"],
                              "fp32_met": c4["fp32"]["max_rel_vs_fp64"] <= tol32,
                              "bf16_maxrel_vs_fp64": c4["bf16"]["max_rel_vs_fp64"],
                              "bf16_note": "no closed form used: deviation from FP64 as measured"}
    return blk


def run_reference(args):
    """The oracle arm: every step is one whole FP64 oracle step of the bench workload on the
    host's cores (the oracle as it stands; the level advances from step to step)."""
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    timer = OracleTimer(args.workload)
    n = timer.n
    for _ in range(args.warmup):
        timer.full_step()
    times = [timer.full_step() for _ in range(args.steps)]
    t_all = sum(times)
    value = args.steps * n * n / t_all / 1e6
    v1, sample1 = timer.one_thread(5.0)
    sample = f"{args.steps} whole MMFD steps of the {n}x{n} grid, direct form, {timer.cores} OpenMP threads"
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": t_all / args.steps * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": args.workload, "grid": [n, n], "lattice": "D2Q9",
                                              "pde": "NSE (He-Luo)", "levels": 2},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": timer.cores, "kind": "oracle", "sample": sample,
                             "one_thread": {"value": v1, "cores": 1, "sample": sample1}},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def run_split(args):
    """One solve of the workload split into slabs over the ranks (y slabs in 2D, z slabs in 3D;
    paper_2505_17057_gb300/slab.py).  Each rank's solver steps its rows plus one halo row on each
    side as a periodic grid; after every step the ranks swap their first / last owned rows over
    NCCL (point-to-point, into local receive buffers) and write them into the neighbours' halo
    rows with mmfd_set_rows.  With one rank the halo rows are the rank's own (periodic).  The
    value counts the owned nodes of all ranks (total work fixed: strong scaling)."""
    import numpy as np
    import torch
    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    from paper_2505_17057_gb300 import configs, mmfd
    from paper_2505_17057_gb300 import slab as SL
    kind, n = args.workload.split("_")
    n = int(n)
    maker = {"tgv2d": configs.tgv2d_4096, "nse3d": configs.nse3d_512, "cde3d": configs.cde3d_512,
             "lcde2d": configs.lcde2d_8192}[kind]
    desc_kw, fields, _ = maker(n=n, storage=args.storage)
    dim = 3 if kind.endswith("3d") else 2
    sl = SL.make_slab(rank, ws, fields[0].shape[0], 1)
    rows = sl.global_rows()
    local_fields = [np.ascontiguousarray(f[rows]) for f in fields]
    del fields
    n_local = list(desc_kw["n"][:-1]) + [sl.local_rows]
    stream = torch.cuda.Stream()
    # halo rows travel as FP64 values: exact for every storage (FP32 / BF16 offsets from the
    # reference state come back unchanged), so the slabs compute what one grid would
    dt, tdt = mmfd.MMFD_DT_F64, torch.float64
    with torch.cuda.stream(stream):
        s = mmfd.Solver(mmfd.make_desc(**{**desc_kw, "n": n_local}), stream=stream)
        s.set_fields(local_fields)
        if args.tune:
            s.autotune(None)
        info = s.get_info()
        nf = len(local_fields)
        row_shape = local_fields[0].shape[1:]
        bufs = {k: [torch.empty(row_shape, dtype=tdt, device="cuda") for _ in range(nf)]
                for k in ("send_lo", "send_hi", "recv_lo", "recv_hi")}
        ptr = {k: [t.data_ptr() for t in v] for k, v in bufs.items()}

        def step():
            s.step(1)
            mmfd.mmfd_get_rows(s.h, 0, 1, 1, ptr["send_lo"], mmfd.MMFD_DEVICE, dt)
            mmfd.mmfd_get_rows(s.h, 0, sl.rows, 1, ptr["send_hi"], mmfd.MMFD_DEVICE, dt)
            SL.exchange(sl, bufs["send_lo"], bufs["send_hi"], bufs["recv_lo"], bufs["recv_hi"])
            mmfd.mmfd_set_rows(s.h, 0, 0, 1, ptr["recv_lo"], mmfd.MMFD_DEVICE, dt)
            mmfd.mmfd_set_rows(s.h, 0, sl.rows + 1, 1, ptr["recv_hi"], mmfd.MMFD_DEVICE, dt)

        def barrier():
            if ws > 1:
                torch.distributed.barrier()

        for _ in range(args.warmup):
            step()
        torch.cuda.synchronize()
        barrier()
        torch.cuda.synchronize()
        sampler = ClockSampler(local)
        sampler.start()
        t0 = torch.cuda.Event(enable_timing=True)
        t1 = torch.cuda.Event(enable_timing=True)
        t0.record(stream)
        for _ in range(args.steps):
            step()
        t1.record(stream)
        torch.cuda.synchronize()
        barrier()
        torch.cuda.synchronize()
        total_ms = max_over_ranks(t0.elapsed_time(t1), "cuda")

        def more_steps(k):
            for _ in range(k):
                step()

        # every rank runs the same number of exchange steps (the count comes from the max over ranks)
        clock_window(more_steps, total_ms / args.steps)
        barrier()
        clocks = sampler.stop()
        clocks["window"] = f"the timed region and about {CLOCK_WINDOW_S:.0f} s of the same steps after it (untimed)"
        nodes_all = int(np.prod(desc_kw["n"]))
        value = nodes_all * args.steps / (total_ms / 1e3) / 1e6
        s.close()
    if rank == 0:
        halo_bytes = 2 * nf * int(np.prod(row_shape)) * 8
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
                "scaling": "strong", "vs_baseline": None,
                "dtype": {"fp32": "f32", "bf16": "bf16-offset storage, f32 arithmetic", "fp64": "f64"}[args.storage],
                "data": "synthetic",
                "config": {"workload": args.workload, "grid": desc_kw["n"], "lattice": desc_kw["lattice"],
                           "pde": desc_kw["pde"], "levels": desc_kw["levels"], "storage": args.storage,
                           "parallelism": f"slab{ws}", "slab_axis": "z" if dim == 3 else "y",
                           "rows_per_rank": sl.rows, "halo_rows": 1, "halo_bytes_sent_per_rank_per_step": halo_bytes,
                           "kernel": info.kernel.decode()},
                "clocks": clocks, "gpu_launches": args.steps * 5}
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def run_ours(args):
    import numpy as np
    import torch

    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    from paper_2505_17057_gb300 import configs, mmfd

    kind, n = args.workload.split("_")
    n = int(n)
    # srccde2d: a time-dependent source, set (from device memory) before every step
    has_src = kind == "srccde2d"
    if has_src:
        desc_kw, fields, fields_m1, source = configs.srccde2d_4096(n=n, storage=args.storage)
    else:
        maker = {"tgv2d": configs.tgv2d_4096, "cde3d": configs.cde3d_512, "nse3d": configs.nse3d_512,
                 "ncde2d": configs.ncde2d_1024, "lcde2d": configs.lcde2d_8192,
                 "theta2d": configs.theta2d_4096}[kind]
        desc_kw, fields, _ = maker(n=n, storage=args.storage)
    dim = 3 if kind.endswith("3d") else 2
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        d = mmfd.make_desc(**desc_kw, temporal_depth=args.depth)
        s = mmfd.Solver(d, stream=stream)
        s.set_fields(fields)
        srcs = []
        if has_src:
            s.set_fields(fields_m1, level=1)
            # eight consecutive source levels, cycled (the values repeat; the work per step does not)
            srcs = [torch.tensor(source(m)[0], dtype=torch.float32, device="cuda") for m in range(-1, 7)]
            s.set_source([srcs[0]], level=1)
            s.set_source([srcs[1]])
        tuned = None
        if args.tune:
            # outside the timed region: trial launches write only the spare buffer
            t = s.autotune(None)
            tuned = {"temporal_depth": t.temporal_depth, "rows_per_item": t.rows_per_item,
                     "candidates": t.candidates, "ms_per_step": t.ms_per_step}
        info = s.get_info()
        # steps per timed launch group: a theta-scheme solver's depth counts fused Jacobi sweeps,
        # one step each
        depth = 1 if info.sweeps > 0 else max(1, info.temporal_depth)
        nodes = n ** dim
        bytes_per_lu = info.bytes_per_lu

        def barrier():
            if ws > 1:
                torch.distributed.barrier()

        def set_src(i):
            if has_src:
                s.set_source([srcs[1 + i % 7]])

        # warm-up
        if has_src:
            for i in range(args.warmup):
                set_src(i)
                s.step(1)
        else:
            s.step(args.warmup * depth)
        torch.cuda.synchronize()
        barrier()
        torch.cuda.synchronize()
        sampler = ClockSampler(local)
        sampler.start()
        t_start = torch.cuda.Event(enable_timing=True)
        t_end = torch.cuda.Event(enable_timing=True)
        if has_src:
            # a source is set before every step: events around each step launch time the step
            # kernel apart from the source upload
            ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
            t_start.record(stream)
            for i in range(args.steps):
                set_src(i)
                ev[i][0].record(stream)
                s.step(depth)
                ev[i][1].record(stream)
            t_end.record(stream)
        else:
            # one mmfd_step call for the whole timed region: the library issues the launches back
            # to back, so no per-launch host round trip (event records, a ctypes call) paces a
            # short kernel; its average launch time is the region's time over the launches
            ev = None
            t_start.record(stream)
            s.step(args.steps * depth)
            t_end.record(stream)
        torch.cuda.synchronize()
        barrier()
        torch.cuda.synchronize()
        total_ms = t_start.elapsed_time(t_end)
        clock_window(lambda k: s.step(k * depth), total_ms / args.steps)
        clocks = sampler.stop()
        clocks["window"] = f"the timed region and about {CLOCK_WINDOW_S:.0f} s of the same launches after it (untimed)"
        launch_ms = [a.elapsed_time(b) for a, b in ev] if ev is not None else [t_start.elapsed_time(t_end) / args.steps]
        total_ms = max_over_ranks(total_ms, "cuda")
        steps_done = args.steps * depth
        ms_per_step = total_ms / steps_done
        value = job_mlups(ws, nodes, steps_done, total_ms / 1e3)

        # roofline of the dominant (only) kernel: compulsory bytes per launch / launch time
        peak, peak_kind = measured_peaks()
        avg_launch_s = statistics.mean(launch_ms) / 1e3
        # a launch reads and writes the stored level once, whatever its temporal depth
        alg_bytes = bytes_per_lu * nodes
        effective = bytes_per_lu * nodes * depth / avg_launch_s / 1e9
        kernel_name = info.kernel.decode()
        # theta-scheme: one step is the right-hand side plus info.sweeps Jacobi sweeps; its events,
        # bytes and traffic are those of the whole step.  Fused (jd > 1), the right-hand side's pass
        # also writes the first sweep's result and the others run jd per launch.  Compulsory bytes:
        # the right-hand side reads the level and writes rhs (fused: and the iterate), each sweep
        # launch reads the iterate and rhs and writes the next iterate; the effective figure counts
        # every sweep as unfused.
        theta = info.sweeps > 0
        jd = max(1, info.temporal_depth)
        left = info.sweeps - 1 if jd > 1 else info.sweeps
        sweep_launches = -(-left // jd)
        launches_per_step = (1 + sweep_launches) if theta else 1
        theta_launches = None
        if theta:
            # what one step launches: the right-hand side, then the sweeps (fused jd per launch, a
            # remainder on a shallower fused launch)
            full, rem = divmod(left, jd)
            if jd > 1:
                parts = ["k_theta (right-hand side and first sweep)", f"{full} x k_theta ({jd} sweeps each)"]
                if rem:
                    parts.append(f"1 x k_theta ({rem} sweeps)")
            else:
                parts = [kernel_name.replace("_src", "") + " (right-hand side)", f"{info.sweeps} x {kernel_name}"]
            theta_launches = " + ".join(parts)
            es = {"fp32": 4, "fp64": 8}[args.storage]
            alg_bytes = es * ((3 if jd > 1 else 2) + 3 * sweep_launches) * nodes
            effective = bytes_per_lu * nodes / avg_launch_s / 1e9
        achieved = alg_bytes / avg_launch_s / 1e9
        traffic = traffic_from_profile("k_march2d_theta" if theta else kernel_name, args.workload,
                                       jd if theta else depth, info.sweeps, args.storage)

        # end to end through the public API: every step uploads the level from pinned host memory,
        # advances it and copies the stepped level back to pinned host memory (the step's result);
        # a second variant reads back only the FP64 field sums (a diagnostic of the step)
        e2e_steps = max(3, min(args.steps, 20))
        pinned = [torch.from_numpy(np.ascontiguousarray(f, dtype=np.float32)).pin_memory() for f in fields]
        host_ptrs = [p.data_ptr() for p in pinned]
        back = [torch.empty(p.shape, dtype=torch.float32).pin_memory() for p in pinned]
        back_ptrs = [b.data_ptr() for b in back]
        h2d = sum(p.numel() * 4 for p in pinned)
        src_ptrs = []
        if has_src:
            # the step's source comes from the host too
            src_pinned = [torch.from_numpy(np.ascontiguousarray(source(0)[0], dtype=np.float32)).pin_memory()]
            src_ptrs = [p.data_ptr() for p in src_pinned]
            h2d += sum(p.numel() * 4 for p in src_pinned)

        def e2e_step(read_level):
            mmfd.mmfd_set_fields(s.h, 0, host_ptrs, mmfd.MMFD_HOST, mmfd.MMFD_DT_F32)
            if has_src:
                mmfd.mmfd_set_source(s.h, 0, src_ptrs, mmfd.MMFD_HOST, mmfd.MMFD_DT_F32)
            s.step(1)
            if read_level:
                mmfd.mmfd_fields(s.h, 0, back_ptrs, mmfd.MMFD_HOST, mmfd.MMFD_DT_F32)
            else:
                s.reduce(mmfd.MMFD_RED_SUM)

        def e2e_run(read_level):
            for _ in range(2):
                e2e_step(read_level)
            torch.cuda.synchronize()
            barrier()
            t0 = time.perf_counter()
            for _ in range(e2e_steps):
                e2e_step(read_level)
            torch.cuda.synchronize()
            return job_mlups(ws, nodes, e2e_steps, max_over_ranks(time.perf_counter() - t0, "cuda"))

        e2e_value = e2e_run(True)
        d2h = sum(b.numel() * 4 for b in back)
        e2e_sums_value = e2e_run(False)
        e2e_pipe = None
        if not has_src and ws == 1:
            try:
                e2e_pipe = e2e_two_streams(mmfd, desc_kw, s, fields, host_ptrs, back_ptrs, e2e_steps, nodes)
            except Exception as e:   # the serial figure above stands; this variant is reported void
                e2e_pipe = {"value": None, "error": f"{type(e).__name__}: {e}"[:200]}
        s.close()

        # the plain one-step-per-launch kernel on the same workload, when the headline launch
        # advances several steps: its own MLUPS and fraction of the HBM roofline (one launch reads
        # and writes the level once per step)
        plain_step = None
        if depth > 1 and not theta and not has_src:
            d1 = mmfd.make_desc(**desc_kw, temporal_depth=1)
            s1 = mmfd.Solver(d1, stream=stream)
            s1.set_fields(fields)
            if args.tune:
                s1.autotune(None)
            info1 = s1.get_info()
            s1.step(args.warmup)
            torch.cuda.synchronize()
            n1 = max(10, min(args.steps, 100))
            ev1 = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(n1)]
            for i in range(n1):
                ev1[i][0].record(stream)
                s1.step(1)
                ev1[i][1].record(stream)
            torch.cuda.synchronize()
            ms1 = statistics.mean(a.elapsed_time(b) for a, b in ev1)
            s1.close()
            ach1 = info1.bytes_per_lu * nodes / (ms1 / 1e3) / 1e9
            plain_step = {"value": nodes / (ms1 / 1e3) / 1e6, "unit": UNIT, "kernel": info1.kernel.decode(),
                          "avg_launch_ms": ms1, "steps": n1,
                          "roofline": {"bound": "hbm", "achieved": ach1, "peak": peak, "unit": "GB/s",
                                       "frac": ach1 / peak, "peak_kind": peak_kind,
                                       "alg_bytes_per_launch": info1.bytes_per_lu * nodes}}

    if rank != 0:
        if ws > 1:
            torch.distributed.destroy_process_group()
        return 0
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": {"fp32": "f32", "bf16": "bf16-offset storage, f32 arithmetic",
                                       "fp64": "f64"}[args.storage],
        "data": "synthetic",
        "config": {"workload": args.workload, "grid": [n] * dim, "lattice": desc_kw["lattice"],
                   "pde": {"NSE": "NSE (He-Luo)"}.get(desc_kw["pde"], desc_kw["pde"]),
                   "levels": desc_kw["levels"], "storage": args.storage,
                   "temporal_depth": jd if theta else depth,
                   **({"source": "su, set from device memory before every step"} if has_src else {}),
                   **({"theta": desc_kw["theta"], "dt": desc_kw["dt"], "jacobi_sweeps": info.sweeps,
                       "sweeps_per_launch": jd} if theta else {}),
                   "autotuned": tuned,
                   "parallelism": f"replicas{ws}" if ws > 1 else "single",
                   "l2": l2_note(info.device_bytes, info.levels_stored)[0]},
        "roofline": {"bound": l2_note(info.device_bytes, info.levels_stored)[1], "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": achieved / peak, "traffic": traffic,
                     "frac_of_nominal": achieved / NOMINAL_HBM_GBS,
                     "kernel": theta_launches if theta else kernel_name,
                     "peak_kind": peak_kind,
                     "alg_bytes_per_launch": alg_bytes, "avg_launch_ms": avg_launch_s * 1e3,
                     "effective_gbs": effective,
                     **({"launches_per_step": launches_per_step,
                         "note": "per theta step: alg bytes, time and traffic of its 1 + sweeps launches"}
                        if theta else {})},
        "clocks": clocks,
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                "steps": e2e_steps, "read_back": "the stepped level, FP32, into page-locked host memory",
                **({"two_streams": e2e_pipe} if e2e_pipe else {}),
                "sums_only": {"value": e2e_sums_value, "unit": UNIT, "h2d_bytes_per_step": h2d,
                              "d2h_bytes_per_step": 8 * len(pinned),
                              "read_back": "the FP64 field sums of the stepped level"}},
        "gpu_launches": args.steps * (2 if has_src else launches_per_step),
    }
    if plain_step is not None:
        line["plain_step"] = plain_step
    if ws == 1 and args.accuracy:
        with torch.cuda.stream(stream):
            line["accuracy"] = accuracy_block()
    if args.serve > 0:
        with torch.cuda.stream(stream):
            line["serving"] = serving_bench(args.serve, 5, mmfd, stream)
    if ws == 1 and not args.no_cpu_baseline and args.workload.startswith("tgv2d"):
        timer = OracleTimer(args.workload)
        v, sample = timer.measure(3)
        v1, sample1 = timer.one_thread(5.0)
        line["cpu_baseline"] = {"value": v, "unit": UNIT, "cores": timer.cores, "kind": "oracle", "sample": sample,
                                "one_thread": {"value": v1, "cores": 1, "sample": sample1}}
    print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="tgv2d_4096")
    ap.add_argument("--storage", default="fp32", choices=["fp32", "bf16", "fp64"])
    ap.add_argument("--depth", type=int, default=0,
                    help="temporal blocking depth: 0 = the autotuner picks among the depths the solver "
                         "allows (every step is still computed; blocked launches fuse several), "
                         "1 = one step per launch, T = T steps per launch")
    ap.add_argument("--no-tune", dest="tune", action="store_false",
                    help="skip the autotuner (work-item height from the launcher's heuristic)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-accuracy", dest="accuracy", action="store_false",
                    help="skip the accuracy block (errors at the stated step counts against FP64 / closed forms)")
    ap.add_argument("--serve", type=int, default=200, help="requests in the serving run (0 = skip)")
    ap.add_argument("--split", default="none", choices=["none", "slab"],
                    help="slab: one solve split over the ranks with halo exchange (default: one solve per rank)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    if args.split == "slab":
        return run_split(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
