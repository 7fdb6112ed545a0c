"""Benchmark of the SWR-Galerkin sweep on GB300.

One step = the whole hot path on the 2-electron ground-state workload
([-12,12]^2, 4x4 subdomains, 24x24 Gaussians each): swr_assemble (quadrature,
local Galerkin systems, orthonormalisation, step-matrix inverses, projection
of phi0) followed by swr_iterate until the interface residual Res(k) <= 1e-8.
Metric: local subdomain solves per second (one solve = one time step of one
subdomain), with the time-to-residual reported beside it.  The same line
carries bounded measurements of the two larger workloads (`extra_workloads`):
the 512-instance uneven batch (Schwarz iterations of every instance) and the
64-subdomain real-time problem (one Schwarz iteration of 1000 Crank-Nicolson
steps).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gb300|reference]

Under torchrun every rank solves its own replica of the workload on its own
GPU (independent problems, no data-path collective; weak scaling); the time
is the max over ranks.  `--impl reference` times the FP64 CPU oracle on the
host cores instead (rank 0 only).
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

TOL = 1e-8
KMAX = 200
METRIC = "SWR time-to-1e-8 interface residual; subdomain solves/s vs plain FP64 GPU path"
# FP64 and FP32 (non-tensor) FMA rates of one GB300, measured on this machine with
# independent FMA chains over all SMs (the ceilings of the window kernel)
FP32_PEAK_TFLOPS = 67.7
# 56-bit fixed-point products on the integer pipes: 4.5 multiply-adds per clock
# and SM (FP64 quality), 152 SMs at 1.92 GHz
FIXED_PEAK_TFLOPS = 2.6
# DRAM traffic of the window kernels from one ncu capture each (profiles/): bytes per
# launch, or for the batched case bytes per algorithmic byte, valid only while the
# source of the kernel and of the device functions it calls is the one that was
# profiled (sha256 prefix over those functions' text in swr_window.cu)
KERNEL_FUNCS = {
    "k_window_fused": ["release_barrier", "block_sums2", "two_sum", "make_task_cache", "z_rows_sm", "df32_acc",
                       "k_window_fused"],
    "k_window_2ph<true>": ["reduce_barrier", "two_sum", "make_task_cache", "mirror_sid", "swap_index",
                           "mirror_weight", "diagonal_anti", "z_rows_sm", "z_rows_staged", "prefetch_l2",
                           "prefetch_rows", "df32_acc", "df32_rows4", "k_window_2ph"],
}
KERNEL_FUNCS["k_window_split"] = ["mbar_wait", "split_stage_rows", "reduce_barrier_sd", "split_cbar", "split_cbar_or",
                                  "mbar_arrive", "z_rows_group", "split_chunk", "ds_add", "split_row", "two_sum",
                                  "make_task_cache", "mirror_sid", "swap_index", "mirror_weight", "diagonal_anti",
                                  "df32_acc", "k_window_split"]
KERNEL_FUNCS["k_window_2ph<true>@batched"] = KERNEL_FUNCS["k_window_2ph<true>"]
KERNEL_FUNCS["k_window_split@batched"] = KERNEL_FUNCS["k_window_split"]
KERNEL_FUNCS["k_window_cluster"] = ["cl_rsqrt", "k_window_cluster"]
# FP64 plans: on chip (one cluster per instance), one pass over the grid, or two phases.
FP64_WINDOW = "k_window_onchip / k_window_fx / k_window_2ph<false>"
PROFILED_TRAFFIC = {
    "k_window_fused": ("123b4a784de2ee96", 329.5e6, "profiles/k_window_fused_tise_2e_16sd.md"),
    "k_window_2ph<true>@batched": ("cbd72ea8633a4ed0", 1.192, "profiles/k_window_2ph_df32_batched_uneven.md"),
    "k_window_split@batched": ("e908166e69fb5910", 1.030, "profiles/k_window_split_batched_uneven.md"),
    # the captured launch is a 1723-step window; the traffic is the history rows and
    # Robin sources, proportional to the window length like the algorithmic bytes
    "k_window_cluster": ("01d810867459c710", 259.04e6, "profiles/k_window_cluster_tise_2e_16sd.md"),
}


def kernel_source_hash(kernel):
    """sha256 prefix of the text of the functions `kernel` is built from."""
    import hashlib
    import re
    csrc = os.path.join(ROOT, "paper_1710_02401_gb300", "csrc")
    src = open(os.path.join(csrc, "swr_window.cu")).read() + open(os.path.join(csrc, "swr_cluster.cu")).read()
    h = hashlib.sha256()
    for fn in KERNEL_FUNCS[kernel]:
        m = re.search(r"^[^\n]*\b" + re.escape(fn) + r"\(.*?^}\n", src, re.M | re.S)
        if m is None:
            return None
        h.update(m.group(0).encode())
    return h.hexdigest()[:16]


def profiled_traffic(kernel):
    rec = PROFILED_TRAFFIC.get(kernel)
    if rec is None or kernel not in KERNEL_FUNCS or rec[0] != kernel_source_hash(kernel):
        return None, None
    return rec[1], rec[2]


BATCHED = "batched_uneven_512"


def workload(name: str):
    from paper_1710_02401_gb300 import problems as P
    if name == BATCHED:
        return P.batched_uneven(512)
    if name == "tise_2e_16sd":
        return P.tise_2e_16_subdomains()
    if name == "tise_1d_2sd":
        return P.tise_1d_two_subdomains()
    if name == "tdse_2e_64sd":
        return P.tdse_2e_64_subdomains()
    raise SystemExit(f"unknown workload {name}")


def batched_config(insts) -> dict:
    n1 = sum(1 for i in insts if i.n_elec == 1)
    kk = [kd ** i.n_elec for i in insts for kd in i.K_d]
    return {"workload": BATCHED, "instances": len(insts), "one_electron": n1, "two_electron": len(insts) - n1,
            "subdomains": sum(i.n_sub for i in insts), "K_min": min(kk), "K_max": max(kk),
            "K_mean": sum(kk) / len(kk), "seed": 171002401, "dt": 0.1, "mu": "10.0", "ngf_tol": 1e-12,
            "max_steps": max(i.max_steps for i in insts), "l2": "flushed (256 MB write) before every step; step matrices (>=100 GB per chunk) "
            "exceed L2", "parallelism": "instances sharded over ranks (no data-path collective)",
            "step": "one Schwarz iteration of every instance (chunks sized to the free HBM, each one "
                    "persistent window launch per iteration, replayed from a captured CUDA graph)"}


def workload_config(name: str, inst) -> dict:
    return {"workload": name, "n_elec": inst.n_elec, "box": list(inst.box), "L": inst.L,
            "subdomains": inst.n_sub, "K_d": inst.K_d, "K": inst.K_d ** inst.n_elec,
            "nodes_per_coord": (inst.n_mid + 2) * inst.q_p, "dt": inst.dt, "mu": str(inst.mu),
            "tol": TOL, "kmax": KMAX, "l2": "flushed (256 MB write) before every step",
            "parallelism": "replicas (one independent problem per GPU)",
            **({"symmetry": "antisymmetric", "phi0_center": list(inst.phi0_center)}
               if getattr(inst, "symmetry", "none") == "antisymmetric" else {})}


class ClockSampler:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.path = os.path.join(tempfile.gettempdir(), f"swr_clocks_{os.getpid()}.csv")

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index),
                 "--query-gpu=clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
                 "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
                 "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap",
                 "--format=csv,noheader,nounits", "-lms", "200"], stdout=self.f, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.f.close()
        rows = []
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 8:
                continue
            try:
                rows.append((float(parts[0]), float(parts[1]), parts[4:8]))
            except ValueError:
                continue
        if not rows:
            return None
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for _, _, r in rows for i, v in enumerate(r) if v.lower() == "active"})
        return {"sm_mhz": statistics.median(r[0] for r in rows), "sm_max_mhz": max(r[1] for r in rows),
                "reasons": reasons, "samples": len(rows)}


def oracle_sample(inst, gpu_solves_per_iter=None):
    """Times the FP64 CPU oracle on this host: assembly of all local systems,
    then the first Schwarz iteration (zero initial traces).  Returns
    (solves/s of the iteration, description, assembly seconds)."""
    from oracle import swr_oracle as O
    t0 = time.perf_counter()
    locs = O.assemble(inst)
    t_asm = time.perf_counter() - t0
    t1 = time.perf_counter()
    r = O.run_swr(inst, kmax=1, tol=0.0, locs=locs)
    t_it = time.perf_counter() - t1
    solves = r.records[0].n_win * inst.n_sub
    desc = (f"oracle (numpy FP64, dense quadrature + LU) on the same workload: first Schwarz "
            f"iteration, {solves} local step solves in {t_it:.2f} s; local assembly of all "
            f"{inst.n_sub} subdomains took {t_asm:.2f} s and is not in the rate")
    return solves / t_it, desc, t_asm


def batched_oracle_sample(insts):
    """Bounded oracle sample of the batched workload: the first Schwarz
    iteration of its smallest 1-electron and smallest 2-electron instances
    (fewest subdomains), local assembly excluded from the rate."""
    from oracle import swr_oracle as O
    pick = [min((i for i in insts if i.n_elec == n), key=lambda i: (i.n_sub, sum(i.K_d))) for n in (1, 2)]
    solves, t_it = 0, 0.0
    for inst in pick:
        locs = O.assemble(inst)
        t0 = time.perf_counter()
        r = O.run_swr(inst, kmax=1, tol=0.0, locs=locs)
        t_it += time.perf_counter() - t0
        solves += r.records[0].n_win * inst.n_sub
    desc = (f"oracle (numpy FP64) on the batch's smallest 1-electron and 2-electron instances "
            f"({pick[0].n_sub} and {pick[1].n_sub} subdomains): first Schwarz iteration, {solves} local "
            f"step solves in {t_it:.2f} s, local assembly excluded")
    return solves, t_it, desc


def run_reference(args, inst, name):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    if name == BATCHED:
        for _ in range(args.warmup):
            batched_oracle_sample(inst)
        solves, t_tot = 0, 0.0
        for _ in range(args.steps):
            n, t, desc = batched_oracle_sample(inst)
            solves += n
            t_tot += t
        value = solves / t_tot
        print(json.dumps({
            "impl": "reference", "metric": METRIC, "value": value, "unit": "subdomain solves/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * t_tot / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": batched_config(inst),
            "cpu_baseline": {"value": value, "unit": "subdomain solves/s", "cores": os.cpu_count(),
                             "kind": "oracle", "sample": "each step: " + desc},
            "e2e": {"value": value, "unit": "subdomain solves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        }))
        return
    from oracle import swr_oracle as O
    locs = O.assemble(inst)
    for _ in range(args.warmup):
        O.run_swr(inst, kmax=1, tol=0.0, locs=locs)
    t_tot, solves = 0.0, 0
    for _ in range(args.steps):
        t0 = time.perf_counter()
        r = O.run_swr(inst, kmax=1, tol=0.0, locs=locs)
        t_tot += time.perf_counter() - t0
        solves += r.records[0].n_win * inst.n_sub
    value = solves / t_tot
    cores = os.cpu_count()
    sample = ("each step: first Schwarz iteration (zero initial traces) of the FP64 oracle on the "
              "full workload, local systems assembled once before the timed steps")
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": "subdomain solves/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * t_tot / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": workload_config(name, inst),
        "cpu_baseline": {"value": value, "unit": "subdomain solves/s", "cores": cores, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": value, "unit": "subdomain solves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


PRECISIONS = ("mixed", "fp64", "fp32")
DTYPES = {"mixed": "f32x2 (double-single) step matrices, f64 reductions", "fp64": "f64",
          "fp32": "f32 step matrices (double-single products) then f32x2 refinement, f64 reductions"}


def prec_code(S, name):
    return {"mixed": S.PREC_MIXED, "fp64": S.PREC_FP64, "fp32": S.PREC_FP32_REFINED}[name]


def hbm_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        return json.load(open(path))["hbm_gbs"], "MEASURED_PEAKS.json hbm_gbs (measured copy bandwidth)"
    return 6800.0, "fallback 6.8 TB/s (no MEASURED_PEAKS.json)"


def batched_measure(args, insts, env, prec_name, steps, warmup, sample_clocks):
    """The uneven batch: instances sharded over ranks, cut into chunks that fit
    the free HBM; per chunk setup + assembly + window autotune (untimed), W
    warm-up and K timed Schwarz iterations (CUDA events around each swr_step,
    L2 flushed before each)."""
    S, torch, dist, dev, stream, flush, world, rank, local = env
    from paper_1710_02401_gb300 import dist as D
    mine = [insts[i] for i in D.shard(insts, rank, world)]

    def chunks_for(prec):
        free, _ = torch.cuda.mem_get_info(dev)
        budget = 0.85 * free
        out, cur, cur_b = [], [], 0
        for inst in mine:
            b = S.workspace_bytes(inst, prec) + (1 << 20)
            if cur and cur_b + b > budget:
                out.append(cur)
                cur, cur_b = [], 0
            cur.append(inst)
            cur_b += b
        if cur:
            out.append(cur)
        return out

    def run(prec_name, steps, warmup, sample_clocks):
        prec = prec_code(S, prec_name)
        t_ms, solves, wbytes, wms, wlaunch, launches = 0.0, 0, 0.0, 0.0, 0, 0
        e2e_wall, e2e_solves, h2d, d2h, tunes, energies, first_e = 0.0, 0, 0, 0, [], [], []
        chunks = chunks_for(prec)
        torch.cuda.synchronize(dev)
        if world > 1:
            dist.barrier()
        sampler = ClockSampler(local) if sample_clocks else None
        if sampler:
            sampler.start()
        for chunk in chunks:
            torch.cuda.synchronize(dev)
            w0 = time.perf_counter()
            s = S.SWR(chunk, precision=prec, device=str(dev), stream=stream, rows_per_task=args.rows_per_task,
                      window_variant=args.window_variant if prec != S.PREC_FP64 else 0)
            s.assemble()
            tunes.append(s.window_plan() if args.no_autotune else s.autotune(steps=24))
            for w in range(warmup):
                e2e_solves += s.step().subdomain_solves
                if w == 0:
                    first_e += [float(x) for x in s.energy()]
            c0 = s.counters()
            for _ in range(steps):
                flush.zero_()
                e0 = torch.cuda.Event(enable_timing=True)
                e1 = torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                r = s.step()
                e1.record(stream)
                e1.synchronize()
                t_ms += e0.elapsed_time(e1)
                solves += r.subdomain_solves
                e2e_solves += r.subdomain_solves
            c1 = s.counters()
            energies += [float(x) for x in s.energy()]
            s.close()
            del s
            torch.cuda.synchronize(dev)
            e2e_wall += time.perf_counter() - w0
            wbytes += c1["window_bytes_alg"] - c0["window_bytes_alg"]
            wms += c1["window_ms"] - c0["window_ms"]
            wlaunch += int(c1["window_launches"] - c0["window_launches"])
            launches += int(c1["kernel_launches"] - c0["kernel_launches"])
            h2d += int(c1["h2d_bytes"])
            d2h += int(c1["d2h_bytes"])
        clocks = sampler.stop() if sampler else None
        t_max, solves_all = D.combine(t_ms * 1e-3, solves)
        e_max, e_solves_all = D.combine(e2e_wall, e2e_solves)
        return dict(value=solves_all / t_max, t_max=t_max, wbytes=wbytes, wms=wms, wlaunch=wlaunch,
                    launches=launches, e2e=e_solves_all / e_max, h2d=h2d, d2h=d2h, tunes=tunes,
                    chunks=len(chunks), clocks=clocks, energies=energies, first_e=first_e)

    return run(prec_name, steps, warmup, sample_clocks)


def batched_roofline(S, prec_name, r):
    """HBM roofline of the batched window: algorithmic step-matrix bytes over
    the window kernel's CUDA-event time."""
    peak, peak_src = hbm_peak()
    gbs = r["wbytes"] / (r["wms"] * 1e-3) / 1e9 if r["wms"] > 0 else 0.0
    kname = "k_window_2ph<true>" if prec_name != "fp64" else "k_window_2ph<false>"
    n_split = sum(t["variant"] == S.WINDOW_SPLIT for t in r["tunes"])
    if prec_name != "fp64" and 2 * n_split > len(r["tunes"]):
        kname = "k_window_split"
    bpe = {"mixed": "8 bytes (FP32 hi/lo planes)", "fp64": "8 bytes (FP64)",
           "fp32": "4 bytes (FP32-rounded hi plane) before the switch, 8 after"}[prec_name]
    roof = {"kernel": kname, "bound": "hbm", "achieved": gbs, "peak": peak, "unit": "GB/s",
            "frac": gbs / peak, "peak_source": peak_src,
            "algorithmic": f"{bpe} of the step-matrix inverse per element per local step solve, K^2 elements per "
                           "solve; each chunk's matrices (>= 100 GB) stream from HBM every step",
            "window_ms_per_launch": r["wms"] / max(1, r["wlaunch"])}
    ratio, src = profiled_traffic(kname + "@batched")
    roof["traffic"] = ratio * r["wbytes"] / max(1, r["wlaunch"]) if ratio else None
    roof["traffic_source"] = src
    return roof


def run_batched(args, insts, env):
    S, torch, dist, dev, stream, flush, world, rank, local = env
    main_run = batched_measure(args, insts, env, args.precision, args.steps, args.warmup, True)
    other = None
    if not args.no_compare:
        other_name = "fp64" if args.precision != "fp64" else "mixed"
        other = batched_measure(args, insts, env, other_name, args.steps, args.warmup, False)
        other["name"] = other_name
    if rank != 0:
        return
    roof = batched_roofline(S, args.precision, main_run)
    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        n, t, desc = batched_oracle_sample(insts)
        cpu = {"value": n / t, "unit": "subdomain solves/s", "cores": os.cpu_count(), "kind": "oracle",
               "sample": desc}
    it = args.warmup + args.steps
    out = {
        "metric": METRIC, "value": main_run["value"], "unit": "subdomain solves/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * main_run["t_max"] / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": DTYPES[args.precision],
        "data": "synthetic", "config": dict(batched_config(insts), chunks=main_run["chunks"]),
        "precision": args.precision, "roofline": roof, "cpu_baseline": cpu,
        "e2e": {"value": main_run["e2e"], "unit": "subdomain solves/s",
                "h2d_bytes_per_step": main_run["h2d"] // it, "d2h_bytes_per_step": main_run["d2h"] // it,
                "note": "whole public-API path per chunk: setup from host descriptors, assembly, autotune, "
                        "all warm-up and timed iterations, energy read-back, teardown"},
        "gpu_launches": main_run["launches"],
        "clocks": main_run["clocks"],
        "autotune": [{k: t[k] for k in ("variant", "rows_per_task", "tasks", "ctas", "task_state_global")}
                     for t in main_run["tunes"]],
        "energy_first": main_run["energies"][:4],
    }
    if other is not None:
        out["other_precision"] = {"precision": other["name"], "value": other["value"],
                                  "ms_per_step": 1e3 * other["t_max"] / args.steps,
                                  "speedup_of_headline": main_run["value"] / other["value"],
                                  # same inputs: the first Schwarz iteration of every instance
                                  "max_rel_energy_difference_first_iteration": max(
                                      abs(a - b) / max(abs(b), 1e-300)
                                      for a, b in zip(main_run["first_e"], other["first_e"])),
                                  "note": "later iterations of the 1-electron instances with 30-64 subdomains "
                                          "separate between precisions: their Schwarz trajectories amplify "
                                          "1e-14 perturbations to O(0.1) within three iterations (also in the "
                                          "oracle)"}
    print(json.dumps(out))


def extra_batched(args, env):
    """Bounded measurement of the 512-instance uneven batch: per chunk one
    warm-up and `extra_iterations` timed Schwarz iterations of every instance."""
    S = env[0]
    insts = workload(BATCHED)
    k = max(1, args.extra_iterations)
    r = batched_measure(args, insts, env, args.precision, k, 1, False)
    return {"precision": args.precision, "value": r["value"], "unit": "subdomain solves/s",
            "ms_per_schwarz_iteration": 1e3 * r["t_max"] / k, "iterations_timed": k, "warmup": 1,
            "subdomains": sum(i.n_sub for i in insts), "chunks": r["chunks"],
            "roofline": batched_roofline(S, args.precision, r), "gpu_launches": r["launches"],
            "note": "Schwarz iterations 2..1+k of every instance (each chunk of instances that fits the free HBM "
                    "is set up, assembled and autotuned untimed); step matrices stream from HBM"}


# Real time: the persistent fixed-point window, or the host-launched sweeps of the
# FP32-rounded matrices.
RT_KERNEL = {"fp32": "k_cmv_df32 + Crank-Nicolson element-wise kernels"}


def extra_real_time(args, env):
    """Bounded measurement of the 64-subdomain real-time workload (K = 1024
    complex, 1000 Crank-Nicolson steps): one warm-up and one timed Schwarz
    iteration in the headline precision and in FP64."""
    S, torch, dist, dev, stream, flush, world, rank, local = env
    inst = workload("tdse_2e_64sd")
    out = {}
    for pn in (args.precision, "fp64"):
        s = S.SWR(inst, precision=prec_code(S, pn), device=str(dev), stream=stream)
        s.assemble()
        s.step()
        c0 = s.counters()
        flush.zero_()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        rep = s.step()
        e1.record(stream)
        e1.synchronize()
        c1 = s.counters()
        ms = e0.elapsed_time(e1)
        w_ms = c1["window_ms"] - c0["window_ms"]
        gbs = (c1["window_bytes_alg"] - c0["window_bytes_alg"]) / (w_ms * 1e-3) / 1e9
        hbm, src = hbm_peak()
        out[pn] = {"value": rep.subdomain_solves / (ms * 1e-3), "unit": "subdomain solves/s",
                   "ms_per_schwarz_iteration": ms, "window_ms": w_ms, "fp32_matrices": rep.fp32_matrices,
                   "norm2": float(s.norm2()[0]), "dipole": float(s.dipole()[0]),
                   "tensor_contractions": s.window_plan()["tensor_contractions"],
                   "roofline": {"kernel": RT_KERNEL.get(pn, "k_rt_window"), "bound": "hbm",
                                "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                                "peak_source": src,
                                "algorithmic": "8 bytes per complex element of the symmetric step matrix (its lower "
                                               "triangle in fixed point, or FP32-rounded) per sweep, 16 "
                                               "double-single, (1 + m) sweeps per step"}}
        s.close()
    out[args.precision]["speedup_vs_fp64"] = out[args.precision]["value"] / out["fp64"]["value"]
    out["note"] = "second Schwarz iteration (the first is the warm-up), 1000 Crank-Nicolson steps, L2 flushed"
    return out


def run_real_time_converge(args, S, kmax=80):
    """The real-time 64-subdomain workload from assembly to Res <= 1e-8:
    CUDA-synchronised wall time of assemble + iterate, the iteration count
    and the residual of every iteration."""
    import torch
    inst = workload("tdse_2e_64sd")
    s = S.SWR(inst, precision=prec_code(S, args.precision))
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    s.assemble()
    rep, hist = s.iterate(TOL, kmax)
    torch.cuda.synchronize()
    wall = time.perf_counter() - t0
    out = {"metric": "real-time workload to Res <= 1e-8 (wall time, assembly included)", "value": wall, "unit": "s",
           "higher_is_better": False, "data": "synthetic", "precision": args.precision,
           "config": workload_config("tdse_2e_64sd", inst), "converged": bool(rep.converged),
           "schwarz_iterations": rep.iterations, "res_history": [float(x) for x in hist],
           "subdomain_solves": rep.subdomain_solves, "solves_per_s": rep.subdomain_solves / wall,
           "norm2": float(s.norm2()[0]), "dipole": float(s.dipole()[0])}
    s.close()
    print(json.dumps(out))


def run_lsd(args, S, reps=3):
    """swr_lsd_build at the paper's Test 1 sizes: wall time of the whole call
    (allocation, device work, copies back), best of `reps` after a warm-up,
    and Table 1's inner products of the central subdomain's first four
    determinants with themselves and with the first two of the next subdomain
    in x1."""
    kw = dict(M=10, K=45, kd=40)
    S.lsd_build(**kw)
    best = float("inf")
    for _ in range(reps):
        t0 = time.perf_counter()
        g = S.lsd_build(**kw)
        best = min(best, time.perf_counter() - t0)
    c = 2 + 5 * 2
    out = {"metric": "swr_lsd_build wall time (Test 1 sizes)", "value": best, "unit": "s", "higher_is_better": False,
           "data": "synthetic", "config": {"L": 5, "box": [-8.0, 8.0], "overlap": 0.32, "orbitals_per_subdomain": 10,
                                            "determinants_per_subdomain": 45, "gaussians_per_orbital_basis": 40,
                                            "nuclei": [[-0.5, 1.0], [0.5, 1.0]]},
           "orbital_energies_central": [float(x) for x in g["lam"][2]],
           "table1_vv_offdiag_max": float(abs(g["S_lsd"][c][:4, :4] - __import__("numpy").eye(4)).max()),
           "table1_vw": [[float(x) for x in row] for row in g["G_next"][c][:4, :2]]}
    print(json.dumps(out))


def run_assembly(args, S, reps=3):
    """swr_assemble timed with CUDA events (library counter), best of `reps`
    after one warm-up, for both contraction paths."""
    import torch
    rows = []
    for wname in ("tdse_2e_64sd", "tise_2e_16sd"):
        inst = workload(wname)
        for pname, path in (("fp64", S.CONTRACT_FP64), ("tensor", S.CONTRACT_TENSOR)):
            s = S.SWR(inst, precision=S.PREC_MIXED, contraction_path=path)
            s.assemble()
            best = float("inf")
            for _ in range(reps):
                c0 = s.counters()["assemble_ms"]
                s.assemble()
                best = min(best, s.counters()["assemble_ms"] - c0)
            rows.append({"workload": wname, "contraction": pname, "assemble_ms": best,
                         "subdomains": inst.n_sub, "K": inst.K_d ** inst.n_elec})
            s.close()
            torch.cuda.synchronize()
    out = {"metric": "swr_assemble time (FP64 vs tensor-core contractions)", "unit": "ms",
           "higher_is_better": False, "data": "synthetic", "rows": rows}
    for w in ("tdse_2e_64sd", "tise_2e_16sd"):
        a = [r["assemble_ms"] for r in rows if r["workload"] == w]
        out[f"speedup_{w}"] = a[0] / a[1]
    print(json.dumps(out))


LEARNED_FAMILIES = {
    "small": ("learned_trace_family", "learned_trace_family (2 electrons, [-6,6]^2, 2x2 subdomains, 8x8 Gaussians, "
                                      "40 Crank-Nicolson steps, random nuclei, softening and field phase)"),
    "16sd": ("learned_trace_family_16sd", "learned_trace_family_16sd (2 electrons, [-10,10]^2, 4x4 subdomains with "
                                          "the 64-subdomain real-time workload's core width 5 and overlap 0.5, 10x10 "
                                          "Gaussians, 100 Crank-Nicolson steps, random nuclei, charges, softening "
                                          "and field phase)"),
}


def run_learned(args):
    """Learned initial traces: GPU data generation, training with the
    library's MLP kernels, and the held-out comparison at equal residual."""
    import numpy as np
    import torch
    from paper_1710_02401_gb300 import learn as Lrn
    from paper_1710_02401_gb300 import problems as P
    fam_fn, fam_desc = LEARNED_FAMILIES[args.learned_family]
    family = getattr(P, fam_fn)
    n_train, n_test = args.learned_train, args.learned_test
    t0 = time.perf_counter()
    x, y, done = Lrn.gather_training_set(family(n_train, seed=21))
    torch.cuda.synchronize()
    t_data = time.perf_counter() - t0
    t0 = time.perf_counter()
    model, losses = Lrn.train(x, y, steps=args.learned_steps)
    torch.cuda.synchronize()
    t_train = time.perf_counter() - t0
    r = Lrn.compare_timed(model, family(n_test, seed=99))
    print(json.dumps({"metric": "Schwarz time-to-1e-8 from the learned initial traces vs zero traces",
                      "unit": "s", "higher_is_better": False, "value": r["seconds_learned"],
                      "baseline_zero_guess_s": r["seconds_zero_guess"],
                      "speedup": r["seconds_zero_guess"] / r["seconds_learned"], **r,
                      "training": {"instances": n_train, "subdomains": int(x.shape[0]), "data_seconds": t_data,
                                   "train_seconds": t_train, "adam_steps": args.learned_steps,
                                   "loss_first": losses[0], "loss_last": losses[-1],
                                   "training_iterations_zero_guess_mean": float(np.mean(done))},
                      "config": {"workload": fam_desc, "held_out_instances": n_test, "tol": 1e-8},
                      "data": "synthetic"}))


SWEEP_DT = (0.025, 0.05, 0.1, 0.2)
SWEEP_MU = (2.0, 5.0, 10.0, 20.0, 50.0)
SWEEP_KMAX = 300


def run_sweep(args, inst, name, S):
    """Convergence of the Schwarz iteration over time steps (mu = 10) and Robin
    constants (dt = 0.1), with the Robin transmission condition and the
    classical one (Dirichlet data imposed by penalty with the same mu): for each
    point the Schwarz iterations to Res <= 1e-8 (capped), the mean contraction
    Res(k+1)/Res(k) over the iterations after the first two, the converged
    energy and the solve time (assembly + iterations, mixed precision)."""
    if inst.mode != "tise":
        raise SystemExit("--sweep covers the imaginary-time workloads")
    import torch
    points = [("robin", dt, 10.0) for dt in SWEEP_DT] + [("robin", 0.1, mu) for mu in SWEEP_MU]
    points += [("dirichlet", dt, 10.0) for dt in SWEEP_DT] + [("dirichlet", 0.1, mu) for mu in SWEEP_MU]
    rows, seen = [], set()
    for tc, dt, mu in points:
        if (tc, dt, mu) in seen:
            continue
        seen.add((tc, dt, mu))
        s = S.SWR(inst.replace(tc=tc, dt=dt, mu=mu), precision=S.PREC_MIXED)
        t0 = time.perf_counter()
        s.assemble()
        rep, hist = s.iterate(TOL, SWEEP_KMAX)
        torch.cuda.synchronize()
        sec = time.perf_counter() - t0
        h = [x for x in hist if x > 0]
        rate = None
        if len(h) > 4:
            tail = h[2:]
            rate = math.exp(sum(math.log(b / a) for a, b in zip(tail[:-1], tail[1:])) / (len(tail) - 1))
        rows.append({"tc": tc, "dt": dt, "mu": mu, "iterations": rep.iterations, "converged": bool(rep.converged),
                     "res_last": rep.res_last, "rate": rate, "energy": float(s.energy()[0]), "seconds": sec})
        s.close()
    print(json.dumps({"metric": "Schwarz iterations to Res <= 1e-8 over time step and Robin constant",
                      "unit": "iterations", "workload": name, "precision": "mixed", "kmax": SWEEP_KMAX,
                      "data": "synthetic", "sweep": rows}))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--workload", default="tise_2e_16sd")
    ap.add_argument("--e2e-steps", type=int, default=2)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--precision", default="mixed", choices=list(PRECISIONS),
                    help="precision of the headline line (fp32: FP32-rounded step matrices, then refinement with "
                         "the double-single ones); the plain FP64 path is timed beside it")
    ap.add_argument("--no-extra", action="store_true",
                    help="skip the bounded measurements of the batched and real-time workloads")
    ap.add_argument("--extra-iterations", type=int, default=2,
                    help="timed Schwarz iterations per chunk of the batched extra measurement (after one warm-up)")
    ap.add_argument("--no-compare", action="store_true", help="skip the timing of the other precision")
    ap.add_argument("--iterations", type=int, default=0,
                    help="fixed Schwarz iterations per step instead of iterating to Res <= 1e-8 "
                         "(for the long real-time workload)")
    ap.add_argument("--batch-instances", type=int, default=512,
                    help="batched workload: first N instances of the 512 (a bounded run)")
    ap.add_argument("--max-steps", type=int, default=0,
                    help="batched workload: imaginary-time window cap (default: the instances' 5000)")
    ap.add_argument("--rows-per-task", type=int, default=0, help="batched workload: window row-task size")
    ap.add_argument("--window-variant", type=int, default=0,
                    help="batched workload, mixed precision: window kernel before autotuning (0 automatic, 1 two-phase, "
                         "3 split)")
    ap.add_argument("--no-autotune", action="store_true", help="keep the automatic window plan (no swr_autotune)")
    ap.add_argument("--antisymmetric", action="store_true",
                    help="2-electron imaginary-time workloads: the lowest antisymmetric state (initial Gaussian "
                         "centred at (0.8, -0.8)); the lower subdomain of each mirror pair is not solved")
    ap.add_argument("--learned-family", default="small", choices=["small", "16sd"],
                    help="--learned: the instance family (small: 2x2 subdomains, 40 steps; 16sd: 4x4 subdomains "
                         "of the real-time workload's geometry, 100 steps)")
    ap.add_argument("--learned-train", type=int, default=160, help="--learned: training instances")
    ap.add_argument("--learned-test", type=int, default=24, help="--learned: held-out instances")
    ap.add_argument("--learned-steps", type=int, default=1500, help="--learned: Adam steps")
    ap.add_argument("--learned", action="store_true",
                    help="learned initial traces: train the BF16 MLP on GPU-generated converged traces of the "
                         "reduced real-time family, then time held-out solves to Res <= 1e-8 from zero traces and "
                         "from the learned guess (inference and decoding included); one JSON line")
    ap.add_argument("--assembly", action="store_true",
                    help="time swr_assemble (quadrature, local matrices, orthonormalisation, e-e block, step-matrix "
                         "inversion) with the FP64 and the tensor-core contractions on the real-time 64-subdomain and "
                         "the 2-electron ground-state workloads; one JSON line")
    ap.add_argument("--real-time-converge", action="store_true",
                    help="the 64-subdomain real-time workload (K = 1024 complex, 1000 Crank-Nicolson steps) iterated "
                         "to Res <= 1e-8 in the headline precision: wall time, Schwarz iterations, residual history, "
                         "final norm and dipole; one JSON line")
    ap.add_argument("--lsd", action="store_true",
                    help="local orbitals and local Slater determinants at the paper's Test 1 sizes (L = 5, 10 orbitals "
                         "per subdomain, 45 determinants per subdomain): time of swr_lsd_build (best of three) and "
                         "Table 1's inner products; one JSON line")
    ap.add_argument("--sweep", action="store_true",
                    help="imaginary-time workloads: Schwarz convergence over a grid of time steps and Robin "
                         "constants, Robin and classical (Dirichlet) transmission; one JSON line")
    args = ap.parse_args()
    name = args.workload
    inst = workload(name)
    if args.antisymmetric:
        if name == BATCHED or inst.n_elec != 2 or inst.mode != "tise":
            raise SystemExit("--antisymmetric takes a 2-electron imaginary-time workload")
        inst = inst.replace(symmetry="antisymmetric", phi0_center=(0.8, -0.8))
    if name == BATCHED:
        inst = inst[:args.batch_instances]
        if args.max_steps > 0:
            inst = [i.replace(max_steps=args.max_steps) for i in inst]
    if args.impl == "reference":
        run_reference(args, inst, name)
        return

    import numpy as np
    import torch
    import torch.distributed as dist

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl", init_method="env://")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    from paper_1710_02401_gb300 import build as B
    B.build()
    from paper_1710_02401_gb300 import swr as S

    stream = torch.cuda.current_stream(dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    prec_of = {p: prec_code(S, p) for p in PRECISIONS}
    if name == BATCHED:
        run_batched(args, inst, (S, torch, dist, dev, stream, flush, world, rank, local))
        if world > 1:
            dist.destroy_process_group()
        return
    if args.assembly:
        if rank == 0:
            run_assembly(args, S)
        if world > 1:
            dist.destroy_process_group()
        return
    if args.real_time_converge:
        if rank == 0:
            run_real_time_converge(args, S)
        if world > 1:
            dist.destroy_process_group()
        return
    if args.lsd:
        if rank == 0:
            run_lsd(args, S)
        if world > 1:
            dist.destroy_process_group()
        return
    if args.learned:
        if rank == 0:
            run_learned(args)
        if world > 1:
            dist.destroy_process_group()
        return
    if args.sweep:
        if rank == 0:
            run_sweep(args, inst, name, S)
        if world > 1:
            dist.destroy_process_group()
        return

    def timed(prec_name, steps, warmup, sample_clocks):
        """W untimed + K timed steps (assemble + iterate to Res <= TOL), CUDA
        events on the library's stream, L2 flushed before every step."""
        s = S.SWR(inst, precision=prec_of[prec_name], device=str(dev), stream=stream,
                  window_variant=args.window_variant if prec_name != "fp64" else 0)
        tune = None
        if inst.mode == "tise" and not args.no_autotune:
            s.assemble()
            tune = s.autotune(steps=24)  # the window plan, chosen once (untimed)
        for _ in range(warmup):
            s.assemble()
            s.iterate(TOL if not args.iterations else 0.0, args.iterations or KMAX)
        torch.cuda.synchronize(dev)
        if world > 1:
            dist.barrier()
        sampler = ClockSampler(local) if sample_clocks else None
        if sampler:
            sampler.start()
        c0 = s.counters()
        times, reps = [], []
        for _ in range(steps):
            flush.zero_()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            s.assemble()
            rep, hist = s.iterate(TOL if not args.iterations else 0.0, args.iterations or KMAX)
            e1.record(stream)
            e1.synchronize()
            times.append(e0.elapsed_time(e1))
            reps.append(rep)
        torch.cuda.synchronize(dev)
        if world > 1:
            dist.barrier()
        c1 = s.counters()
        clocks = sampler.stop() if sampler else None
        t_ms = sum(times)
        solves = sum(r.subdomain_solves for r in reps)
        t_max, solves_all = t_ms, solves
        if world > 1:
            t = torch.tensor([t_ms], dtype=torch.float64, device=dev)
            dist.all_reduce(t, op=dist.ReduceOp.MAX)
            t_max = float(t.item())
            n = torch.tensor([solves], dtype=torch.float64, device=dev)
            dist.all_reduce(n, op=dist.ReduceOp.SUM)
            solves_all = int(n.item())
        d = {k: c1[k] - c0[k] for k in c1}
        return dict(s=s, value=solves_all / (t_max * 1e-3), t_max=t_max, reps=reps, counters=d, clocks=clocks,
                    plan=s.window_plan(), tune=tune, fp32_iters=[r.fp32_iterations for r in reps])

    main_run = timed(args.precision, args.steps, args.warmup, True)
    other = None
    if not args.no_compare:
        other_name = "fp64" if args.precision != "fp64" else "mixed"
        other = timed(other_name, max(1, min(args.steps, 2)), 1, False)
        other["name"] = other_name
    extras = None
    if world == 1 and not args.no_extra and name == "tise_2e_16sd":
        env = (S, torch, dist, dev, stream, flush, world, rank, local)
        extras = {"batched_uneven_512": extra_batched(args, env), "tdse_2e_64sd": extra_real_time(args, env)}
    third = None
    if not args.no_compare and args.precision != "mixed" and inst.mode == "tise":
        third = timed("mixed", max(1, min(args.steps, 2)), 1, False)
        third["name"] = "mixed"
    s = main_run["s"]
    reps = main_run["reps"]
    cnt = main_run["counters"]
    w_ms, w_launch, w_flops = cnt["window_ms"], cnt["window_launches"], cnt["window_flops"]
    # dominant kernel: the time window.  Roofline of the hot path's local step
    # (the factor-apply, HBM/L2-bound): algorithmic step-matrix bytes over the
    # window kernels' CUDA-event time against the measured HBM copy bandwidth
    hbm, hbm_src = hbm_peak()
    gbs = cnt["window_bytes_alg"] / (w_ms * 1e-3) / 1e9 if w_ms > 0 else 0.0
    tflops = w_flops / (w_ms * 1e-3) / 1e12 if w_ms > 0 else 0.0
    bpe = {"mixed": "8 bytes (FP32 hi/lo pair)", "fp64": "8 bytes (FP64)",
           "fp32": "4 bytes (FP32-rounded, hi plane) before the switch to the refinement, 8 after"}[args.precision]
    if inst.mode == "tdse":
        kname = RT_KERNEL.get(args.precision, "k_rt_window")
        if args.precision == "fp32":
            alg = (f"2 x {bpe} of G0 per complex element and sweep, (1 + m) sweeps per Crank-Nicolson step; "
                   "G0 (1.07 GB) does not fit in L2")
        else:
            alg = ("8 bytes of the symmetric G0 per complex element and sweep (its lower triangle, 28 + 28 bits per "
                   "component), (1 + m) sweeps per Crank-Nicolson step; the kernel is bound by its integer products")
        alu = {"achieved": tflops, "peak": FP32_PEAK_TFLOPS / 6.0 if args.precision == "fp32" else FIXED_PEAK_TFLOPS,
               "unit": "TFLOP/s", "algorithmic": "8 K^2 FP64-equivalent flops per complex sweep"}
    else:
        kname = {S.WINDOW_FUSED: "k_window_fused", S.WINDOW_SPLIT: "k_window_split",
                 S.WINDOW_RESIDENT: "k_window_resident", S.WINDOW_CLUSTER: "k_window_cluster"}.get(
            main_run["plan"]["variant"], "k_window_2ph<true>" if args.precision != "fp64" else FP64_WINDOW)
        if kname == "k_window_cluster":
            alg = (f"{bpe} of the step-matrix inverse per element, K^2 elements per local step solve (the "
                   "factor-apply); the cluster window keeps every subdomain's 2.65 MB of step matrix on chip "
                   "(G_hi in shared memory, G_lo in tensor memory) for the whole window, so these bytes are read "
                   "from SRAM and the fraction is the algorithmic rate against the HBM copy peak, not DRAM traffic")
        else:
            alg = (f"{bpe} of the step-matrix inverse per element, K^2 elements per local step solve (the "
                   "factor-apply); the 2-electron workload's 42.5 MB of step matrices stay in L2, so the kernel is "
                   "bounded by its per-step grid barrier and L2 latency, not by HBM")
        alu = {"achieved": tflops, "peak": FIXED_PEAK_TFLOPS if args.precision == "fp64" else FP32_PEAK_TFLOPS / 6.0,
               "unit": "TFLOP/s", "algorithmic": "2 K^2 FP64-equivalent flops per local step solve",
               "peak_source": "56-bit fixed-point products on the integer pipes (2.6 TFLOP/s FP64-equivalent; the FP64 "
                              "FMA rate is 1.01 TFLOP/s) or FP32 FMA rate / 6 (67.7 TFLOP/s / 6: a double-single "
                              "product-sum spends 12 FP32 operations per 2 FP64-equivalent flops), measured on this "
                              "pool's GB300 with independent FMA chains"}
    roof = {"kernel": kname, "bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
            "peak_source": hbm_src, "algorithmic": alg, "secondary_alu": alu}
    traffic, src = profiled_traffic(roof["kernel"])
    roof["traffic"] = traffic
    roof["traffic_source"] = src
    roof["window_ms_per_launch"] = w_ms / max(w_launch, 1)
    n_it = max(1, sum(r.iterations for r in reps))
    roof["post_window_ms_per_iteration"] = (cnt["step_ms"] - w_ms) / n_it
    roof["assemble_ms_per_step"] = cnt["assemble_ms"] / max(1, args.steps)
    # solved subdomains per step (antisymmetric states: one of each mirror pair)
    n_solved = inst.L * (inst.L + 1) // 2 if getattr(inst, "symmetry", "none") == "antisymmetric" else inst.n_sub
    roof["step_us"] = 1e3 * w_ms / max(1.0, cnt["solves"] / n_solved)
    launches = int(cnt["kernel_launches"])

    # end to end through the public API: setup from host descriptors, assembly,
    # iterations, read-back of energies and psi at all nodes, teardown
    e2e_val, h2d, d2h = None, 0, 0
    if args.e2e_steps > 0:
        e_solves, e_time = 0, 0.0
        for _ in range(args.e2e_steps):
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            se = S.SWR(inst, precision=prec_of[args.precision], device=str(dev), stream=stream)
            se.assemble()
            if inst.mode == "tise" and not args.no_autotune:
                se.autotune(steps=24)
            rep_e, _ = se.iterate(TOL if not args.iterations else 0.0, args.iterations or KMAX)
            energy = se.energy()
            psi = se.psi_nodes()
            ce = se.counters()
            se.close()
            torch.cuda.synchronize(dev)
            e_time += time.perf_counter() - t0
            e_solves += rep_e.subdomain_solves
            h2d, d2h = int(ce["h2d_bytes"]), int(ce["d2h_bytes"])
            del se
        e2e_val = e_solves / e_time

    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return
    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        v, desc, t_asm = oracle_sample(inst)
        cpu = {"value": v, "unit": "subdomain solves/s", "cores": os.cpu_count(), "kind": "oracle",
               "sample": desc}
    out = {
        "metric": METRIC, "value": main_run["value"], "unit": "subdomain solves/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": main_run["t_max"] / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": DTYPES[args.precision],
        "data": "synthetic", "config": workload_config(name, inst),
        "precision": args.precision,
        "time_to_residual_s": main_run["t_max"] / args.steps * 1e-3,
        "schwarz_iterations": [r.iterations for r in reps], "converged": all(r.converged for r in reps),
        "res_last": [r.res_last for r in reps],
        "energy": float(s.energy()[0]),
        "cvtot": float(s.cvtot()[0]),
        "roofline": roof,
        "cpu_baseline": cpu,
        "e2e": {"value": e2e_val, "unit": "subdomain solves/s", "h2d_bytes_per_step": h2d,
                "d2h_bytes_per_step": d2h},
        "gpu_launches": launches,
        "clocks": main_run["clocks"],
        "window_plan": {k: main_run["plan"][k] for k in ("variant", "rows_per_task", "tasks", "ctas", "graph",
                                                         "tensor_contractions")},
    }
    if main_run["tune"] is not None:
        out["window_plan"]["autotune_us_per_step"] = {"chosen": 1e6 * main_run["tune"]["seconds_per_step"],
                                                      "automatic": 1e6 * main_run["tune"]["seconds_default"]}
    if other is not None:
        o_reps = other["reps"]
        out["other_precision"] = {
            "precision": other["name"], "value": other["value"],
            "time_to_residual_s": other["t_max"] / len(o_reps) * 1e-3,
            "schwarz_iterations": [r.iterations for r in o_reps],
            "energy": float(other["s"].energy()[0]),
            "speedup_of_headline": main_run["value"] / other["value"],
        }
        if inst.mode == "tise":
            out["other_precision"]["energy_difference_relative"] = abs(out["energy"] - out["other_precision"]["energy"]) \
                / abs(out["other_precision"]["energy"])
    if third is not None:
        t_reps = third["reps"]
        out["double_single_precision"] = {
            "value": third["value"], "time_to_residual_s": third["t_max"] / len(t_reps) * 1e-3,
            "schwarz_iterations": [r.iterations for r in t_reps], "energy": float(third["s"].energy()[0]),
            "speedup_of_headline": main_run["value"] / third["value"]}
    if args.precision == "fp32":
        out["fp32_phase_iterations"] = main_run["fp32_iters"]
    if extras is not None:
        out["extra_workloads"] = extras
    print(json.dumps(out))
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
