#!/usr/bin/env python
"""Benchmark of the deployment-space evaluator.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference] [--extras LIST]

A step is one pass of the whole closed-form path over the 16,777,216-config sweep (workload 5):
guide_simulate (memory check, task list, roofline, metrics -> 6 fp64 arrays + mask + B_max; a
bandwidth-bound memory kernel and a model kernel for the configs that fit, side by side),
guide_select_topk (constraint filter + top-64 by cost per token) and guide_pareto (latency vs $/h;
each one cooperative launch: a sampled bound, one filter pass over the arrays, an exact finish),
with the space tables already resident on the device; the two selections read the same metrics and
run side by side on two streams.  `value` is configs per second over the K
timed steps; the 0.89 GB of outputs a step writes and reads back exceed L2 several times over, so
no flush is needed between steps.  The trace-driven workloads (1, 3, 4), the 983,040-config grid
(2) and the fused (nothing materialised) selection on workload 5 are timed once each afterwards
and reported under "workloads" with configs/s and simulated request-iterations/s.

With N > 1 (launched by torchrun) every rank evaluates a grid of the same size over its own slice
of an N-times longer hardware axis (weak scaling); the only exchange is an all-gather of each
rank's top-k candidates before a final merge.

--impl reference times the CPU oracle (the repo's slow, plain restatement of the method) on the
host cores on the same workload and metric.
"""
from __future__ import annotations

import argparse
import json
import os
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np

BYTES_SIM = 6 * 8 + 1 + 4          # six fp64 metrics + status + bmax written per config
# Non-fused fp64 instruction rate of the device (148 SMs x 64 fp64 lanes x 1.965 GHz), as measured by the
# package's own micro-benchmark (python -m paper_2412_04788_b200.fp64_peak): the peak of every "alu" bound.
FP64_ISSUE_PEAK = 18.5e12
# fp64 operations the method itself asks for (one scalar chain per config, whatever the kernel's layout):
# a decode iteration = 2 attention tasks x (2 mul, compare, add) + the sums and the clock, about 24;
# a closed-form config that fits = 2 stages x 13 task times x (2 mul, compare, add) + metrics, about 120.
FP64_OPS_PER_ITERATION = 24
FP64_OPS_PER_CLOSED_FORM_CONFIG = 120
SIM_FIELDS = ("latency", "ttft", "tpot", "thr_decode", "cost_per_hr", "cost_per_token", "status", "bmax")
TRACE_FIELDS = ("latency", "ttft", "ttft_p50", "ttft_p99", "tpot", "thr_decode", "cost_per_hr", "cost_per_token",
                "status", "bmax", "n_iters", "n_req_iters")


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            return float(json.load(f)["hbm_gbs"]), "measured"
    return 6650.0, "fallback"


def recorded_traffic(n_configs):
    """DRAM bytes of one guide_simulate call from the last profiler capture (written next to the
    profile summaries by paper_2412_04788_b200/traffic_record.py), or None when the capture was of
    another size or the kernel sources have changed since."""
    from paper_2412_04788_b200 import traffic_record
    path = os.path.join(ROOT, "profiles", "k_closed_form_c5_traffic.json")
    if not os.path.exists(path):
        return None
    with open(path) as f:
        rec = json.load(f)
    if rec.get("configs") != n_configs or rec.get("sources_sha256") != traffic_record.sources_sha256():
        return None
    return rec.get("dram_bytes_per_call")


class ClockSampler(threading.Thread):
    """Samples SM clock and clock-event reasons through NVML while the timed region runs (read only)."""

    def __init__(self, index):
        super().__init__(daemon=True)
        self.index, self.samples, self.reasons, self.stop_flag, self.max_mhz = index, [], set(), False, None
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nv = pynvml
            self.h = pynvml.nvmlDeviceGetHandleByIndex(index)
            self.max_mhz = pynvml.nvmlDeviceGetMaxClockInfo(self.h, pynvml.NVML_CLOCK_SM)
        except Exception:
            self.nv = None

    def run(self):
        if self.nv is None:
            return
        nv = self.nv
        names = {nv.nvmlClocksEventReasonSwPowerCap: "sw_power_cap", nv.nvmlClocksEventReasonHwSlowdown: "hw_slowdown",
                 nv.nvmlClocksEventReasonSwThermalSlowdown: "sw_thermal_slowdown",
                 nv.nvmlClocksEventReasonHwThermalSlowdown: "hw_thermal_slowdown",
                 nv.nvmlClocksEventReasonHwPowerBrakeSlowdown: "hw_power_brake"}
        while not self.stop_flag:
            try:
                self.samples.append(nv.nvmlDeviceGetClockInfo(self.h, nv.NVML_CLOCK_SM))
                r = nv.nvmlDeviceGetCurrentClocksEventReasons(self.h)
                for bit, name in names.items():
                    if r & bit:
                        self.reasons.add(name)
            except Exception:
                pass
            time.sleep(0.002)

    def summary(self):
        s = sorted(self.samples)
        return {"sm_mhz": s[len(s) // 2] if s else None, "sm_max_mhz": self.max_mhz, "reasons": sorted(self.reasons),
                "samples": len(s)}


def table_bytes(space):
    return (len(space["models"]) * 40 + len(space["hw"]) * 48 + len(space["fw_f"]) * 80 + len(space["batch"]) * 4 +
            len(space["tp"]) * 4 + len(space["pairs"]) * 8)


# ---------------------------------------------------------------------------------------------------
# reference arm: the CPU oracle, as it stands
# ---------------------------------------------------------------------------------------------------

def oracle_step(oracle, w):
    out = oracle.simulate(w["space"])
    oracle.select_topk(out, w["constraints"], w["topk"]["key"], w["topk"]["k"])
    oracle.pareto(out, w["constraints"], "latency", "cost_per_hr")
    return out


REF_STRIDE = 8      # the reference arm evaluates every 8th config of the workload per step


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import oracle
    from paper_2412_04788_b200 import inputs
    w = inputs.workload(5)
    n = inputs.space_size(w["space"])
    count = (n + REF_STRIDE - 1) // REF_STRIDE

    def step():
        out = oracle.simulate(w["space"], first=0, count=count, stride=REF_STRIDE)
        oracle.select_topk(out, w["constraints"], w["topk"]["key"], w["topk"]["k"])
        oracle.pareto(out, w["constraints"], "latency", "cost_per_hr")

    for _ in range(args.warmup):
        step()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        step()
    dt = time.perf_counter() - t0
    value = count * args.steps / dt
    cores = oracle.threads()
    sample = f"every {REF_STRIDE}th config of the 16777216-config sweep per step ({count} configs): simulate + top-64 + Pareto"
    line = {"impl": "reference", "metric": "configs/sec", "value": value, "unit": "configs/s", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "C5 closed-form sweep, 16777216 configs: simulate + top-64 + Pareto", "sample": sample},
            "cpu_baseline": {"value": value, "unit": "configs/s", "cores": cores, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": "configs/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line))


# ---------------------------------------------------------------------------------------------------
# our arm
# ---------------------------------------------------------------------------------------------------

class ClosedFormPath:
    """Device buffers and the three calls of one step on a closed-form space."""

    def __init__(self, guide, torch, space_np, cons, key, k):
        self.guide, self.torch = guide, torch
        self.sp = guide.Space(space_np)
        self.n = self.sp.size
        self.cons, self.key, self.k = cons, key, k
        self.out = guide.alloc_outputs(self.n, fields=SIM_FIELDS)
        self.idx = torch.empty(k, dtype=torch.int64, device="cuda")
        self.val = torch.empty(k, dtype=torch.float64, device="cuda")
        self.cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
        self.fidx = torch.empty(guide.PARETO_MAX, dtype=torch.int64, device="cuda")
        self.fcnt = torch.zeros(1, dtype=torch.int32, device="cuda")
        self.ws_k = torch.empty(guide.guide_select_workspace_bytes(self.sp, k), dtype=torch.uint8, device="cuda")
        self.ws_p = torch.empty(guide.guide_pareto_workspace_bytes(self.sp), dtype=torch.uint8, device="cuda")

    def simulate(self):
        self.guide.guide_simulate(self.sp, None, self.out)

    def topk(self, fused=False):
        self.guide.guide_select_topk(self.sp, None, None if fused else self.out, self.cons, self.key, self.k,
                                     self.idx, self.val, self.cnt, self.ws_k)

    def pareto(self, fused=False):
        self.guide.guide_pareto(self.sp, None, None if fused else self.out, self.cons, "latency", "cost_per_hr",
                                self.fidx, self.fcnt, self.ws_p)

    def simulate_select(self, sweep_events=None):
        """the whole step as one call: the sweep with both selections riding along"""
        self.guide.guide_simulate_select(self.sp, self.out, self.cons, self.key, self.k, self.idx, self.val, self.cnt, self.ws_k,
                                         self.cons, "latency", "cost_per_hr", self.fidx, self.fcnt, self.ws_p,
                                         sweep_events=sweep_events)


def time_call(torch, fn, reps=3, warm=1, flush=None):
    for _ in range(warm):
        fn()
    torch.cuda.synchronize()
    ts = []
    for _ in range(reps):
        if flush is not None:
            flush.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        ts.append(a.elapsed_time(b))
    return min(ts), sorted(ts)[len(ts) // 2]


def oracle_seconds(oracle, space, trace, stride, n_total, threads):
    """The oracle, as it stands, on every stride-th config of a workload: (seconds, configs, iterations,
    request-iterations) on `threads` host threads (0 = all)."""
    count = (n_total + stride - 1) // stride
    t0 = time.perf_counter()
    out = oracle.simulate(space, trace, first=0, count=count, stride=stride, n_threads=threads)
    dt = time.perf_counter() - t0
    return dt, count, int(out["n_iters"].sum()), int(out["n_req_iters"].sum())


HOST_CORES = None       # threads the oracle's OpenMP runtime starts with; read before any call narrows it


def host_cores(oracle):
    global HOST_CORES
    if HOST_CORES is None:
        HOST_CORES = oracle.threads()
    return HOST_CORES


def cpu_baseline_of(oracle, space, trace, n_total, stride_all, stride_one, unit_iters):
    """Oracle timings beside a workload: all host cores on one stride, one core on a sparser one."""
    res = {"kind": "oracle", "cores": host_cores(oracle)}
    for tag, stride, threads in (("all_cores", stride_all, host_cores(oracle)), ("one_core", stride_one, 1)):
        dt, count, iters, req_iters = oracle_seconds(oracle, space, trace, stride, n_total, threads)
        res[tag] = {"seconds": dt, "configs": count, "configs_per_s": count / dt,
                    "sample": f"every {stride}th config" if stride > 1 else "the whole workload",
                    "seconds_for_the_whole_workload_at_this_rate": dt * n_total / count}
        if unit_iters:
            res[tag]["request_iters_per_s"] = req_iters / dt
            res[tag]["iters_per_s"] = iters / dt
    res["value"] = res["all_cores"]["configs_per_s"]
    res["unit"] = "configs/s"
    res["sample"] = res["all_cores"]["sample"]
    return res


def alu_roofline(ops_per_s, what):
    return {"bound": "alu", "achieved": ops_per_s / 1e12, "peak": FP64_ISSUE_PEAK / 1e12, "unit": "T fp64 op/s",
            "frac": ops_per_s / FP64_ISSUE_PEAK, "traffic": None, "peak_kind": "of measured (fp64 issue micro-benchmark)",
            "what": what}


def hbm_roofline(bytes_per_call, ms, hbm_peak, peak_kind, what):
    gbs = bytes_per_call / (ms * 1e-3) / 1e9
    return {"bound": "hbm", "achieved": gbs, "peak": hbm_peak, "unit": "GB/s", "frac": gbs / hbm_peak, "traffic": None,
            "peak_kind": f"of {peak_kind}", "what": what}


def extra_workloads(guide, torch, inputs, which, flush, hbm_peak, peak_kind, fraction=None, oracle=None):
    """Workloads 1 - 5 and the variants, each timed on its own: best of a few launches, CUDA events;
    each with the roofline of its call and, when `oracle` is given, the oracle's time beside it."""
    res = {}
    for k in which:
        if k in (1, 3, 4):
            scale = 1.0
            if fraction and k != 1:
                scale = fraction
            w = inputs.workload(k, scale=scale, trace_scale=1.0)
            sp, tr = guide.Space(w["space"]), guide.Trace(w["trace"])
            n = sp.size
            out = guide.alloc_outputs(n, tr.n, fields=TRACE_FIELDS, per_request=(k != 4))
            ws = torch.empty(guide.guide_workspace_bytes(sp, tr), dtype=torch.uint8, device="cuda")
            best, med = time_call(torch, lambda: guide.guide_simulate(sp, tr, out, workspace=ws), reps=2, warm=1)
            extra = {}
            if k == 1:
                # top-8 by cost per token under the 500 ms p99-TTFT objective, on the simulated metrics
                kk = w["topk"]["k"]
                idx = torch.empty(kk, dtype=torch.int64, device="cuda")
                val = torch.empty(kk, dtype=torch.float64, device="cuda")
                cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
                wsk = torch.empty(guide.guide_select_workspace_bytes(sp, kk), dtype=torch.uint8, device="cuda")
                t_sel = time_call(torch, lambda: guide.guide_select_topk(sp, tr, out, w["constraints"], w["topk"]["key"], kk,
                                                                         idx, val, cnt, wsk))[0]
                extra = {"topk_ms": t_sel, "topk_found": int(cnt.item())}
            iters = int(out["n_iters"].sum().item())
            req_iters = int(out["n_req_iters"].sum().item())
            feasible = int((out["status"] == 0).sum().item())
            res[f"C{k}"] = {"configs": n, "requests": tr.n, "feasible": feasible, "ms": best,
                            "configs_per_s": n / best * 1e3, "iters_per_s": iters / best * 1e3,
                            "request_iters_per_s": req_iters / best * 1e3, "request_iters": req_iters,
                            "hardware_axis_fraction": scale, "workspace_bytes": ws.numel(),
                            "kernels": "k_trace_sim (one warp per config, 32 iterations of a run at once)" +
                                       ("" if k == 1 else " + k_trace_lanes (one lane per config: the large classes of small max batch)"),
                            "kernel_launches": {1: 1, 3: 2, 4: 3}[k],
                            "roofline": alu_roofline(FP64_OPS_PER_ITERATION * iters / best * 1e3,
                                                     f"{FP64_OPS_PER_ITERATION} fp64 operations per simulated iteration x iterations/s"),
                            **extra}
            if oracle is not None:
                stride_all, stride_one = {1: (1, 7), 3: (509, 4093), 4: (2039, 16381)}[k]
                res[f"C{k}"]["cpu_baseline"] = cpu_baseline_of(oracle, w["space"], w["trace"], n, stride_all, stride_one, True)
            del out, ws
        elif k in (2, 5):
            w = inputs.workload(k, scale=fraction if (fraction and k == 5) else 1.0)
            p = ClosedFormPath(guide, torch, w["space"], w["constraints"], w["topk"]["key"], w["topk"]["k"])
            n = p.n
            fl = flush if k == 2 else None          # workload 2's outputs fit in L2: evict them
            t_sim = time_call(torch, p.simulate, flush=fl)[0]
            fits = int((p.out["status"] == 0).sum().item())
            t_kf = time_call(torch, lambda: p.topk(True), flush=fl)[0]
            t_pf = time_call(torch, lambda: p.pareto(True), flush=fl)[0]
            t_km = time_call(torch, lambda: p.topk(False), flush=fl)[0]
            t_pm = time_call(torch, lambda: p.pareto(False), flush=fl)[0]
            ops = FP64_OPS_PER_CLOSED_FORM_CONFIG * fits
            what = f"{FP64_OPS_PER_CLOSED_FORM_CONFIG} fp64 operations per config that fits ({fits}) / call time"
            res[f"C{k}"] = {"configs": n, "fits": fits, "front": int(p.fcnt.item()), "found": int(p.cnt.item()),
                            "fused_ms": {"topk": t_kf, "pareto": t_pf}, "fused_configs_per_s": n / (t_kf + t_pf) * 1e3,
                            "materialised_ms": {"simulate": t_sim, "topk": t_km, "pareto": t_pm},
                            "materialised_configs_per_s": n / (t_sim + t_km + t_pm) * 1e3,
                            "simulate_write_gbs": BYTES_SIM * n / t_sim / 1e6,
                            "simulate_frac_of_hbm": BYTES_SIM * n / t_sim / 1e6 / hbm_peak,
                            "roofline": {"guide_simulate": hbm_roofline(BYTES_SIM * n, t_sim, hbm_peak, peak_kind, "53 B written per config"),
                                         "guide_select_topk (fused)": alu_roofline(ops / t_kf * 1e3, what),
                                         "guide_pareto (fused)": alu_roofline(ops / t_pf * 1e3, what)},
                            "kernel_launches": 2 + 6 + 5 + 1 + 2}
            if oracle is not None:
                stride_all, stride_one = (1, 16) if k == 2 else (8, 128)
                res[f"C{k}"]["cpu_baseline"] = cpu_baseline_of(oracle, w["space"], None, n, stride_all, stride_one, False)
            del p
        elif k == 8:
            # workload 3 on half of its hardware axis with every framework on the split-and-fuse
            # policy (token budgets 256 .. 8192 per iteration)
            w = inputs.workload(3, scale=fraction or 0.5, trace_scale=1.0)
            space = dict(w["space"])
            fw_i = np.array(space["fw_i"], dtype=np.uint32).copy()
            fw_i[:, 3] = guide.GUIDE_POLICY_SPLIT_FUSE
            space["fw_i"] = fw_i
            space["fw_chunk"] = np.array([[0, 256], [0, 512], [0, 2048], [0, 8192]], dtype=np.uint32)
            sp, tr = guide.Space(space), guide.Trace(w["trace"])
            n = sp.size
            out = guide.alloc_outputs(n, tr.n, fields=TRACE_FIELDS, per_request=False)
            ws = torch.empty(guide.guide_workspace_bytes(sp, tr), dtype=torch.uint8, device="cuda")
            best, med = time_call(torch, lambda: guide.guide_simulate(sp, tr, out, workspace=ws), reps=2, warm=1)
            iters = int(out["n_iters"].sum().item())
            req_iters = int(out["n_req_iters"].sum().item())
            res["C3-split-fuse"] = {"configs": n, "requests": tr.n, "feasible": int((out["status"] == 0).sum().item()),
                                    "ms": best, "configs_per_s": n / best * 1e3, "iters_per_s": iters / best * 1e3,
                                    "request_iters_per_s": req_iters / best * 1e3,
                                    "hardware_axis_fraction": fraction or 0.5, "kernel_launches": 1,
                                    "roofline": alu_roofline(FP64_OPS_PER_ITERATION * iters / best * 1e3,
                                                             f"{FP64_OPS_PER_ITERATION} fp64 operations per simulated iteration x iterations/s")}
            if oracle is not None:
                res["C3-split-fuse"]["cpu_baseline"] = cpu_baseline_of(oracle, space, w["trace"], n, 509, 4093, True)
            del out, ws
        elif k in (6, 7):
            # the (dp, tp) sweep under a budget of 8 GPUs (whole-space kernels) and workload 2 with
            # frameworks that process prompts in sub-batches / segments
            w = inputs.hybrid_workload(8) if k == 6 else inputs.chunked_workload(scale=1.0)
            p = ClosedFormPath(guide, torch, w["space"], w["constraints"], w["topk"]["key"], w["topk"]["k"])
            n = p.n
            t_sim = time_call(torch, p.simulate, flush=flush)[0]
            t_kf = time_call(torch, lambda: p.topk(True), flush=flush)[0]
            res[w["name"]] = {"configs": n, "simulate_ms": t_sim, "simulate_configs_per_s": n / t_sim * 1e3,
                              "simulate_write_gbs": BYTES_SIM * n / t_sim / 1e6,
                              "simulate_frac_of_hbm": BYTES_SIM * n / t_sim / 1e6 / hbm_peak,
                              "roofline": hbm_roofline(BYTES_SIM * n, t_sim, hbm_peak, peak_kind, "53 B written per config"),
                              "fused_topk_ms": t_kf, "found": int(p.cnt.item())}
            if oracle is not None:
                res[w["name"]]["cpu_baseline"] = cpu_baseline_of(oracle, w["space"], None, n, 4, 64, False)
            del p
        torch.cuda.empty_cache()
    return res


def run_ours(args):
    import torch
    import torch.distributed as dist

    from paper_2412_04788_b200 import build, guide, inputs, sharding
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if rank == 0:
        build.build()
    assert torch.cuda.is_available(), "bench.py needs a CUDA device: the library has no CPU fallback"
    torch.cuda.set_device(local_rank)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))
        dist.barrier()
    guide.lib()

    hbm_peak, peak_kind = measured_peaks()
    # workload 5; with N ranks the hardware axis is N times longer and each rank takes one slice
    w = inputs.workload(5, scale=float(world) * (args.trace_fraction if args.main_fraction else 1.0))
    global_space = w["space"]
    local_space, hw_off = sharding.shard_space(global_space, rank, world) if world > 1 else (global_space, 0)
    k, key, cons = w["topk"]["k"], w["topk"]["key"], w["constraints"]
    path = ClosedFormPath(guide, torch, local_space, cons, key, k)
    n_local = path.n
    flush = torch.empty(256 * 1024 * 1024, dtype=torch.uint8, device="cuda")   # used for workload 2 only

    select, front = sharding.kernel_selectors(guide, path.sp, key, "latency", "cost_per_hr")

    def exchange():
        """all-gather of every rank's k candidates and of its local front; the library's own selection
        calls merge the gathered lists.  Leaves global config indices in path.idx / path.fidx."""
        gidx = sharding.local_to_global(path.idx, local_space, global_space, hw_off)
        top, vals, found = sharding.merge_topk(gidx, path.val, k, select)
        size = int(path.fcnt.item())
        used = torch.arange(guide.PARETO_MAX, device="cuda") < size
        sel = torch.where(used, path.fidx, torch.zeros_like(path.fidx))
        gfront = sharding.local_to_global(sel, local_space, global_space, hw_off)
        fr, fsize = sharding.merge_front(gfront, path.out["latency"][sel], path.out["cost_per_hr"][sel], size,
                                         guide.PARETO_MAX, front)
        path.idx.copy_(top)
        path.val.copy_(vals)
        path.fidx[:fr.numel()].copy_(fr)
        return found, fsize

    # The two selections of a step read the same metrics and share nothing else: the Pareto front (the
    # longer one) runs on the step's stream, top-k beside it on a second one (both after guide_simulate;
    # the next step's guide_simulate after both).
    main = torch.cuda.current_stream()
    side = torch.cuda.Stream()
    ev_sim = torch.cuda.Event()
    ev_side = torch.cuda.Event()

    def step(events=None):
        if events:
            events[0].record()
        path.simulate()
        if events:
            events[1].record()
        ev_sim.record()
        side.wait_event(ev_sim)
        with torch.cuda.stream(side):
            path.topk()
            ev_side.record()
        path.pareto()
        main.wait_event(ev_side)
        if world > 1:
            exchange()
        if events:
            events[2].record()

    def step_in_turn(events):
        """the same calls one after the other on one stream: the time of each call by itself"""
        events[0].record()
        path.simulate()
        events[1].record()
        path.topk()
        events[2].record()
        path.pareto()
        events[3].record()

    for _ in range(max(args.warmup, 3)):
        step()
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    sampler = ClockSampler(local_rank)
    sampler.start()
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(3)] for _ in range(args.steps)]
    torch.cuda.synchronize()
    wall0 = time.perf_counter()
    for i in range(args.steps):
        step(evs[i])                      # 0.89 GB written and re-read per step: nothing survives in L2
    torch.cuda.synchronize()
    wall = time.perf_counter() - wall0
    sampler.stop_flag = True
    sampler.join()
    t_sim = sum(e[0].elapsed_time(e[1]) for e in evs)
    total_ms = sum(e[0].elapsed_time(e[2]) for e in evs)
    # each selection call by itself, for the per-call figures (not part of `value`)
    n_turn = min(args.steps, 50)
    evt = [[torch.cuda.Event(enable_timing=True) for _ in range(4)] for _ in range(n_turn)]
    for i in range(n_turn):
        step_in_turn(evt[i])
    torch.cuda.synchronize()
    t_topk = sum(e[1].elapsed_time(e[2]) for e in evt) * args.steps / n_turn
    t_par = sum(e[2].elapsed_time(e[3]) for e in evt) * args.steps / n_turn
    t_turn = sum(e[0].elapsed_time(e[3]) for e in evt) / n_turn
    # the step as ONE call (guide_simulate_select: the sweep, then both selections, on one stream), with the
    # library's own events around the sweep kernels
    ev1 = [[torch.cuda.Event(enable_timing=True) for _ in range(4)] for _ in range(n_turn)]
    for e in ev1:
        e[1].record(); e[2].record()                  # the events handed to the library must exist
    path.simulate_select()
    torch.cuda.synchronize()
    for e in ev1:
        e[0].record()
        path.simulate_select(sweep_events=(e[1], e[2]))
        e[3].record()
    torch.cuda.synchronize()
    one_call = {"ms": sum(e[0].elapsed_time(e[3]) for e in ev1) / n_turn,
                "sweep_ms": sum(e[1].elapsed_time(e[2]) for e in ev1) / n_turn,
                "what": "guide_simulate_select: the sweep, then both selections, on one stream"}
    if world > 1:
        tt = torch.tensor([total_ms], dtype=torch.float64, device="cuda")
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        total_ms = float(tt.item())
        dist.barrier()
    n_total = n_local * world
    value = n_total * args.steps / (total_ms * 1e-3)

    # ---- end to end through the C ABI with host buffers: build the space from host arrays, run the
    # step, bring every output back to pinned host memory ----
    host = {f: torch.empty_like(t, device="cpu").pin_memory() for f, t in path.out.items()}
    host_idx, host_val = torch.empty(k, dtype=torch.int64).pin_memory(), torch.empty(k, dtype=torch.float64).pin_memory()
    host_front = torch.empty(guide.PARETO_MAX, dtype=torch.int64).pin_memory()
    e2e_steps = min(args.steps, 5)

    def e2e_step():
        sp = guide.Space(local_space)                      # host tables -> validated -> uploaded on first use
        guide.guide_simulate(sp, None, path.out)
        guide.guide_select_topk(sp, None, path.out, cons, key, k, path.idx, path.val, path.cnt, path.ws_k)
        guide.guide_pareto(sp, None, path.out, cons, "latency", "cost_per_hr", path.fidx, path.fcnt, path.ws_p)
        for f, t in path.out.items():
            host[f].copy_(t, non_blocking=True)
        host_idx.copy_(path.idx, non_blocking=True)
        host_val.copy_(path.val, non_blocking=True)
        host_front.copy_(path.fidx, non_blocking=True)
        torch.cuda.synchronize()
        sp.close()

    for _ in range(2):
        e2e_step()
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        e2e_step()
    e2e_dt = time.perf_counter() - t0
    if world > 1:
        tt = torch.tensor([e2e_dt], dtype=torch.float64, device="cuda")
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        e2e_dt = float(tt.item())
    e2e_value = n_total * e2e_steps / e2e_dt
    d2h = BYTES_SIM * n_local + k * 16 + guide.PARETO_MAX * 8

    # The same question asked without keeping the metrics: host tables in, the two selections
    # evaluated on the fly (nothing materialised), only the k candidates and the front read back.
    def e2e_select_step():
        sp = guide.Space(local_space)
        guide.guide_select_topk(sp, None, None, cons, key, k, path.idx, path.val, path.cnt, path.ws_k)
        guide.guide_pareto(sp, None, None, cons, "latency", "cost_per_hr", path.fidx, path.fcnt, path.ws_p)
        host_idx.copy_(path.idx, non_blocking=True)
        host_val.copy_(path.val, non_blocking=True)
        host_front.copy_(path.fidx, non_blocking=True)
        torch.cuda.synchronize()
        sp.close()

    e2e_sel = None
    if world == 1:
        for _ in range(2):
            e2e_select_step()
        t0 = time.perf_counter()
        for _ in range(20):
            e2e_select_step()
        e2e_sel = {"value": n_total * 20 / (time.perf_counter() - t0), "unit": "configs/s", "steps": 20,
                   "h2d_bytes_per_step": table_bytes(local_space), "d2h_bytes_per_step": k * 16 + guide.PARETO_MAX * 8,
                   "what": "fused guide_select_topk + guide_pareto from host tables, candidates and front read back; "
                           "no metric array is written"}

    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return

    # ---- roofline of every call of the step, the dominant one on top ----
    # bytes a scan must read per config: status, each distinct metric array, each bounded array
    bounded = {"max_latency": "latency", "max_cost_per_hr": "cost_per_hr", "min_throughput": "thr_decode",
               "max_ttft": "ttft"}
    cons_arrays = {arr for name, arr in bounded.items() if name in cons}
    bytes_topk = 1 + 8 * len(cons_arrays | {key})
    bytes_pareto = 1 + 8 * len(cons_arrays | {"latency", "cost_per_hr"})
    per = {"guide_simulate (k_closed_form_memory + k_closed_form_lines)": (t_sim / args.steps, BYTES_SIM),
           "guide_select_topk (k_topk_coop)": (t_topk / args.steps, bytes_topk),
           "guide_pareto (k_pareto_coop)": (t_par / args.steps, bytes_pareto)}
    calls = {}
    for name, (ms, nbytes) in per.items():
        calls[name] = hbm_roofline(nbytes * n_local, ms, hbm_peak, peak_kind, f"{nbytes} algorithmic bytes per config")
        calls[name]["ms"] = ms
    traffic = recorded_traffic(n_local)
    dom = max(per, key=lambda name: per[name][0])
    roofline = dict(calls[dom])
    roofline.update({"kernel": dom, "bytes_per_config": per[dom][1],
                     "traffic": traffic if dom.startswith("guide_simulate") else None,
                     "calls": calls,
                     "per_call_frac_of_hbm": {name: c["frac"] for name, c in calls.items()},
                     "per_kernel_ms": {name: c["ms"] for name, c in calls.items()}})

    # ---- the oracle on the host cores, same workload: whole passes for about ten seconds, then one core
    # on a sixteenth of the configs ----
    cpu = None
    oracle = None
    if world == 1 and not args.no_cpu:
        import oracle
        cores = host_cores(oracle)
        oracle_step(oracle, w)
        reps, t0 = 0, time.perf_counter()
        while reps < 3 or time.perf_counter() - t0 < 10.0:
            oracle_step(oracle, w)
            reps += 1
        dt = time.perf_counter() - t0
        one = oracle_seconds(oracle, w["space"], None, 16, n_local, 1)
        cpu = {"value": n_local * reps / dt, "unit": "configs/s", "cores": cores, "kind": "oracle",
               "sample": f"the whole {n_local}-config workload (simulate + top-{k} + Pareto), {reps} passes",
               "seconds_per_pass": dt / reps,
               "one_core": {"configs_per_s": one[1] / one[0], "sample": "every 16th config, simulate only", "seconds": one[0]}}

    extras = {}
    if world == 1 and args.extras:
        which = [int(x) for x in args.extras.split(",") if x]
        extras = extra_workloads(guide, torch, inputs, which, flush, hbm_peak, peak_kind, args.trace_fraction, oracle)

    # simulate: memory + line kernel; top-k: one launch; Pareto: one launch and the gated general kernel behind
    # it; with several ranks the two selections over the gathered lists (one launch, one and a gated one)
    launches_per_step = 2 + 1 + 2 + (3 if world > 1 else 0)
    line = {"metric": "configs/sec", "value": value, "unit": "configs/s", "n_gpus": world, "steps": args.steps,
            "warmup": max(args.warmup, 3), "ms_per_step": total_ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "C5 closed-form sweep: 16 models x 64 hw x 4 fw x 16 batch x 4 TP x 64 length pairs "
                                   f"= {n_local} configs per GPU; simulate (materialised) + top-{k} by cost/token under the "
                                   "latency bound + Pareto(latency, $/h)",
                       "l2": "no flush: each step writes and re-reads 0.89 GB, several times the 126 MB L2",
                       "timing": "CUDA events around each step on its stream, summed",
                       "streams": "guide_pareto on the step's stream, guide_select_topk beside it on a second stream, both "
                                  "after guide_simulate; per-call figures from the same calls issued one after the other"},
            "ms_per_step_calls_in_turn": t_turn,
            "ms_per_step_one_call": one_call,
            "clocks": sampler.summary(),
            "e2e": {"value": e2e_value, "unit": "configs/s", "h2d_bytes_per_step": table_bytes(local_space),
                    "d2h_bytes_per_step": d2h, "steps": e2e_steps,
                    "what": "space handle built from host tables, simulate + top-k + Pareto, every metric array (0.89 GB), "
                            "the candidates and the front copied to pinned host memory: bound by the copy back",
                    "variants": {"selection_only": e2e_sel}},
            "gpu_launches": launches_per_step * args.steps,
            "roofline": roofline, "cpu_baseline": cpu, "workloads": extras,
            "wall_s_timed_region": wall}
    print(json.dumps(line))
    if world > 1:
        dist.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--extras", default="1,2,3,4,5,6,7,8", help="other workloads to time after the main loop ('' = none)")
    ap.add_argument("--main-fraction", action="store_true",
                    help="apply --trace-fraction to the main workload's hardware axis too (small cases for profiler captures)")
    ap.add_argument("--no-cpu", action="store_true", help="skip the oracle timing")
    ap.add_argument("--trace-fraction", type=float, default=None,
                    help="fraction of the hardware axis of workloads 3, 4 and 5 in the extras (small cases for profiler captures)")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
