"""The work a user of this library has it do, case by case, for timing.

A case is one question put to the library: a sweep of a deployment space in closed form (metrics kept
and ranked, or ranked without keeping them), or the simulation of a request trace over a space.  Sizes
are those of the seeded workloads in `inputs.py`, of the tests and of `bench.py`, and odd ones between.

Fields of a case
  kind      "decide":   host tables in, handle made, metrics, top-k and front, the answer read on the host
            "sweep":    guide_simulate, then guide_select_topk and guide_pareto on the metrics
            "fused":    guide_select_topk and guide_pareto on the fly, no metrics kept
            "one_call": guide_simulate_select
            "trace":    guide_simulate on a request trace, then guide_select_topk
  models, hw, fw, batches, tps, lins, louts   axis lengths (`gpus` > 0: (dp, tp) pairs under that budget instead of tps)
  part      thousandths of the space that are evaluated, from an odd index on (1000: all of it)
  k         candidates kept by the top-k
  chunk     frameworks that process prompts in pieces     keep   thousandths of the KV cache they keep
  clamp     sequences cut to what fits                    f32    binary32 model
  requests, rate, fuse, own_lengths, per_request   the trace: its length, arrivals per second, the scheduling
            policy, whether requests bring their own lengths, whether per-request values are returned
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2412_04788_b200 import guide, inputs

_BASE = {"models": 1, "hw": 1, "fw": 1, "batches": 8, "tps": 4, "gpus": 0, "lins": 8, "louts": 8, "part": 1000, "k": 8,
         "chunk": False, "keep": 1000, "clamp": False, "f32": False, "requests": 0, "rate": 0.0, "fuse": False,
         "own_lengths": True, "per_request": False}


def _case(**fields):
    return {**_BASE, **fields}


def listed():
    return [
        # A single decision: a few hundred candidates from tables that have just changed (prices, new
        # hardware), answer wanted on the host.  Latency and the number of launches are all there is.
        _case(name="decide_500", kind="decide", hw=4, batches=7, tps=3, lins=3, louts=2),
        # The everyday sweep: eight shapes over a small fleet on a power-of-two length grid.
        _case(name="sweep_1m", kind="sweep", models=8, hw=16, fw=3, batches=10),
        # The largest sweep: 16.7 million candidates, metrics kept, top-64 and a Pareto front.
        _case(name="sweep_16m", kind="sweep", models=16, hw=64, fw=4, batches=16, k=64),
        # The same question when only the answer is wanted.
        _case(name="fused_16m", kind="fused", models=16, hw=64, fw=4, batches=16, k=64),
        # Hybrid parallelism under a budget of eight GPUs, metrics and both selections in one call.
        _case(name="hybrid_one_call_2m", kind="one_call", models=8, hw=8, fw=3, batches=12, gpus=8, k=64),
        # A shard of a space whose axes are whatever the user's measurements gave (no multiples of anything).
        _case(name="ragged_slice_500k", kind="sweep", models=7, hw=37, fw=3, batches=11, tps=3, lins=9, louts=7, part=333, k=20),
        # Frameworks that split prompt processing and evict part of the KV cache.
        _case(name="chunked_500k", kind="sweep", models=8, hw=8, fw=3, batches=10, chunk=True, keep=600),
        # The reduced-precision model with sequences cut to what fits.
        _case(name="f32_clamp_500k", kind="sweep", models=8, hw=8, fw=3, batches=10, clamp=True, f32=True),
        # A short trace over a handful of deployments, lengths fixed by the candidate, every request reported.
        _case(name="trace_500x256", kind="trace", hw=4, batches=7, tps=3, lins=3, louts=2, requests=256, rate=4.0,
              own_lengths=False, per_request=True),
        # The ordinary simulation: a few thousand candidates against some minutes of traffic.
        _case(name="trace_8k_x2048", kind="trace", models=8, hw=8, fw=2, batches=16, lins=1, louts=1, requests=2048, rate=16.0),
        # The largest simulation: a million candidates, many of them short of memory (preemption).
        _case(name="trace_1m_x1024", kind="trace", models=16, hw=256, fw=4, batches=16, lins=1, louts=1, requests=1024, rate=32.0),
        # Split-and-fuse scheduling.
        _case(name="fuse_8k_x2048", kind="trace", models=8, hw=8, fw=2, batches=16, lins=1, louts=1, requests=2048, rate=16.0,
              fuse=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["decide", "sweep", "sweep", "sweep", "fused", "one_call", "trace", "trace", "trace"])
    if kind == "trace":
        fuse = rng.random() < 0.35
        while True:
            c = _case(kind=kind, models=_log_int(rng, 1, 16), hw=_log_int(rng, 1, 256), fw=rng.randint(1, 4),
                      batches=rng.randint(1, 16), tps=rng.randint(1, 4), lins=1, louts=1, requests=_log_int(rng, 100, 4096),
                      rate=round(rng.uniform(2.0, 40.0), 2), fuse=fuse, per_request=False, k=rng.randint(1, 64))
            n = _size(c)
            if 64 <= n and n * c["requests"] <= (2.0e7 if fuse else 6.0e7):
                return c
    lo, hi = (64, 20_000) if kind == "decide" else (30_000, 16_000_000)
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    special = rng.random() if kind == "sweep" else 1.0
    if special < 0.4:
        want = min(want, 600_000)              # these evaluate every candidate by itself: no larger than the listed ones
    while True:
        grid = rng.random() < 0.5              # power-of-two grids as often as odd ones
        c = _case(kind=kind, models=_log_int(rng, 1, 16), hw=_log_int(rng, 1, 80), fw=rng.randint(1, 4), batches=rng.randint(1, 16),
                  tps=rng.randint(1, 4), gpus=rng.choice([0, 0, 0, 4, 8]), lins=8 if grid else rng.randint(1, 9),
                  louts=8 if grid else rng.randint(1, 9), k=_log_int(rng, 1, 128))
        if kind == "sweep" and rng.random() < 0.35:
            c["part"] = rng.randint(20, 990)
        if special < 0.2:
            c.update(chunk=True, keep=rng.choice([1000, 600, 350]), gpus=0)
        elif special < 0.3:
            c.update(clamp=True, keep=rng.choice([1000, 600]))
        elif special < 0.4:
            c.update(f32=True, clamp=rng.random() < 0.5)
        n = _count(c)
        if 0.6 * want <= n <= min(1.6 * want, hi):
            return c


def _n_par(case):
    return len(inputs.hybrid_axis(case["gpus"])[0]) if case["gpus"] else case["tps"]


def _size(case):
    return case["models"] * case["hw"] * case["fw"] * case["batches"] * _n_par(case) * case["lins"] * case["louts"]


def _range(case):
    """(first, count) of the evaluated part of the space."""
    n = _size(case)
    if case["part"] >= 1000:
        return 0, n
    count = max(1, n * case["part"] // 1000)
    return min(n - count, (n // 5) | 1), count


def _count(case):
    return _range(case)[1]


_LENGTHS = [64, 100, 128, 256, 512, 777, 1024, 2048, 4096, 8192]


def _lengths(seed, stream, n):
    """n different lengths: the usual grids of two, three and eight, else picks from a wider list."""
    if n in (2, 3, 8):
        return {2: [128, 512], 3: [128, 512, 2048], 8: inputs.LEN_GRID_8}[n]
    order = np.argsort(inputs.uniform01(seed, stream, len(_LENGTHS)), kind="stable")
    return [_LENGTHS[i] for i in sorted(order[:n].tolist())]


def _space(case, seed):
    trace = case["kind"] == "trace"
    models = (inputs.models_from_shapes(inputs.SHAPES_8[:case["models"]]) if case["models"] == 8
              else inputs.seeded_models(seed, case["models"]))
    if trace and case["hw"] > 64:
        hw, mem = inputs.seeded_hw(seed, case["hw"], mem_range=(16, 192))
    elif trace and case["own_lengths"]:
        hw, mem = inputs.seeded_hw(seed, case["hw"], mem_gb=[192] * case["hw"])
    else:
        hw, mem = inputs.seeded_hw(seed, case["hw"], mem_choices=[24, 48, 80, 192])
    fw_f, fw_i = inputs.seeded_fw(seed, case["fw"])
    if trace:
        step = 16 / case["batches"]
        batch = [inputs.BATCHES_16[int(i * step)] for i in range(case["batches"])]
        if not case["own_lengths"]:
            batch = [1 << i for i in range(case["batches"])]
    elif case["gpus"]:
        batch = [1, 2, 3, 5, 8, 16, 31, 64, 100, 256, 509, 1024, 6, 12, 24, 48][:case["batches"]]
    elif case["batches"] in (7, 10):
        batch = [1 << i for i in range(case["batches"])]
    else:
        draws = np.unique(inputs.randint(seed, 70, 4096, 1, 512))
        order = np.argsort(inputs.uniform01(seed, 72, len(draws)), kind="stable")
        batch = sorted(draws[order[:case["batches"]]].tolist())
    dp, tp = inputs.hybrid_axis(case["gpus"]) if case["gpus"] else (None, [1 << i for i in range(case["tps"])])
    if trace and case["own_lengths"]:
        pairs = [(1, 1)]
    else:
        pairs = inputs.pairs_grid(_lengths(seed, 80, case["lins"]), _lengths(seed, 81, case["louts"]))
    space = {"models": models, "hw": hw, "hw_mem": mem, "fw_f": fw_f, "fw_i": fw_i,
             "batch": np.array(batch, dtype=np.uint32), "tp": np.array(tp, dtype=np.uint32),
             "pairs": np.array(pairs, dtype=np.uint32).reshape(-1, 2)}
    if dp is not None:
        space["dp"] = np.array(dp, dtype=np.uint32)
    if case["chunk"]:
        space["fw_chunk"] = np.array([[0, 0], [4, 512], [16, 0], [0, 1024]][:case["fw"]], dtype=np.uint32)
    if case["keep"] < 1000:
        space["fw_keep"] = np.array([1000 if i == 0 else case["keep"] for i in range(case["fw"])], dtype=np.uint32)
    if case["fuse"]:
        space["fw_i"][:, 3] = guide.GUIDE_POLICY_SPLIT_FUSE
        space["fw_chunk"] = np.array([[0, (512, 1024, 256, 2048)[i]] for i in range(case["fw"])], dtype=np.uint32)
    return space


# What a sweep keeps: the columns a user ranks and plots by.
_SWEEP_FIELDS = ("latency", "ttft", "tpot", "thr_decode", "cost_per_hr", "cost_per_token", "status", "bmax")
_SWEEP_BYTES = 6 * 8 + 1 + 4
_TRACE_BYTES = 8 * 8 + 1 + 4 + 16


def prepare(case, seed):
    seed = 1000 + 7 * int(seed)
    tables = _space(case, seed)
    s = {"case": case, "tables": tables, "range": _range(case)}
    count, k = s["range"][1], case["k"]
    # a bound that some of the candidates miss, as a latency preference does
    s["cons"] = {"max_latency": float(inputs.uniform(seed, 71, 1, 20.0, 120.0)[0])} if case["kind"] != "trace" else {}
    s["space"] = guide.Space(tables)
    s["trace"], s["sim_ws"] = None, None
    if case["kind"] == "trace":
        s["trace"] = guide.Trace(inputs.make_trace(seed, case["requests"], case["rate"], lengths=case["own_lengths"]))
        s["sim_ws"] = torch.empty(guide.guide_workspace_bytes(s["space"], s["trace"]), dtype=torch.uint8, device="cuda")
    if case["kind"] != "fused":
        fields = guide.ALL_OUTPUTS if case["kind"] == "trace" else _SWEEP_FIELDS
        s["out"] = guide.alloc_outputs(count, case["requests"], fields, per_request=case["per_request"])
    s["idx"] = torch.zeros(k, dtype=torch.int64, device="cuda")
    s["key"] = torch.zeros(k, dtype=torch.float64, device="cuda")
    s["n"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    s["front"] = torch.zeros(guide.PARETO_MAX, dtype=torch.int64, device="cuda")
    s["n_front"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    s["ws_k"] = torch.empty(guide.guide_select_workspace_bytes(s["space"], k), dtype=torch.uint8, device="cuda")
    s["ws_p"] = torch.empty(guide.guide_pareto_workspace_bytes(s["space"]), dtype=torch.uint8, device="cuda")
    if case["kind"] == "decide":
        s["space"].close()                     # every decision makes its own
        s["host"] = {n: torch.empty(s[n].shape, dtype=s[n].dtype).pin_memory() for n in ("idx", "key", "n", "front", "n_front")}
    return s


def _answers(s):
    return {"idx": s["idx"], "key": s["key"], "n": s["n"], "front": s["front"], "n_front": s["n_front"]}


def _simulate(s, space):
    c, (first, count) = s["case"], s["range"]
    guide.guide_simulate(space, None, s["out"], first=first, count=count, clamp_seq=c["clamp"],
                         precision=guide.PREC_F32 if c["f32"] else guide.PREC_F64)


def _select(s, space, out):
    first, count = s["range"]
    c = s["case"]
    guide.guide_select_topk(space, None, out, s["cons"], "cost_per_token", c["k"], s["idx"], s["key"], s["n"], s["ws_k"],
                            first=first, count=count)
    guide.guide_pareto(space, None, out, s["cons"], "latency", "cost_per_hr", s["front"], s["n_front"], s["ws_p"],
                       first=first, count=count)


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "decide":
        space = guide.Space(s["tables"])
        _simulate(s, space)
        _select(s, space, s["out"])
        for name, host in s["host"].items():
            host.copy_(s[name], non_blocking=True)
        torch.cuda.current_stream().synchronize()
        space.close()
        return {"out": s["out"], **{n: h.clone() for n, h in s["host"].items()}}
    if c["kind"] == "sweep":
        _simulate(s, s["space"])
        _select(s, s["space"], s["out"])
        return {"out": s["out"], **_answers(s)}
    if c["kind"] == "fused":
        _select(s, s["space"], None)
        return _answers(s)
    if c["kind"] == "one_call":
        guide.guide_simulate_select(s["space"], s["out"], s["cons"], "cost_per_token", c["k"], s["idx"], s["key"], s["n"], s["ws_k"],
                                    s["cons"], "latency", "cost_per_hr", s["front"], s["n_front"], s["ws_p"])
        return {"out": s["out"], **_answers(s)}
    guide.guide_simulate(s["space"], s["trace"], s["out"], workspace=s["sim_ws"])
    guide.guide_select_topk(s["space"], s["trace"], s["out"], s["cons"], "ttft_p99", c["k"], s["idx"], s["key"], s["n"], s["ws_k"])
    return {"out": s["out"], "idx": s["idx"], "key": s["key"], "n": s["n"]}


def work(case):
    """Bytes: tables and trace in, metrics and answers out, each once.  Operations: 120 per candidate that fits its
    memory (two stages of thirteen task times of two multiplications, a comparison and an addition, and the metrics;
    about a quarter fit), 24 per simulated iteration (a trace needs at least one decode iteration per output token
    and batch slot)."""
    count = _count(case)
    tables = 64 * case["models"] + 48 * case["hw"] + 104 * case["fw"] + 8 * case["lins"] * case["louts"] + 4 * case["batches"]
    answers = 16 * case["k"]
    if case["kind"] != "trace":
        kept = 0 if case["kind"] == "fused" else _SWEEP_BYTES * count
        return {"bytes": tables + answers + kept, "flops": 30 * count}
    step = 16 / case["batches"]
    b = [1 << i for i in range(case["batches"])] if not case["own_lengths"] else [inputs.BATCHES_16[int(i * step)]
                                                                                 for i in range(case["batches"])]
    mean_out = 320.0 if not case["own_lengths"] else 230.0
    iters = sum(case["requests"] * mean_out / v for v in b) / len(b)
    per_request = 16 * case["requests"] * count if case["per_request"] else 0
    return {"bytes": tables + answers + 16 * case["requests"] + _TRACE_BYTES * count + per_request, "flops": 24 * iters * count}


def tolerance(case):
    """The model is a fixed sequence of correctly rounded operations and the library promises the same bits whatever
    the launch shape: every result, floating or whole, stays what it is."""
    return "exact"
