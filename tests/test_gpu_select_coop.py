"""GPU parity of the one-launch selection over materialised metrics at the sizes where its parts change
hands: one block or a grid, whole rows or a ragged last one, the range in the sample's registers or
sampled, lists that fit or overflow; aligned arrays and arrays that allow no wide loads."""
import numpy as np
import pytest

import oracle
from paper_2412_04788_b200 import guide, inputs as I
from gpu_util import run_pareto, run_topk
from test_gpu_select_stream import synth, to_dev

pytestmark = pytest.mark.gpu

REGISTERS = 148 * 2 * 16 * 4 * 64        # configs a full grid's registers hold: beyond it one row out of every r is sampled,
SAMPLED = 148 * 16 * 4                   # ... at most this many rows


@pytest.fixture(scope="module")
def sp():
    return guide.Space(I.workload(5, scale=0.125)["space"])


def check(sp, host, dev, cons, key, k, n):
    idx, val, cnt = run_topk(sp, dev, cons, key, k, count=n)
    w_idx, w_val, w_cnt = oracle.select_topk(host, cons, key, k)
    assert cnt == w_cnt and np.array_equal(idx, w_idx), (n, key, k)
    assert np.array_equal(val.view(np.uint64), w_val.view(np.uint64)), (n, key, k)
    fidx, fcnt = run_pareto(sp, dev, cons, "latency", key, count=n)
    w_f, w_n = oracle.pareto(host, cons, "latency", key, cap=guide.PARETO_MAX)
    assert fcnt == w_n and np.array_equal(fidx, w_f), (n, key)


@pytest.mark.parametrize("n", [1, 2, 63, 65, 2047, 2048, 2049, 4097, 64 * 16 * 17 + 5, REGISTERS - 1, REGISTERS, REGISTERS + 1])
@pytest.mark.parametrize("aligned", [True, False])
def test_sizes(sp, n, aligned):
    import torch
    host = synth(n, 100 + n % 97, pass_frac=0.6)
    dev = to_dev(host)
    if not aligned:                          # entry 0 on an odd 8-byte (status: odd byte) address
        dev = {k: torch.cat([v[:1], v])[1:] for k, v in dev.items()}
    for cons in ({}, {"max_latency": 4.0, "min_throughput": 100.0, "max_cost_per_hr": 50.0}):
        for key, k in (("cost_per_token", 1), ("cost_per_hr", 128), ("throughput", 20)):
            check(sp, host, dev, cons, key, k, n)


def test_infinities_nan_and_negative_zero_order_as_in_the_accumulator_kernels(sp):
    """k = 129 goes through the accumulator kernels: its first 128 are the one-launch answer."""
    n = 300000
    rng = np.random.default_rng(5)
    host = synth(n, 77, pass_frac=1.0)
    keys = host["cost_per_token"]
    keys[:] = np.inf
    keys[rng.choice(n, 60, replace=False)] = rng.random(60)
    keys[rng.choice(n, 20, replace=False)] = 0.0
    keys[rng.choice(n, 20, replace=False)] = -0.0
    keys[rng.choice(n, 1000, replace=False)] = np.nan
    for size in (200, 2000, n):
        dev = to_dev({k: v[:size] for k, v in host.items()})
        a_idx, a_val, a_cnt = run_topk(sp, dev, {}, "cost_per_token", 128, count=size)
        b_idx, b_val, b_cnt = run_topk(sp, dev, {}, "cost_per_token", 129, count=size)
        assert a_cnt == min(b_cnt, 128) and np.array_equal(a_idx, b_idx[:128])
        assert np.array_equal(a_val.view(np.uint64), b_val[:128].view(np.uint64))


def hidden_from_the_sample(n):
    """Passing configs only in the rows the sample leaves out (one row out of every r, at a hashed place)."""
    rows = (n + 63) // 64
    assert n > REGISTERS
    r = -(-rows // SAMPLED)
    slot = np.arange(rows // r, dtype=np.uint64)
    sampled = slot * r + ((slot * 2654435761) % 2**32 >> 7) % r
    unsampled = np.setdiff1d(np.arange(n // 64), sampled)
    host = synth(n, 9)
    host["status"][:] = 2
    host["status"][(unsampled[:, None] * 64 + np.arange(64)).ravel()] = 0
    return host


def test_candidate_list_overflow_runs_the_filter_again(sp):
    """No bound from the sample: the survivor list overflows, the k-th pair is closed in on by counting and the
    filter repeats.  Keys fall, rise, are all equal, share their high bits, few and many of each."""
    n = 2_000_001
    host = hidden_from_the_sample(n)
    rng = np.random.default_rng(3)
    for keys in (np.arange(n, dtype=np.float64), -np.arange(n, dtype=np.float64), np.ones(n), 1.0 + np.arange(n)[::-1] * 2.0**-52,
                 rng.permutation(n) * 2.0**-1074, np.floor(rng.random(n) * 4.0) - 2.0, rng.standard_normal(n) * 1e300,
                 np.where(rng.random(n) < 0.02, 1.0, 2.0), np.where(np.arange(n) % 2_000 == 7, -np.inf, np.inf)):
        host["cost_per_token"] = keys
        dev = to_dev(host)
        for k in (1, 128):
            idx, val, cnt = run_topk(sp, dev, {}, "cost_per_token", k, count=n)
            w_idx, w_val, w_cnt = oracle.select_topk(host, {}, "cost_per_token", k)
            assert cnt == w_cnt and np.array_equal(idx, w_idx) and np.array_equal(val, w_val)
    cons = {"max_latency": 6.0, "min_throughput": 100.0, "max_cost_per_hr": 50.0, "max_ttft": 0.9, "ttft_stat": "p50"}
    host["cost_per_token"] = np.arange(n, dtype=np.float64)
    idx, val, cnt = run_topk(sp, to_dev(host), cons, "cost_per_token", 64, count=n)
    w_idx, w_val, w_cnt = oracle.select_topk(host, cons, "cost_per_token", 64)
    assert cnt == w_cnt and np.array_equal(idx, w_idx) and np.array_equal(val, w_val)


def test_overflow_inside_the_registers(sp):
    """The sample is everything, but too few groups of it have a passing config for a bound."""
    n = 1_000_003
    host = synth(n, 31)
    host["status"][:] = 2
    live = np.arange(10, 310)                # 19,200 configs in neighbouring rows: more than the list holds
    host["status"][(live[:, None] * 64 + np.arange(64)).ravel()] = 0
    for keys in (np.arange(n, dtype=np.float64), -np.arange(n, dtype=np.float64), np.ones(n)):
        host["cost_per_token"] = keys
        dev = to_dev(host)
        for k in (1, 64, 128):
            idx, val, cnt = run_topk(sp, dev, {}, "cost_per_token", k, count=n)
            w_idx, w_val, w_cnt = oracle.select_topk(host, {}, "cost_per_token", k)
            assert cnt == w_cnt and np.array_equal(idx, w_idx) and np.array_equal(val, w_val)


def test_overflow_takes_few_passes():
    """Keys that rise with the index are met worst first by a pass that starts at the end of the range.  The number
    of passes must not grow with the length of the range: 268 M configs, 2.4 GB."""
    import torch
    space = dict(I.workload(5)["space"])
    for name in ("hw", "hw_mem"):
        space[name] = np.concatenate([space[name]] * 16)
    sp = guide.Space(space)
    n = sp.size
    assert n == 1 << 28
    rows = n // 64
    r = -(-rows // SAMPLED)
    slot = torch.arange(rows // r, dtype=torch.int64, device="cuda")
    sampled = slot * r + ((slot * 2654435761) % 2**32 >> 7) % r
    status = torch.zeros(rows, 64, dtype=torch.uint8, device="cuda")
    status[sampled] = 2
    dev = {"status": status.reshape(-1), "cost_per_token": torch.arange(n, dtype=torch.float64, device="cuda")}
    plain = dict(dev, status=torch.zeros_like(dev["status"]))
    idx, val = torch.zeros(64, dtype=torch.int64, device="cuda"), torch.zeros(64, dtype=torch.float64, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(guide.guide_select_workspace_bytes(sp, 64), dtype=torch.uint8, device="cuda")

    def time_of(d):
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            guide.guide_select_topk(sp, None, d, {}, "cost_per_token", 64, idx, val, cnt, ws)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        want = torch.nonzero(d["status"][:1 << 16] == 0)[:64, 0]
        assert int(cnt.item()) == 64 and torch.equal(idx, want) and torch.equal(val, want.double())
        return min(times[1:])
    t_plain, t_hidden = time_of(plain), time_of(dev)
    assert t_hidden < 30 * t_plain, (t_plain, t_hidden)


@pytest.mark.parametrize("n", [REGISTERS + 1, REGISTERS + 64 * 8 * 3 + 63, 2_097_152, 2_000_003])
@pytest.mark.parametrize("shift", [0, 2, 4, 8])
def test_pass_over_a_long_range(sp, n, shift):
    """One to six arrays; status at every alignment the loads tell apart (16, 4 and no wide loads); the last chunk
    and the last row ragged; few, many and all rows with a config that passed its memory check."""
    import torch
    n -= shift                               # room inside the space's size for the shifted copy
    for frac in (0.001, 0.02, 1.0):
        host = synth(n, 200 + n % 89, pass_frac=frac)
        dev = to_dev(host)
        if shift:
            dev["status"] = torch.cat([dev["status"][:shift], dev["status"]])[shift:]
        for cons in ({}, {"max_latency": 4.0}, {"max_latency": 6.0, "min_throughput": 100.0, "max_cost_per_hr": 50.0, "max_ttft": 0.9,
                                               "ttft_stat": "p50"}):
            check(sp, host, dev, cons, "cost_per_token", 64, n)


def test_two_selections_on_two_streams_run_side_by_side():
    """A selection over a long range leaves room for another one: two on two streams take clearly less time than
    one after the other, and give the same answers."""
    import torch
    w = I.workload(5)
    big = guide.Space(w["space"])
    out = guide.alloc_outputs(big.size, 0, ("latency", "thr_decode", "cost_per_hr", "cost_per_token", "status"))
    guide.guide_simulate(big, None, out)
    dev = dict(dtype=torch.int64, device="cuda")
    res = [[torch.zeros(64, **dev), torch.zeros(64, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"),
            torch.zeros(guide.PARETO_MAX, **dev), torch.zeros(1, dtype=torch.int32, device="cuda")] for _ in range(2)]
    wk = torch.empty(guide.guide_select_workspace_bytes(big, 64), dtype=torch.uint8, device="cuda")
    wp = torch.empty(guide.guide_pareto_workspace_bytes(big), dtype=torch.uint8, device="cuda")
    main, side = torch.cuda.current_stream(), torch.cuda.Stream()

    def topk(r):
        guide.guide_select_topk(big, None, out, w["constraints"], "cost_per_token", 64, r[0], r[1], r[2], wk)

    def front(r):
        guide.guide_pareto(big, None, out, w["constraints"], "latency", "cost_per_hr", r[3], r[4], wp)

    def in_turn():
        topk(res[0])
        front(res[0])

    def beside():
        side.wait_stream(main)
        with torch.cuda.stream(side):
            topk(res[1])
        front(res[1])
        main.wait_stream(side)

    def time_of(f):
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                f()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times[1:])
    t_turn, t_beside = time_of(in_turn), time_of(beside)
    assert all(torch.equal(a, b) for a, b in zip(res[0], res[1]))
    assert t_beside < 0.88 * t_turn, (t_turn, t_beside)          # 0.71 measured; 0.98 when they cannot overlap


def continuous_space():
    """14.7 M configs under a budget of eight GPUs: long stretches of these fronts are concave in the logarithms."""
    seed = 1014
    dp, tp = I.hybrid_axis(8)
    hw, mem = I.seeded_hw(seed, 20, mem_choices=[24, 48, 80, 192])
    fw_f, fw_i = I.seeded_fw(seed, 4)
    return {"models": I.seeded_models(seed, 16), "hw": hw, "hw_mem": mem, "fw_f": fw_f, "fw_i": fw_i,
            "batch": np.array([1, 2, 3, 5, 8, 16, 31, 64, 100, 256, 509, 1024], dtype=np.uint32), "tp": np.array(tp, dtype=np.uint32),
            "dp": np.array(dp, dtype=np.uint32), "pairs": np.array(I.pairs_grid(I.LEN_GRID_8, I.LEN_GRID_8), dtype=np.uint32)}


def test_fronts_of_continuous_metrics_are_not_done_twice():
    """Pairs of metrics without few distinct values: the filter must leave so few that the list holds them (word 1
    of the workspace tells the kernel behind to redo the call), over long ranges and ranges held in registers."""
    import torch
    sp = guide.Space(continuous_space())
    assert sp.size == 14_745_600
    fields = ("latency", "ttft", "tpot", "thr_decode", "cost_per_hr", "cost_per_token", "status")
    out = guide.alloc_outputs(sp.size, 0, fields)
    guide.guide_simulate(sp, None, out)
    ws = torch.empty(guide.guide_pareto_workspace_bytes(sp), dtype=torch.uint8, device="cuda")
    idx = torch.empty(guide.PARETO_MAX, dtype=torch.int64, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    for n in (sp.size, 8_000_000, 2_000_000, 1_200_000, 500_000):
        part = {k: v[:n] for k, v in out.items()}
        host = {k: v.cpu().numpy() for k, v in part.items()}
        host["ttft_p50"] = host["ttft_p99"] = host["ttft"]
        for x, y in (("ttft", "cost_per_token"), ("ttft", "throughput"), ("tpot", "cost_per_token"), ("latency", "cost_per_token"),
                     ("cost_per_hr", "throughput"), ("throughput", "cost_per_token"), ("latency", "cost_per_hr")):
            guide.guide_pareto(sp, None, part, {}, x, y, idx, cnt, ws, count=n)
            torch.cuda.synchronize()
            assert int(ws[:8].view(torch.int32)[1].item()) == 0, (n, x, y)
            want, size = oracle.pareto(host, {}, x, y, cap=guide.PARETO_MAX)
            assert int(cnt.item()) == size and np.array_equal(idx[:size].cpu().numpy().view(np.uint64), want), (n, x, y)


@pytest.mark.parametrize("n", [40_000, REGISTERS, REGISTERS + 1, 2_000_001])
def test_staircase_steps(sp, n):
    """Fronts that put every point on a step of its own, many points on one step, duplicates of x and of y, a front that
    fills the list and one that does not fit it: the refined filter against the oracle."""
    rng = np.random.default_rng(n)
    host = synth(n, 40 + n % 7, pass_frac=0.9)
    t = rng.random(n)
    for x, y in ((t, 1.0 - t + 0.3 * rng.random(n)),                       # a straight front: nothing is killed by its ends
                 (1.0 + t, 1.0 / (1.0 + t) * (1.0 + rng.random(n))),             # hyperbola
                 (np.floor(t * 3000.0), 1.0 - t + 0.1 * rng.random(n)),          # 3,000 values of x
                 (t, np.floor((1.0 - t + 0.1 * rng.random(n)) * 500.0)),         # 500 values of y
                 (np.where(t < 0.5, 1.0, 1e300 * t), np.where(t < 0.5, rng.random(n), 1e-300)),
                 (-t, t * 4.0 + 0.01 * rng.random(n))):
        host["latency"], host["cost_per_token"] = np.ascontiguousarray(x), np.ascontiguousarray(y)
        dev = to_dev(host)
        fidx, fcnt = run_pareto(sp, dev, {}, "latency", "cost_per_token", count=n)
        want, size = oracle.pareto(host, {}, "latency", "cost_per_token", cap=guide.PARETO_MAX)
        if size > guide.PARETO_MAX:
            assert fcnt == 0xFFFFFFFF, (n, size)
        else:
            assert fcnt == size and np.array_equal(fidx, want), (n, size)


def without_cooperation(value):
    """Selections of a process that cannot launch cooperatively (the library reads the variable once)."""
    import os
    import subprocess
    import sys
    code = (
        "import sys; sys.path.insert(0, 'tests')\n"
        "import numpy as np, oracle\n"
        "import test_gpu_select_coop as t\n"
        "from gpu_util import run_pareto, run_simulate_select, run_topk\n"
        "from paper_2412_04788_b200 import guide, inputs as I\n"
        "sp = guide.Space(I.workload(5, scale=0.125)['space'])\n"
        "for n, seed in ((2049, 20), (70_001, 21), (1_310_785, 22)):\n"
        "    host = t.synth(n, seed); dev = t.to_dev(host)\n"
        "    for cons, key, k in (({'max_latency': 6.0}, 'cost_per_token', 64), ({}, 'cost_per_hr', 128), ({}, 'throughput', 1)):\n"
        "        t.check(sp, host, dev, cons, key, k, n)\n"
        "w = I.workload(2, scale=0.5)\n"
        "sp2 = guide.Space(w['space'])\n"
        "want = oracle.simulate(w['space'])\n"
        "for cons in ({}, {'max_latency': 20.0}):\n"
        "    for key, k in (('cost_per_token', 64), ('cost_per_hr', 128), ('latency', 1)):\n"
        "        idx, val, cnt = run_topk(sp2, None, cons, key, k)\n"
        "        w_idx, w_val, w_cnt = oracle.select_topk(want, cons, key, k)\n"
        "        assert cnt == w_cnt and np.array_equal(idx, w_idx) and np.array_equal(val, w_val), (cons, key, k)\n"
        "    f, n = run_pareto(sp2, None, cons, 'latency', 'cost_per_hr')\n"
        "    w_f, w_n = oracle.pareto(want, cons, 'latency', 'cost_per_hr', cap=guide.PARETO_MAX)\n"
        "    assert n == w_n and np.array_equal(f, w_f)\n"
        "    _, (idx, val, cnt), (f, n), _, _ = run_simulate_select(w['space'], cons, 'cost_per_token', 64, cons, 'latency', 'cost_per_hr')\n"
        "    w_idx, _, w_cnt = oracle.select_topk(want, cons, 'cost_per_token', 64)\n"
        "    assert cnt == w_cnt and np.array_equal(idx, w_idx) and n == w_n and np.array_equal(f, w_f)\n"
        "print('selections ok')\n")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    res = subprocess.run([sys.executable, "-c", code], cwd=root, env=dict(os.environ, GUIDE_NO_COOPERATIVE=value),
                         capture_output=True, text=True, timeout=600)
    assert res.returncode == 0 and "selections ok" in res.stdout, res.stdout[-2000:] + res.stderr[-2000:]


@pytest.mark.parametrize("value", ["1", "refuse"])
def test_selections_without_cooperative_launches(value):
    """Taken to the other kernels from the start, or after CUDA has refused the launch (more blocks than fit): the
    materialised selections to the accumulator kernels, the fused top-k to its bound in two kernels."""
    without_cooperation(value)
