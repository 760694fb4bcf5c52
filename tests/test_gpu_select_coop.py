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

REGISTERS = 148 * 2 * 16 * 4 * 64        # configs a full grid's registers hold: beyond it one row out of every r is sampled


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


def test_candidate_list_overflow_runs_the_filter_again(sp):
    """Passing configs only in the rows the sample leaves out (one row of every two is sampled at this
    size, at a hashed place): no bound, the survivor list overflows, and the filter repeats with a closer
    bound of what it holds until the survivors fit.  Keys fall, rise and are all equal."""
    n = 2_000_001
    assert REGISTERS < n < 2 * REGISTERS
    slot = np.arange(n // 64 // 2, dtype=np.uint64)
    sampled = slot * 2 + ((slot * 2654435761) % 2**32 >> 7) % 2
    unsampled = np.setdiff1d(np.arange(n // 64), sampled)
    host = synth(n, 9)
    host["status"][:] = 2
    host["status"][(unsampled[:, None] * 64 + np.arange(64)).ravel()] = 0
    for keys in (np.arange(n, dtype=np.float64), -np.arange(n, dtype=np.float64), np.ones(n)):
        host["cost_per_token"] = keys
        dev = to_dev(host)
        for k in (1, 128):
            idx, val, cnt = run_topk(sp, dev, {}, "cost_per_token", k, count=n)
            w_idx, w_val, w_cnt = oracle.select_topk(host, {}, "cost_per_token", k)
            assert cnt == w_cnt and np.array_equal(idx, w_idx) and np.array_equal(val, w_val)
