"""The closed form takes its stage tables from products of doubles when the host finds every count of the space small
enough, from 64-bit integers otherwise.  Spaces on both sides of the limits, against the oracle bit for bit: the
one-thread-per-config kernels (binary64 and binary32, prompt splitting, eviction, clamp, both time and TP models), the
tiled kernel, the whole-space kernels by foursomes and by lines, and the fused selections' model walk."""
import numpy as np
import pytest

import oracle
from paper_2412_04788_b200 import guide, inputs as I
from gpu_util import bit_mismatches, run_pareto, run_simulate, run_topk

pytestmark = pytest.mark.gpu


def space(batch, lengths, chunk):
    w = I.workload(2, scale=0.0625)["space"]
    s = {k: np.array(v, copy=True) for k, v in w.items() if isinstance(v, np.ndarray)}
    s["batch"] = np.array(batch, dtype=np.uint32)
    s["pairs"] = np.array([(a, b) for a in lengths for b in lengths], dtype=np.uint32)
    s["hw_mem"] = np.full_like(s["hw_mem"], 10 ** 15)            # everything fits: every config is evaluated
    n_f = len(s["fw_f"])
    if chunk:
        s["fw_chunk"] = np.array([[0, 0], [3, 100], [0, 4096], [7, 0]][:n_f], dtype=np.uint32)
        s["fw_keep"] = np.array([1000, 700, 1000, 350][:n_f], dtype=np.uint32)
    return s


CASES = [("small", [1, 5, 64], [1, 33, 700]),                     # every count exact
         ("large", [1, 509, 512], [100, 8192]),                   # FLOP counts near 2^52: byte sums exact
         ("huge", [3, 4096], [1000, 100000]),                     # byte sums beyond 2^52: integer tables
         ("one token", [1, 2], [1])]


@pytest.mark.parametrize("name,batch,lengths", CASES)
@pytest.mark.parametrize("chunk", [False, True])
def test_both_sides_of_the_limits(name, batch, lengths, chunk):
    s = space(batch, lengths, chunk=chunk)
    n = int(len(s["models"]) * len(s["hw"]) * len(s["fw_f"]) * len(s["batch"]) * len(s["tp"]) * len(s["pairs"]))
    # a slice of less than half: the one-thread-per-config kernel; of more: the tiled one where the axes suit it
    for part in (dict(first=n // 5 | 1, count=n // 3), dict(first=1, count=n - 2)):
        for tm, tpm in ((0, 0), (1, 1)):
            for kw in ({}, {"clamp_seq": 1}):
                got, _, _, _ = run_simulate(s, None, time_model=tm, tp_model=tpm, clamp_seq=bool(kw), **part)
                want = oracle.simulate(s, time_model=tm, tp_model=tpm, **part, **kw)
                assert not any(bit_mismatches(got, want).values()), (name, tm, kw, bit_mismatches(got, want))
                assert np.array_equal(got["status"], want["status"]) and np.array_equal(got["n_req_iters"], want["n_req_iters"])
            got, _, _, _ = run_simulate(s, None, time_model=tm, tp_model=tpm, precision=guide.PREC_F32, **part)
            want = oracle.simulate(s, time_model=tm, tp_model=tpm, precision="f32", **part)
            assert not any(bit_mismatches(got, want).values()), (name, "f32", tm, bit_mismatches(got, want))


LENGTHS_6, LENGTHS_8 = [1, 33, 100, 512, 700, 4096], [1, 16, 33, 100, 512, 700, 4096, 8192]
BELOW, BEYOND = list(range(1, 41)), list(range(1, 40)) + [4096]
WHOLE = [("foursomes, below", BELOW, LENGTHS_6), ("foursomes, beyond", BEYOND, LENGTHS_6[:5] + [100000]),
         ("lines, below", BELOW, LENGTHS_8), ("lines, beyond", BEYOND, LENGTHS_8[:7] + [100000])]


@pytest.mark.parametrize("name,batch,lengths", WHOLE)
@pytest.mark.parametrize("tm,tpm", [(0, 0), (1, 1)])
def test_whole_space_kernels_on_both_sides(name, batch, lengths, tm, tpm):
    """36 length pairs per (batch, TP) point: the foursome walk; 64: the line walk, and enough configs for the fused
    selections over the model walk.  With a batch of 4,096 and lengths of 100,000 the byte sums pass 2^52."""
    s = space(batch, lengths, chunk=False)
    s["hw"], s["hw_mem"] = np.concatenate([s["hw"]] * 2), np.array([10 ** 15, 6 * 10 ** 11], dtype=np.uint64)
    n = len(s["models"]) * len(s["hw"]) * len(s["fw_f"]) * len(s["batch"]) * len(s["tp"]) * len(s["pairs"])
    assert n >= (1 << 18 if "lines" in name else 1 << 16)
    got, _, sp, _ = run_simulate(s, None, time_model=tm, tp_model=tpm)
    want = oracle.simulate(s, time_model=tm, tp_model=tpm)
    assert not any(bit_mismatches(got, want).values()), (name, bit_mismatches(got, want))
    for f in ("status", "bmax", "n_iters", "n_req_iters"):
        assert np.array_equal(got[f], want[f]), f
    if "lines" not in name:
        return
    for key, k in (("cost_per_token", 64), ("latency", 8)):
        idx, val, cnt = run_topk(sp, None, {}, key, k, time_model=tm, tp_model=tpm)
        w_idx, w_val, w_cnt = oracle.select_topk(want, {}, key, k)
        assert cnt == w_cnt and np.array_equal(idx, w_idx) and np.array_equal(val.view(np.uint64), w_val.view(np.uint64))
    fidx, fcnt = run_pareto(sp, None, {}, "ttft", "cost_per_token", time_model=tm, tp_model=tpm)
    w_f, w_n = oracle.pareto(want, {}, "ttft", "cost_per_token", cap=guide.PARETO_MAX)
    assert fcnt == w_n and np.array_equal(fidx, w_f)
