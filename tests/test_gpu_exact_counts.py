"""The one-thread-per-config evaluation takes its stage tables from products of doubles when the host finds
every count of the space small enough, from 64-bit integers otherwise.  Spaces on both sides of the limits,
against the oracle bit for bit: binary64 and binary32, prompt splitting, eviction, clamp, both time and TP models."""
import numpy as np
import pytest

import oracle
from paper_2412_04788_b200 import guide, inputs as I
from gpu_util import bit_mismatches, run_simulate

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
    part = dict(first=1, count=n - 2)                             # a slice: the one-thread-per-config kernel whatever the axes
    for tm, tpm in ((0, 0), (1, 1)):
        for kw in ({}, {"clamp_seq": 1}):
            got, _, _, _ = run_simulate(s, None, time_model=tm, tp_model=tpm, clamp_seq=bool(kw), **part)
            want = oracle.simulate(s, time_model=tm, tp_model=tpm, **part, **kw)
            assert not any(bit_mismatches(got, want).values()), (name, tm, kw, bit_mismatches(got, want))
            assert np.array_equal(got["status"], want["status"]) and np.array_equal(got["n_req_iters"], want["n_req_iters"])
        got, _, _, _ = run_simulate(s, None, time_model=tm, tp_model=tpm, precision=guide.PREC_F32, **part)
        want = oracle.simulate(s, time_model=tm, tp_model=tpm, precision="f32", **part)
        assert not any(bit_mismatches(got, want).values()), (name, "f32", tm, bit_mismatches(got, want))
