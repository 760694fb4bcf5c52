"""Device memory of handles is kept for the next handle: results must not depend on what a block held
before, on which thread or stream used it, or on the order of creation and destruction."""
import threading

import numpy as np
import pytest

import oracle
from paper_2412_04788_b200 import guide, inputs as I
from gpu_util import bit_mismatches, run_simulate

pytestmark = pytest.mark.gpu


def spaces():
    return [I.workload(1)["space"], I.workload(2, scale=0.0625)["space"], I.workload(4, scale=1 / 256)["space"]]


def test_handles_made_and_destroyed_in_turn():
    """More live handles than blocks are kept, destroyed in another order, then made again."""
    want = [oracle.simulate(w) for w in spaces()]
    for order in ((0, 1, 2, 0, 1, 2, 0), (2, 1, 0)):
        live = []
        for i in order:
            got, _, sp, _ = run_simulate(spaces()[i])
            assert not any(bit_mismatches(got, want[i]).values()) and np.array_equal(got["status"], want[i]["status"])
            live.append(sp)
        for sp in live[::2] + live[1::2]:
            sp.close()


def test_handles_on_several_threads_and_streams():
    import torch
    w = spaces()
    want = [oracle.simulate(x) for x in w]
    errors = []

    def work(i):
        try:
            stream = torch.cuda.Stream()
            for rep in range(8):
                j = (i + rep) % len(w)
                sp = guide.Space(w[j])
                out = guide.alloc_outputs(sp.size)
                torch.cuda.current_stream().synchronize()
                guide.guide_simulate(sp, None, out, stream=stream)
                if rep % 2:
                    stream.synchronize()
                sp.close()                               # with the sweep perhaps still running
                stream.synchronize()
                got = {k: v.cpu().numpy() for k, v in out.items()}
                assert not any(bit_mismatches(got, want[j]).values())
        except Exception as e:                           # noqa: BLE001 - reported by the main thread
            errors.append(repr(e))
    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
