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


def test_fresh_threads_lose_no_memory():
    """Threads whose first CUDA call is one of this library's, each with a handle of its own: what one leaves
    behind serves the next, and nothing is lost on the way."""
    import torch
    w = I.workload(4)["space"]                           # tables of about half a megabyte
    count = 4096
    sp = guide.Space(w)
    out = guide.alloc_outputs(count)
    stream = torch.cuda.current_stream()
    guide.guide_simulate(sp, None, out, count=count)
    torch.cuda.synchronize()
    want = {k: v.clone() for k, v in out.items()}
    errors = []

    def question():
        try:
            mine = guide.Space(w)
            guide.guide_simulate(mine, None, out, count=count, stream=stream)
            mine.close()
        except Exception as e:                           # noqa: BLE001 - reported by the main thread
            errors.append(repr(e))

    def run(n):
        for _ in range(n):
            t = threading.Thread(target=question)
            t.start()
            t.join()
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]
    before = run(8)                                      # the pool has its blocks
    after = run(64)
    assert not errors, errors
    assert all(torch.equal(want[k], out[k]) for k in want)
    assert before - after < 8 << 20, f"{(before - after) >> 20} MB lost"


@pytest.mark.parametrize("mode,thread", [("relaxed", False), ("relaxed", True), ("thread_local", True)])
def test_destroyed_during_a_capture(mode, thread):
    """A handle that is destroyed while a stream is being captured (by the collector, on another thread) does not
    end the capture."""
    import torch
    w = spaces()[0]
    sp = guide.Space(w)
    out = guide.alloc_outputs(sp.size)
    guide.guide_simulate(sp, None, out)
    torch.cuda.synchronize()
    x = torch.zeros(1, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode=mode):
        x.add_(1.0)
        if thread:
            t = threading.Thread(target=sp.close)
            t.start()
            t.join()
        else:
            sp.close()
        x.add_(1.0)
    x.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert x.item() == 2.0


def test_captured_use_and_the_next_handle():
    """A graph that holds a handle's kernels may run on any stream, until the handle is destroyed: its memory is
    not handed to a handle that is used meanwhile."""
    import torch
    w = spaces()
    want = [oracle.simulate(x) for x in w[:2]]
    a = guide.Space(w[0])
    out_a = guide.alloc_outputs(a.size)
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    guide.guide_simulate(a, None, out_a, stream=side)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        guide.guide_simulate(a, None, out_a)
    for v in out_a.values():
        v.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        for _ in range(50):
            g.replay()
    a.close()
    b = guide.Space(w[1])
    out_b = guide.alloc_outputs(b.size)
    guide.guide_simulate(b, None, out_b, stream=side)
    torch.cuda.synchronize()
    for out, ref in ((out_a, want[0]), (out_b, want[1])):
        assert not any(bit_mismatches({k: v.cpu().numpy() for k, v in out.items()}, ref).values())
    b.close()
