"""Device memory of programs and contexts: what is freed in stream order waits for no
other work, and what is kept for later loads is bounded over all contexts."""
import numpy as np
import pytest

import synth
from parity import ARCH

pytestmark = pytest.mark.gpu

SLOTS = dict(search_slots=152)  # small search arenas: these tests are about the programs' memory


def dev(samples):
    import torch
    return torch.from_numpy(np.ascontiguousarray(samples).view(np.int64)).cuda()


class Busy:
    """Half a second of work on a stream of its own."""

    def __init__(self):
        import torch
        self.stream, self.done = torch.cuda.Stream(), torch.cuda.Event()
        with torch.cuda.stream(self.stream):
            torch.cuda._sleep(1_000_000_000)
            self.done.record()

    def running(self):
        return not self.done.query()


def small_program(n=4):
    P = synth.make_program(synth.batched_params(n, np.random.default_rng(n), n), 1.0)
    return P, dev(P.samples(200_000, seed=n))


@pytest.mark.parametrize("what", ["plain", "launch_stats", "export", "graph"])
def test_unload_async_waits_for_no_other_stream(what):
    """A program with launch statistics, an exported graph or a captured step is freed in
    its stream's order while another stream is busy."""
    import torch
    import paper_2009_04061_gb300 as g
    P, d = small_program()
    own = torch.cuda.Stream()
    with g.Context(ARCH, SLOTS) as c:
        prog = c.load_program(P)
        if what == "launch_stats":
            prog.set_launch_stats(synth.launch_stats(P.n_functions, 1), g.gpa_sm_model_of_device())
        if what == "graph":
            prog.capture_step(d)
            prog.launch_step(own)
        prog.reset(own)
        prog.ingest(d, stream=own)
        prog.blame(own)
        if what == "export":
            prog.unpruned_edges(own)
        own.synchronize()
        other = Busy()
        prog.unload_async(own)
        assert other.running()
        own.synchronize()
        assert other.running()
        other.stream.synchronize()


def test_memory_kept_is_bounded_over_contexts():
    """What unloaded programs gave back is kept once for all contexts of a device, not by
    each of them, is there for every context, and is given back with the last one."""
    import torch
    import paper_2009_04061_gb300 as g
    P = synth.make_program(synth.batched_params(60, np.random.default_rng(3), 3), 1.0)
    with g.Context(ARCH, SLOTS) as first:     # (what a process's first context leaves for good)
        first.load_program(P).unload()
    torch.cuda.synchronize()
    base = torch.cuda.mem_get_info()[0]
    ctxs = [g.Context(ARCH, SLOTS) for _ in range(5)]
    try:
        need = ctxs[0].footprint(P)
        assert 100 << 20 < need < 512 << 20
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        for c in ctxs:
            c.load_program(P).unload()
        torch.cuda.synchronize()
        kept = before - torch.cuda.mem_get_info()[0]
        assert kept < 2 * need, (kept, need)
    finally:
        for c in ctxs:
            c.close()
    torch.cuda.synchronize()
    assert base - torch.cuda.mem_get_info()[0] < 64 << 20
