"""Which tier a search runs in, and what the tiers decide, from small programs made for
each case and from one large kernel: results against the oracle, sizes and counts from
the status."""
import numpy as np
import pytest

import synth
from parity import ARCH, assert_edges_equal, assert_full_parity, oracle_run
from progbuild import I, program

pytestmark = pytest.mark.gpu

# lanes of 4 and 8 nodes, warps and CTAs of 16: larger searches run in the program's own tier
SMALL = dict(small_search_nodes=4, mid_search_nodes=8, max_search_nodes=16, search_slots=16)


def dev(samples):
    import torch
    return torch.from_numpy(np.ascontiguousarray(samples).view(np.int64)).cuda()


def steps(ctx, P, s, n):
    """n steps of one program: (info, edges) of each, and the last one's results."""
    prog = ctx.load_program(P)
    try:
        d = dev(s)
        out = []
        for _ in range(n):
            prog.reset()
            prog.ingest(d)
            prog.blame()
            adv = prog.advise()
            st, info = prog.status()
            assert st == 0, info
            out.append((info, prog.edges()))
        cnt, bad = prog.counts()
        rin, rout = prog.reaching()
        last = dict(status=st, info=info, counts=cnt, invalid=bad, rin=rin, rout=rout, blame=prog.blame_counts(),
                    edges=prog.edges(), advice=adv)
        return out, last
    finally:
        prog.unload()


def test_larger_searches_are_counted_on_every_step():
    """Searches queued straight for the largest tiers on later steps count as they did
    when smaller tiers handed them on."""
    import paper_2009_04061_gb300 as g
    P = synth.make_program(synth.batched_params(12, np.random.default_rng(12), 12), 1.0)
    s = P.samples(600_000, seed=12)
    with g.Context(ARCH, SMALL) as c:
        out, last = steps(c, P, s, 3)
    assert_full_parity(last, oracle_run(P, s))
    n = [info["tier3_searches"] for info, _ in out]
    assert out[0][0]["max_nodes"] > 16 and n[0] > 0
    assert n == n[:1] * 3, n


def test_first_step_of_a_large_kernel():
    """On a first step no search's size is known: the thousands that fill the
    shared-memory warps' lists go to CTAs, and the step takes at most three times as long
    as one that knows them (two is what it measures, four with those searches a warp each).
    Both give the same edges."""
    import torch
    import paper_2009_04061_gb300 as g
    P = synth.make_program([dict(n_instr=30_000, n_loops=6, max_depth=4, n_regs=255, ldg_pct=30, zipf_s=1.1,
                                 seed=1_000_003)], 1.0)
    d = dev(P.samples(2_000_000, seed=5))
    times, edges = [], []
    with g.Context(ARCH) as c:
        for _ in range(3):
            prog = c.load_program(P)
            for k in range(3):
                prog.reset()
                prog.ingest(d)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                a.record()
                prog.blame()
                b.record()
                torch.cuda.synchronize()
                times.append(a.elapsed_time(b))
                if len(times) <= 3:
                    edges.append(prog.edges())
            assert prog.status()[0] == 0
            prog.unload()
    for e in edges[1:]:
        assert_edges_equal(e, edges[0])
    first, second, later = (min(times[k::3]) for k in range(3))
    print(f"first {first:.2f} ms, second {second:.2f}, third {later:.2f}")
    assert first < 3 * later and second < 1.5 * later
