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


def by_cta(kind):
    """One search of a CTA whose source S the reader W cuts on the shortest path:
      blocks: nothing else leads from S to the use;
      layers: neither does a back edge, but a long block N beside W does;
      whole:  a path through the loop's back edge does, longer than any latency.
    Off S's paths or on them, a chain of 40 blocks makes the graph too large for the
    smaller tiers."""
    chain = 40
    r1 = ["R1"]
    blocks = [[I("MOV", ["R2"], ["R3"])],                                      # 0 entry
              [I("MOV", ["R5"], ["R3"]) for _ in range(12)],                   # 1 loop header
              [I("IADD", r1, ["R3"])],                                         # 2 S
              [I("IADD", ["R6"], r1)],                                         # 3 W
              [I("MOV", ["R7"], ["R3"]) for _ in range(30)],                   # 4 N
              [I("MOV", ["R8"], ["R3"])]]                                      # 5 B, around S
    J, Y = 6, 7
    L = Y + chain
    blocks.append([I("IADD", ["R9"], r1)])                                     # J, the use
    blocks += [[I("MOV", ["R10"], ["R3"])] for _ in range(chain)]              # Y ...
    blocks += [[I("MOV", ["R11"], ["R3"])], [I("EXIT")]]                       # L, exit
    succ = [[1], [2, 4, 5], [3], [J], [J], [J], [L]] + [[k + 1] for k in range(Y, L)] + [[1, L + 1], []]
    if kind == "layers":
        succ[1], succ[2] = [2, 5], [3, 4]
    succ[2 if kind == "whole" else 1].append(Y)
    P = program([(blocks, succ, [(1, list(range(1, L + 1)), -1)])])
    use = sum(len(b) for b in blocks[:J])
    s = np.array([(use << 24) | (2 << 20) | (1 << 19)] * 7 + [((use - 1) << 24)], dtype=np.uint64)
    return P, s, use


@pytest.mark.parametrize("kind,edges,nodes", [("blocks", 0, (1, 16)), ("layers", 1, (1, 16)), ("whole", 1, (40, 60))])
def test_what_decides_a_search_of_a_cta(kind, edges, nodes):
    """Rule 2 on the function's blocks, on the layers of back edges that the sources need,
    and on the whole graph. On later steps only the CTA meets the search, so the nodes
    tell how far its graph grew."""
    import paper_2009_04061_gb300 as g
    P, s, use = by_cta(kind)
    with g.Context(ARCH, SMALL) as c:
        out, last = steps(c, P, s, 3)
    assert_full_parity(last, oracle_run(P, s))
    assert len(last["edges"]["j"]) == edges
    assert out[0][0]["max_nodes"] >= 16
    for info, _ in out[1:]:
        assert nodes[0] <= info["max_nodes"] <= nodes[1], info
        assert info["tier3_searches"] == 1 == info["general_searches"]


def test_largest_searches_on_later_steps():
    """Searches beyond 2^18 nodes, handed on by every tier before and queued straight for
    their CTAs: the same edges, blame and counts."""
    import paper_2009_04061_gb300 as g
    P = synth.make_program([dict(n_instr=120_000, n_loops=24, max_depth=4, n_regs=255, ldg_pct=30, zipf_s=1.1,
                                 seed=1_000_003)], 1.0)
    s = P.samples(2_000_000, seed=5)
    with g.Context(ARCH) as c:
        out, _ = steps(c, P, s, 3)
    assert out[0][0]["max_nodes"] > 1 << 18
    n = [(info["tier3_searches"], info["general_searches"]) for info, _ in out]
    assert n[0][0] == n[1][0] == n[2][0], n
    for _, e in out[1:]:
        assert_edges_equal(e, out[0][1])


@pytest.mark.parametrize("nb", [2000, 4000])
def test_reaching_definitions_of_a_large_function_with_other_loops(nb):
    """Loops whose bodies are not natural ones (a listed block that leads to no latch), on both
    sides of the staged fixpoint's limit: the larger function takes the windowed kernel."""
    import oracle
    import paper_2009_04061_gb300 as g
    rng = np.random.default_rng(nb)
    regs = [f"R{k}" for k in range(60)]
    blocks = [[I("IADD", [regs[rng.integers(60)]], [regs[rng.integers(60)]])] for _ in range(nb - 1)] + [[I("EXIT")]]
    succ = [[k + 1] for k in range(nb - 1)] + [[]]
    loops = [(10, list(range(10, nb // 2 + 1)) + [nb - 5], -1), (nb // 4, list(range(nb // 4, nb // 3 + 1)), 0)]
    for h, body, _ in loops:
        succ[max(b for b in body if b < nb - 5)].append(h)
    for k in rng.choice(nb - 100, 200, replace=False):
        succ[k].append(int(k + rng.integers(2, 90)))
    P = program([(blocks, [sorted(set(x)) for x in succ], loops)])
    with g.Context(ARCH, dict(search_slots=16)) as c:
        prog = c.load_program(P)
        prog.reset()
        prog.blame()
        rin, rout = prog.reaching()
        st, info = prog.status()
        prog.unload()
    orin, orout = oracle.reaching(P)
    assert st == 0 and info["sweeps"] > 1
    assert np.array_equal(rin, orin) and np.array_equal(rout, orout)
