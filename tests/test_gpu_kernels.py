"""Kernels and dispatch rules at the sizes where they can go wrong: tile edges
and remainders of the scan and the aggregation, the arena sizes of the search
tiers, the fixpoint's largest staged functions and those beyond, advice tiles,
the export's buffer, and the load's validation. Everything is integers and
compared exactly; FP64 speedups within the suite's 1e-12."""
import numpy as np
import pytest

import oracle
import synth
from parity import ARCH, assert_edges_equal, assert_full_parity, gpu_run, oracle_run
from progbuild import I, program

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2009_04061_gb300 as g
    c = g.Context(ARCH)
    yield c
    c.close()


def dev(samples):
    import torch
    return torch.from_numpy(np.ascontiguousarray(samples).view(np.int64)).cuda()


@pytest.mark.parametrize("n", [1, 7, 4095, 4096, 4097, 8193, 3 * 4096 + 17, 1 << 24])
@pytest.mark.parametrize("offset", [0, 1, 4])
def test_scan_tiles_and_alignment(n, offset):
    """One tile, its edges, several, the largest size; 16-byte aligned buffers and not."""
    import torch
    import paper_2009_04061_gb300 as g
    x = np.random.default_rng(n + offset).integers(-3, 9, n).astype(np.int32)
    buf = torch.full((n + offset + 1,), 77, dtype=torch.int32, device="cuda")
    buf[offset:offset + n] = torch.from_numpy(x).cuda()
    total = torch.zeros(1, dtype=torch.int32, device="cuda")
    g.gpa_exclusive_scan_noalloc(buf[offset:offset + n], total)
    c = np.cumsum(x.astype(np.int64))
    got = buf.cpu().numpy()
    assert np.array_equal(got[offset:offset + n], np.concatenate([[0], c[:-1]]).astype(np.int32))
    assert np.all(got[:offset] == 77) and got[-1] == 77
    assert int(total.item()) == int(c[-1])


@pytest.mark.parametrize("order", ["launch", "interleaved"])
@pytest.mark.parametrize("n", [1, 2, 8191, 8192, 8193, 12 * 8192 + 5, 1000 * 8192 + 3])
def test_aggregation_chunks(ctx, n, order):
    """Streams of less than a tile up to more than one tile a chunk, runs and kernels
    interleaved, a start on and off a 16-byte boundary."""
    P = synth.make_program(synth.batched_params(30, np.random.default_rng(4), 4), 1.0)
    s = P.samples(n + 1, seed=n, order=order, invalid_ppm=1000)
    prog = ctx.load_program(P)
    try:
        d = dev(s)
        for skip in (0, 1):
            prog.reset()
            prog.ingest(d[skip:skip + n])
            cnt, bad = prog.counts()
            want, wbad = oracle.histogram(P, s[skip:skip + n])
            assert bad == wbad and np.array_equal(cnt, want)
    finally:
        prog.unload()


@pytest.mark.parametrize("small,mid,most", [(2, 2, 4), (16, 16, 100), (16, 64, 320), (32, 128, 641), (64, 64, 2560),
                                            (1024, 1024, 0)])
def test_search_arena_sizes(small, mid, most):
    """Arena sizes of the lanes (2 to 128 nodes) and of the shared-memory warps (bounded
    by max_search_nodes, powers of two or not): every size hands on to the next tier, on a
    first step and on steps that know the searches' sizes."""
    import paper_2009_04061_gb300 as g
    P = synth.make_program(synth.batched_params(12, np.random.default_rng(61), 61), 1.0)
    s = P.samples(700_000, seed=61)
    R = oracle_run(P, s)
    with g.Context(ARCH, dict(small_search_nodes=small, mid_search_nodes=mid, max_search_nodes=most,
                              search_slots=64)) as c:
        assert_full_parity(gpu_run(c, P, dev(s)), R)
        prog = c.load_program(P)
        try:
            d = dev(s)
            for _ in range(4):
                prog.reset()
                prog.ingest(d)
                prog.blame()
            st, _ = prog.status()
            assert st == 0
            assert_edges_equal(prog.edges(), R["edges"])
        finally:
            prog.unload()


@pytest.mark.parametrize("seed", [71, 72, 73])
def test_searches_of_a_cta(seed):
    """Every search of more than 16 nodes by a CTA: sources cut on the function's blocks,
    the layers of back edges that the others need, and the whole graph where those do
    not decide; several back edges and guarded defs."""
    import paper_2009_04061_gb300 as g
    rng = np.random.default_rng(seed)
    P = synth.make_program(synth.batched_params(16, rng, seed), 1.0)
    s = P.samples(900_000, seed=seed)
    with g.Context(ARCH, dict(small_search_nodes=4, mid_search_nodes=8, max_search_nodes=16, search_slots=16)) as c:
        assert_full_parity(gpu_run(c, P, dev(s)), oracle_run(P, s))


def test_one_search_slot():
    """A context with a single global-memory arena: the CTAs and the warps take turns with it."""
    import paper_2009_04061_gb300 as g
    P = synth.make_program(synth.batched_params(6, np.random.default_rng(62), 62), 1.0)
    s = P.samples(300_000, seed=62)
    with g.Context(ARCH, dict(small_search_nodes=4, mid_search_nodes=8, max_search_nodes=16, search_slots=1)) as c:
        assert_full_parity(gpu_run(c, P, dev(s)), oracle_run(P, s))


@pytest.mark.parametrize("n_instr", [20_000, 30_011])
def test_large_kernel_steps_agree(ctx, n_instr):
    """Searches of hundreds to tens of thousands of nodes: the first step (every search
    from the smallest tier up) and later ones (each in the tier of its size) give the same
    edges and blame, and a sample of uses equals the oracle's."""
    P = synth.make_program([dict(n_instr=n_instr, n_loops=n_instr // 5000, max_depth=4, n_regs=255, ldg_pct=30,
                                 zipf_s=1.1, seed=1_000_003)], 1.0)
    s = P.samples(2_000_000, seed=5)
    prog = ctx.load_program(P)
    try:
        d = dev(s)
        runs = []
        for _ in range(4):
            prog.reset()
            prog.ingest(d)
            prog.blame()
            st, info = prog.status()
            assert st == 0 and info["max_nodes"] > 5632
            runs.append((prog.edges(), prog.blame_counts()))
        cnt, _ = prog.counts()
        rin, rout = prog.reaching()
    finally:
        prog.unload()
    for e, b in runs[1:]:
        assert_edges_equal(e, runs[0][0])
        assert np.array_equal(b, runs[0][1])
    orin, orout = oracle.reaching(P)
    assert np.array_equal(rin, orin) and np.array_equal(rout, orout)
    e = runs[0][0]
    few = np.flatnonzero(cnt[:, [2, 3, 5, 6]].sum((1, 2)) > 0)
    pick = np.sort(np.random.default_rng(1).choice(few, 40, replace=False))
    keep = np.isin(e["j"], pick)
    assert_edges_equal({k: v[keep] for k, v in e.items()}, oracle.edges_of_uses(P, ARCH, cnt, pick))


@pytest.mark.parametrize("n_loops", [0, 3])
@pytest.mark.parametrize("n_instr", [18_000, 21_500, 23_000, 40_000])
def test_reaching_definitions_around_the_stage_limit(ctx, n_instr, n_loops):
    """Functions on both sides of the staged fixpoint's shared memory (with and without
    loops: the seeded sweep and its rows of zeros), beside small ones."""
    ps = [dict(n_instr=n, n_loops=n_loops, max_depth=3, n_regs=200, seed=n) for n in (60, 700, n_instr)]
    P = synth.make_program(ps, 1.0)
    prog = ctx.load_program(P)
    try:
        prog.reset()
        prog.blame()
        rin, rout = prog.reaching()
        st, _ = prog.status()
    finally:
        prog.unload()
    orin, orout = oracle.reaching(P)
    assert st == 0 and np.array_equal(rin, orin) and np.array_equal(rout, orout)


def test_advice_tile_edges(ctx):
    """Functions of one instruction around the tiles' edges (256 instructions), with equal
    sample counts everywhere, so that hotspots are ties broken by position across tiles."""
    funcs = []
    for n in (2, 31, 32, 33, 255, 256, 257, 511, 513, 1500):
        ins = [I("LDG", ["R1"], ["R2", "R3"], line=k, flags=1) for k in range(n - 1)] + [I("EXIT", line=n)]
        funcs.append(([ins], [[]], []))
    prog = program(funcs)
    ss = []
    for f, (blocks, _, _) in enumerate(funcs):
        for pc in range(len(blocks[0])):
            ss += [(f << 48) | (pc << 24) | (c << 20) | (lat << 19) for c in (0, 1, 3, 5, 8) for lat in ((0, 1) if c else (0,))]
    s = np.array(ss, dtype=np.uint64)
    assert_full_parity(gpu_run(ctx, prog, dev(s)), oracle_run(prog, s))


def test_advice_same_with_both_tile_sizes(ctx):
    """The same functions in a program of few tiles (256 instructions each) and in one
    large enough for tiles of 1,024 have the same advice."""
    ps = synth.batched_params(20, np.random.default_rng(71), 71)
    small = synth.make_program(ps, 1.0)
    many = synth.make_program(ps + [dict(p, seed=p["seed"] + 5) for p in ps * 8], 1.0)
    assert small.n_instr < 1024 * 100 < 1024 * 152 < many.n_instr
    s = small.samples(800_000, seed=71)
    got = []
    for P in (small, many):
        prog = ctx.load_program(P)
        try:
            prog.reset()
            prog.ingest(dev(s))
            prog.blame()
            got.append(prog.advise())
        finally:
            prog.unload()
    for k in ("totals", "matched", "speedup", "rank", "n_hot", "hot"):
        assert np.array_equal(got[0][k], got[1][k][:20], equal_nan=True), k


def test_export_larger_than_its_first_buffer(ctx):
    """40 guarded readers of 40 guarded definitions: 1,600 edges of 160-odd use entries
    outgrow the buffer the export starts with; a second export uses it again."""
    import test_oracle as T
    body = [I("ISETP", ["P0"], ["R9"]), I("ISETP", ["P1"], ["R9"])]
    body += [I("LDG", ["R1"], [], guard="P0") for _ in range(40)]
    body += [I("IADD", ["R4"], ["R1"], guard="P1") for _ in range(40)]
    P = T.one_block(body)
    first = 2 + 40
    s = np.array([((first + k) << 24) | (3 << 20) for k in range(40) for _ in range(3)], dtype=np.uint64)
    prog = ctx.load_program(P)
    try:
        prog.reset()
        prog.ingest(dev(s))
        for _ in range(2):
            x = prog.unpruned_edges()
            key = list(zip(x["use"].tolist(), x["res"].tolist(), x["def"].tolist()))
            assert key == sorted(key)
            want = [(j, r, q["i"], q["dmin"], q["K"], q["dlong"], int(q["dom"]))
                    for j in range(first, first + 40) for r in (1, 256) for q in oracle.search(P, j, r)]
            got = list(zip(*(x[k].tolist() for k in ("use", "res", "def", "dmin", "K", "dlong", "dom"))))
            assert got == sorted(want) and len(got) > int(np.asarray(P["use_res"]).size)
            assert prog.status()[0] == 0
    finally:
        prog.unload()


@pytest.mark.parametrize("length", [2, 3, 5, 15, 16, 17, 40])
@pytest.mark.parametrize("side", ["def", "use"])
def test_lists_that_repeat_a_resource_are_refused(ctx, length, side):
    """An operand list that names a resource twice, at either end or both, is refused; the
    same resource in neighbouring lists is not."""
    import test_oracle as T
    import paper_2009_04061_gb300 as g
    regs = [f"R{k}" for k in range(length)]

    def with_list(names):
        ins = dict(defs=names, uses=["R99"]) if side == "def" else dict(defs=["R99"], uses=names)
        plain = [I("MOV", [regs[-1]], [regs[0]]), I("MOV", [regs[0]], [regs[-1]])]
        return T.one_block([plain[0], I("IADD", **ins), plain[1], I("IADD", **ins)])

    assert ctx.footprint(with_list(regs)) > 0
    for bad in ([regs[0]] + regs[:-1], regs[:-1] + [regs[0]], regs[:-1] + [regs[-2]]):
        with pytest.raises(g.GpaError) as e:
            ctx.footprint(with_list(bad))
        assert e.value.status == -2


def test_reloads_reuse_memory_without_leftovers():
    """Programs loaded and unloaded in turn take their memory from what the context kept:
    each starts from zero counters and gives its own results."""
    import paper_2009_04061_gb300 as g
    progs = [synth.make_program(synth.batched_params(n, np.random.default_rng(n), n), 1.0) for n in (3, 9, 4)]
    with g.Context(ARCH) as c:
        for k in range(6):
            P = progs[k % 3]
            s = P.samples(50_000, seed=k)
            prog = c.load_program(P)
            assert not prog.counts()[0].any()
            prog.ingest(dev(s))
            prog.blame()
            R = oracle_run(P, s)
            assert_edges_equal(prog.edges(), R["edges"])
            assert np.array_equal(prog.blame_counts(), R["blame"])
            prog.unload_async() if k % 2 else prog.unload()
