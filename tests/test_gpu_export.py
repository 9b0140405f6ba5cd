"""The order of the exported dependency graph where a use has many sources."""
import numpy as np
import pytest

import oracle
import synth
from progbuild import I, program

pytestmark = pytest.mark.gpu


def guarded(defs_1, defs_2, uses):
    """A block of guarded definitions of R1 and R2, in turn, none of which covers the
    readers of both behind them; samples of memory stalls at the readers."""
    body = [I("ISETP", ["P0"], ["R9"]), I("ISETP", ["P1"], ["R9"])]
    ks = sorted([(k / defs_1, "R1") for k in range(defs_1)] + [(k / max(defs_2, 1), "R2") for k in range(defs_2)])
    body += [I("LDG", [r], [], guard="P0") for _, r in ks]
    body += [I("IADD", ["R4"], ["R2", "R1"], guard="P1") for _ in range(uses)]
    first = 2 + len(ks)
    P = program([([body + [I("EXIT")]], [[]], [])])
    s = np.array([((first + k) << 24) | (3 << 20) for k in range(uses)], dtype=np.uint64)
    return P, s, first


@pytest.mark.parametrize("defs_1,defs_2,uses", [(1023, 0, 3), (1024, 0, 3), (1025, 0, 3), (700, 700, 40), (2049, 1, 2),
                                               (20000, 12000, 60)])
def test_uses_with_many_sources_are_ordered(defs_1, defs_2, uses):
    """Buckets around the line between comparing and sorting, and far beyond it; a
    resource's sources stay together and ascend."""
    import time
    import torch
    import paper_2009_04061_gb300 as g
    P, s, first = guarded(defs_1, defs_2, uses)
    with g.Context(synth.default_arch(), dict(search_slots=152)) as c:
        prog = c.load_program(P)
        try:
            prog.reset()
            prog.ingest(torch.from_numpy(s.view(np.int64)).cuda())
            prog.unpruned_edges()
            t0 = time.perf_counter()
            x = prog.unpruned_edges()
            print(f"{defs_1}+{defs_2} sources, {uses} uses: {1e3 * (time.perf_counter() - t0):.1f} ms")
            assert prog.status()[0] == 0
        finally:
            prog.unload()
    use, res, d = (x[k].astype(np.int64) for k in ("use", "res", "def"))
    assert use.size == uses * (defs_1 + defs_2 + 1)           # and the guard predicate's definition
    assert np.all(np.diff((use * 512 + res) * (1 << 20) + d) > 0)
    # straight code without unguarded readers: every source at its own distance, none cut
    assert np.array_equal(x["dmin"], use - d) and np.array_equal(x["dlong"], use - d)
    assert not x["K"].any() and not x["dom"].any()
    if defs_1 + defs_2 < 4096:
        for j in (first, first + uses - 1):
            want = [(r, q["i"], q["dmin"], q["K"], q["dlong"], int(q["dom"])) for r in (1, 2, synth.P_BASE + 1)
                    for q in oracle.search(P, j, r)]
            m = use == j
            assert list(zip(*(x[k][m].tolist() for k in ("res", "def", "dmin", "K", "dlong", "dom")))) == sorted(want)
