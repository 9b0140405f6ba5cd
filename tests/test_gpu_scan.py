"""The library's own offsets where their scan takes more tiles than a CTA adds up by
itself: a program of more than a million blocks."""
import numpy as np
import pytest

import oracle
import synth
from parity import ARCH, assert_edges_equal

pytestmark = pytest.mark.gpu


def chains(n_functions, blocks):
    """Functions of `blocks` one-instruction blocks in a row; instruction k writes R(k mod
    97) and reads R((k - 2) mod 97), which the block before the last one wrote."""
    n = n_functions * blocks
    k = np.arange(n) % blocks
    last = k == blocks - 1
    i32 = np.int32
    return dict(
        n_functions=n_functions, n_instr=n, n_blocks=n, n_loops=0, n_lines=1,
        func_instr_off=np.arange(0, n + 1, blocks, dtype=i32), func_block_off=np.arange(0, n + 1, blocks, dtype=i32),
        func_loop_off=np.zeros(n_functions + 1, i32), block_instr_off=np.arange(n + 1, dtype=i32),
        succ_off=np.concatenate([[0], np.cumsum(~last)]).astype(i32), succ=(np.arange(n)[~last] + 1).astype(i32),
        opclass=np.full(n, synth.OP["IMAD"], np.uint8), guard=np.zeros(n, np.uint8), iflags=np.zeros(n, np.uint8),
        line=np.zeros(n, i32), def_off=np.arange(n + 1, dtype=i32), def_res=(k % 97).astype(np.uint16),
        use_off=np.arange(n + 1, dtype=i32), use_res=((k - 2) % 97).astype(np.uint16),
        block_loop=np.full(n, -1, i32), loop_parent=np.zeros(0, i32), loop_header=np.zeros(0, i32))


def test_offsets_of_a_million_blocks():
    """1,100,000 blocks: 17.6M event segments in 4,297 tiles."""
    import torch
    import paper_2009_04061_gb300 as g
    nf, nb = 1100, 1000
    P = chains(nf, nb)
    fs = [0, 1, nf // 2, nf - 2, nf - 1]
    s = np.array([(f << 48) | (pc << 24) | (2 << 20) | (1 << 19) for f in fs for pc in range(nb) for _ in range(1 + pc % 3)],
                 dtype=np.uint64)
    with g.Context(ARCH, dict(search_slots=152)) as c:
        prog = c.load_program(P)
        try:
            prog.reset()
            prog.ingest(torch.from_numpy(s.view(np.int64)).cuda())
            prog.blame()
            assert prog.status()[0] == 0
            cnt, bad = prog.counts()
            edges, blame = prog.edges(), prog.blame_counts()
        finally:
            prog.unload()
    assert bad == 0 and int(cnt.sum()) == s.size
    assert np.array_equal(blame.sum(0), cnt.sum(0))
    uses = np.concatenate([f * nb + np.arange(nb) for f in fs])
    want = oracle.edges_of_uses(P, ARCH, cnt, uses)
    assert len(want["j"]) > len(fs) * (nb - 10)
    assert_edges_equal(edges, want)
