"""The work that users have this library do, as cases that can be timed and compared.

Every case goes through the package's public entry points, on programs and
samples from the seeded generator (synth/), whose workloads this module keeps
to: the plain kernel, Rodinia-shaped programs, batches of many functions, one
very large kernel, and serving sessions. Function sizes are spread evenly over
the logarithm of a workload's range. A case names its functions; the seed gives
their order, the calls among them, the kernels' shares and the samples, so that
results of one case have one shape whatever the seed.
"""
import math

import numpy as np
import torch

import paper_2009_04061_gb300 as gpa
import synth

# Instruction counts per function of each program family (synth.workload).
_RANGES = {"rodinia": (100, 2000), "batched": (50, 20000), "large": (20000, 200000)}


def listed():
    return [
        # One small kernel analysed on its own: latency and launches count.
        dict(name="step_plain", kind="step", family="plain", functions=1, samples=100_000, graph=False,
             launch_stats=False),
        # An application of twenty kernels, profiled again and again: the captured step.
        dict(name="step_rodinia", kind="step", family="rodinia", functions=20, samples=10_000_000, graph=True,
             launch_stats=True),
        # A fleet-sized batch (the flagship workload's shape at half its functions), captured.
        dict(name="step_batched", kind="step", family="batched", functions=1000, samples=120_000_000, graph=True,
             launch_stats=True),
        # One very large kernel, loop nests and many global loads.
        dict(name="step_large", kind="step", family="large", functions=1, instructions=120_000, samples=20_000_000,
             graph=False, launch_stats=False),
        # Serving: a program nobody has seen, from host arrays to advice and out again.
        dict(name="session_small", kind="session", family="batched", functions=3, samples=100_003),
        dict(name="session_medium", kind="session", family="batched", functions=61, samples=2_000_001),
        # Aggregation alone (a rank's chunk of a sharded batch): launch-ordered samples of many kernels ...
        dict(name="ingest_runs", kind="ingest", family="batched", functions=300, samples=100_000_000,
             order="launch", skip=0),
        # ... and kernels interleaved, an odd count, starting off a 16-byte boundary.
        dict(name="ingest_mixed", kind="ingest", family="batched", functions=100, samples=5_000_003,
             order="interleaved", skip=1),
        # The owner's part of a sharded batch: counts in, blame and the pruned dependency graph out.
        dict(name="blame_edges", kind="blame", family="batched", functions=37, samples=3_000_000),
        # Roll-up, matching, estimators and ranking over blame that is there.
        dict(name="advise_batched", kind="advise", family="batched", functions=301, samples=30_000_000),
        # The dependency graph before pruning and its coverage figures.
        dict(name="graph_unpruned", kind="graph", family="batched", functions=25, samples=1_000_000),
        # The library's scan, called where nothing may be allocated.
        dict(name="scan", kind="scan", values=3_000_001),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "session", "session", "ingest", "ingest", "blame", "advise", "graph",
                       "scan"])
    if kind == "scan":
        return dict(kind=kind, values=_loguniform(rng, 1, 1 << 24))
    if kind == "step":
        family = rng.choice(["rodinia", "batched", "batched", "large"])
        c = dict(kind=kind, family=family, graph=rng.random() < 0.5, launch_stats=rng.random() < 0.5)
        if family == "large":
            c.update(functions=1, instructions=_loguniform(rng, 20_000, 45_000), samples=_loguniform(rng, 10**5, 10**7))
        else:
            c.update(functions=_loguniform(rng, 1, 60 if family == "rodinia" else 900),
                     samples=_loguniform(rng, 10**4, 10**8))
        return c
    c = dict(kind=kind, family=rng.choice(["rodinia", "batched"]))
    if kind == "session":
        c.update(functions=_loguniform(rng, 1, 100), samples=_loguniform(rng, 10**4, 10**7))
    elif kind == "ingest":
        c.update(functions=_loguniform(rng, 1, 500), samples=_loguniform(rng, 10**3, 10**8),
                 order=rng.choice(["launch", "launch", "interleaved"]), skip=rng.randrange(2))
    elif kind == "blame":
        c.update(functions=_loguniform(rng, 1, 60), samples=_loguniform(rng, 10**4, 10**7))
    elif kind == "advise":
        c.update(functions=_loguniform(rng, 1, 500), samples=_loguniform(rng, 10**4, 5 * 10**7))
    else:
        c.update(functions=_loguniform(rng, 1, 30), samples=_loguniform(rng, 10**4, 3 * 10**6))
    return c


# ---------------------------------------------------------------- inputs
def _sizes(case):
    """Instructions asked for per function (the generator adds a few to close blocks)."""
    if case["family"] == "plain":
        return [200]
    if "instructions" in case:
        return [case["instructions"]]
    lo, hi = _RANGES[case["family"]]
    n = case["functions"]
    return [int(lo * (hi / lo) ** ((k + 0.5) / n)) for k in range(n)]


def _program(case, seed):
    """The program's arrays, its generator handle and its samples' seed."""
    rng = np.random.default_rng(case["functions"])
    fam = case["family"]
    if fam == "plain":
        params = [dict(n_instr=200, n_loops=1, max_depth=1, n_regs=64, tmpl=1, zipf_s=1.1, seed=0)]
    else:
        params = []
        for k, n in enumerate(_sizes(case)):
            p = dict(n_instr=n, zipf_s=1.1, seed=case["functions"] * 1_000_003 + k)
            if fam == "rodinia":
                nl = int(rng.integers(1, 5))
                p.update(n_loops=nl, max_depth=nl, n_regs=int(rng.integers(32, 129)))
            elif fam == "batched":
                nl = int(min(64, max(0, round(n / 400 + rng.uniform(-0.5, 1.5)))))
                p.update(n_loops=nl, max_depth=5, n_regs=int(rng.integers(64, 256)))
            else:
                p.update(n_loops=max(1, n // 5000), max_depth=4, n_regs=255, ldg_pct=30)
            params.append(p)
        np.random.default_rng(seed).shuffle(params)
    gen = synth.make_program(params, 1.0, seed)
    arrays = synth.add_calls(gen, 0.1, seed) if fam == "batched" and case["functions"] > 1 else gen.arrays
    return gen, arrays


def _samples(case, gen, seed):
    return gen.samples(case["samples"], seed=seed, order=case.get("order", "launch"))


def _to_device(samples, skip=0):
    t = torch.empty(samples.size + skip, dtype=torch.int64, device="cuda")
    t[skip:].copy_(torch.from_numpy(samples.view(np.int64)))
    return t[skip:]


_ctx = None


def _context():
    """The context that a user's program keeps."""
    global _ctx
    if _ctx is None:
        _ctx = gpa.Context(synth.default_arch())
    return _ctx


class _State:
    """What a program holds between calls; unloads its program when dropped."""
    prog = None

    def __init__(self, case):
        self.case = case

    def __del__(self):
        if self.prog is not None:
            self.prog.unload()


def _stats(case, seed):
    return synth.launch_stats(case["functions"], seed)


def _tables(rows, columns, **more):
    """Arrays of the most edges there can be: a table that a program fills on each pass."""
    return dict({k: np.zeros(rows, t) for k, t in columns.items()}, **more)


def _fill(tables, edges):
    n = len(next(iter(edges.values())))
    for k, v in edges.items():
        tables[k][:n] = v
    return dict(tables, n=n)


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind == "scan":
        g = torch.Generator(device="cuda").manual_seed(seed)
        # counts per block or use: small numbers, many of them zero
        s.values = torch.randint(-3, 9, (case["values"],), generator=g, device="cuda", dtype=torch.int32).clamp_(min=0)
        s.buf = torch.empty_like(s.values)
        s.total = torch.zeros(1, dtype=torch.int32, device="cuda")
        return s
    gen, arrays = _program(case, seed)
    samples = _samples(case, gen, seed)
    if kind == "session":
        _context()
        s.arrays = arrays
        s.samples = torch.from_numpy(samples.view(np.int64)).pin_memory()
        return s
    s.prog = _context().load_program(arrays)
    s.samples = _to_device(samples, case.get("skip", 0))
    n_use = int(np.asarray(arrays["use_res"]).size)
    if kind == "step":
        if case["launch_stats"]:
            s.prog.set_launch_stats(_stats(case, seed), gpa.gpa_sm_model_of_device())
        s.out = s.prog.advice_buffers(pinned=True)
        if case["graph"]:
            s.prog.capture_step(s.samples)
    elif kind == "ingest":
        s.counts = torch.empty(s.prog.n_instr * 24, dtype=torch.int64, device="cuda")
    else:
        s.prog.reset()
        s.prog.ingest(s.samples)
        if kind == "blame":
            s.counts = torch.empty(s.prog.n_instr * 24, dtype=torch.int64, device="cuda")
            s.prog.copy_counts(s.counts)
            s.out = _tables(2 * n_use, dict(j=np.int32, i=np.int32, dmin=np.int32, dlong=np.int32, flags=np.uint32),
                            share=np.zeros((2 * n_use, 4, 2), np.int64))
        elif kind == "advise":
            s.prog.set_launch_stats(_stats(case, seed), gpa.gpa_sm_model_of_device())
            s.prog.blame()
            s.out = s.prog.advice_buffers(pinned=True)
        else:
            s.out = _tables(4 * n_use, {k: np.int32 for k in ("use", "def", "res", "dmin", "K", "dlong")},
                            dom=np.zeros(4 * n_use, np.uint8))
        torch.cuda.synchronize()
        s.samples = None
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    kind = s.case["kind"]
    if kind == "step":
        if s.case["graph"]:
            s.prog.launch_step()
            return s.prog.get_advice(out=s.out)
        s.prog.reset()
        s.prog.ingest(s.samples)
        s.prog.blame()
        return s.prog.advise(out=s.out)
    if kind == "session":
        prog = _context().load_program(s.arrays)
        try:
            prog.reset()
            prog.ingest_host(s.samples)
            prog.blame()
            prog.advise(fetch=False)
            code, _ = prog.status()
            if code != 0:
                raise RuntimeError(f"device status {code}")
            return prog.get_advice()
        finally:
            prog.unload_async()
    if kind == "ingest":
        s.prog.reset()
        s.prog.ingest(s.samples)
        s.prog.copy_counts(s.counts)
        return s.counts
    if kind == "blame":
        s.prog.set_counts(s.counts)
        s.prog.blame()
        return dict(blame=s.prog.blame_counts().view(np.int64), edges=_fill(s.out, s.prog.edges()))
    if kind == "advise":
        return s.prog.advise(out=s.out)
    if kind == "graph":
        return dict(coverage=list(s.prog.coverage()), edges=_fill(s.out, s.prog.unpruned_edges()))
    s.buf.copy_(s.values)
    gpa.gpa_exclusive_scan_noalloc(s.buf, s.total)
    return s.buf, s.total


def work(case):
    """Bytes of one pass: inputs read once, outputs written once."""
    if case["kind"] == "scan":
        return dict(bytes=8 * case["values"] + 4, flops=0)
    ni, nf, n = sum(_sizes(case)), case["functions"], case["samples"]
    code = 27 * ni  # operands (3.5 of 2 bytes), their offsets, class, guard, flags, line; blocks of 7 instructions
    counts = 192 * ni
    advice = nf * 2516 + ni * 6  # per function, and per line and loop (a third of a line an instruction)
    by_kind = dict(step=8 * n + code + advice, session=8 * n + code + advice, ingest=8 * n + counts,
                   blame=code + 2 * counts + 30 * ni, advise=2 * counts + 30 * ni + advice,
                   graph=counts + code + 30 * ni)
    return dict(bytes=by_kind[case["kind"]], flops=0)


# ---------------------------------------------------------------- in 64 bits, by numpy
def _counts(arrays, samples):
    """Samples per (instruction, class, latency flag), as a flat array."""
    off = np.asarray(arrays["func_instr_off"], dtype=np.int64)
    x = samples.view(np.int64)
    kernel = (samples >> np.uint64(48)).astype(np.int64)
    pc = (x >> 24) & 0xFFFFFF
    return np.bincount((off[kernel] + pc) * 24 + ((x >> 19) & 31), minlength=int(off[-1]) * 24)


def _parallel(arrays, samples, stats, sm):
    """Eqs. 6-10 with the occupancy rules of gpa_sm_model: (speedup, warps) per function."""
    nf = int(arrays["n_functions"])
    off = np.asarray(arrays["func_instr_off"], dtype=np.int64)
    x = samples.view(np.int64)
    kernel = (samples >> np.uint64(48)).astype(np.int64)
    total = np.bincount(kernel, minlength=nf).astype(np.float64)
    issued = np.bincount(kernel[((x >> 20) & 15) == 0], minlength=nf).astype(np.float64)
    speedup, warps = np.ones((nf, 2)), np.zeros((nf, 2, 2))
    for f in range(nf):
        blocks, threads, regs, smem = (int(stats[k][f]) for k in ("blocks", "threads_per_block", "regs_per_thread",
                                                                 "smem_per_block"))
        wpb = -(-threads // 32)
        unit = sm["reg_alloc_unit"]
        by_regs = (sm["schedulers_per_sm"] * (sm["regs_per_sm"] // sm["schedulers_per_sm"] //
                                              (-(-regs * 32 // unit) * unit)) if regs else math.inf)
        smem_unit = sm["smem_alloc_unit"]
        by_smem = (sm["smem_per_sm"] // (-(-(smem + sm["smem_reserved_per_block"]) // smem_unit) * smem_unit)
                   if smem else math.inf)
        limits = [sm["max_warps_per_sm"] // wpb, by_regs // wpb, by_smem, sm["max_blocks_per_sm"]]
        resident = min(limits)
        per_sm = -(-blocks // sm["n_sms"])
        w = min(resident, per_sm) * wpb / sm["schedulers_per_sm"]
        merged = min(sm["max_warps_per_sm"], by_regs, by_smem * wpb, -(-blocks * wpb // sm["n_sms"]))
        new = [w * blocks / sm["n_sms"], merged / sm["schedulers_per_sm"]]
        match = [blocks < sm["n_sms"], limits.index(resident) == 3 and per_sm >= resident]
        for k in range(2):
            if not match[k]:
                continue
            warps[f, k] = w, new[k]
            if resident > 0 and total[f] > 0 and issued[f] > 0:
                r = issued[f] / total[f]
                gain = (1 - (1 - r) ** new[k]) / (1 - (1 - r) ** w)
                speedup[f, k] = gain / (new[0] / w) if k == 0 else gain
    assert off.size == nf + 1
    return speedup, warps


def exact(case, seed):
    """Outputs that numpy gives directly; the searches behind blame and edges have no such form."""
    kind = case["kind"]
    if kind == "scan":
        v = prepare(case, seed).values.cpu().numpy().astype(np.int64)
        c = np.cumsum(v)
        return np.concatenate([[0], c[:-1]]).astype(np.int32), np.array([c[-1]], np.int32)
    if kind in ("blame", "graph"):
        return None
    gen, arrays = _program(case, seed)
    samples = _samples(case, gen, seed)
    if kind == "ingest":
        return _counts(arrays, samples)
    out = dict.fromkeys(["totals", "matched", "speedup", "rank", "n_hot", "hot", "loop_active", "loop_matched",
                         "loop_speedup", "line_stall", "line_latency", "par_match", "par_speedup", "par_warps",
                         "par_limit"])
    nf = case["functions"]
    if kind == "advise" or case.get("launch_stats"):
        out["par_speedup"], out["par_warps"] = _parallel(arrays, samples, _stats(case, seed),
                                                         gpa.gpa_sm_model_of_device())
    else:
        out["par_speedup"], out["par_warps"] = np.ones((nf, 2)), np.zeros((nf, 2, 2))
    return out
