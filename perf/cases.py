"""What this library's speed is judged by: the calls a user's program makes,
through the public entry points, over the sizes in use.

Three kinds of program use the library.  One evolves a population: it holds a
grid, advances it by some generations and reads the population (and often a
sample) back, over and over; that is every "grid" case, from the 512-agent
grid to the 16.8M-agent one, for island sizes, tournaments, fitness models
and surface widths in use.  One runs many replicates at once ("batch").  One
studies the end state: it samples genomes ("sample") and rebuilds their
phylogeny ("tree").

Synchronous migration only: free-running grids take whatever their
neighbours last published, so two runs on the same inputs give different
populations and cannot be compared value by value.

Every output is a whole number (integer traits, surface words, binary32
fitness as the 32-bit word the genome stores, node indices and times), so
equality with earlier outputs is the whole check and `exact` has nothing to
add.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2404_10861_gb300 import binding as hb

# One Philox4x32-10 block: ten rounds of two wide multiplies and four xors.
OPS_PER_BLOCK = 60

_stream = None


def _the_stream():
    """The one stream of the program; device memory comes from torch's caching
    allocator, as in the benchmark."""
    global _stream
    if _stream is None:
        hb.use_torch_allocator()
        _stream = torch.cuda.Stream()
    return _stream


def _grid(name, rows, cols, gens, n=32, tournament=2, policy="tilted", bits=1, W=2, interval=1,
          p_ben=1e-3, p_del=0.0, coarsen=1, words=1, sigma=0.0, sample=0):
    return dict(name=name, kind="grid", rows=rows, cols=cols, gens=gens, n=n,
                tournament=tournament, policy=policy, bits=bits, W=W, interval=interval,
                p_ben=p_ben, p_del=p_del, coarsen=coarsen, words=words, sigma=sigma,
                sample=sample)


def listed():
    return [
        # the 4x4-island grid of the tiny workload, advanced by one serving
        # slice (256 generations), every island sampled: the smallest call
        _grid("tiny slice", 4, 4, 256, policy="steady", p_ben=0.0, sample=16),
        # the 64x64-island adaptive workload under the 2-bit tilted surface
        _grid("mid 64x64", 64, 64, 256, bits=2),
        # a request of the serving stream's upper middle: half a million
        # agents, whose population fits in L2 but not on the SMs
        _grid("serve 128x128", 128, 128, 256, policy="stretched", p_ben=0.0),
        # the 16.8M-agent grid of the benchmark
        _grid("wafer 512x1024", 512, 1024, 32),
        # the paper's on-hardware trial at its middle size: tournament 5, a
        # third of the mutations deleterious, integer fitness
        _grid("trial 500x500 t5", 500, 500, 16, tournament=5, p_ben=0.003, p_del=0.33),
        # the same trial with the paper's binary32 fitness
        _grid("trial 500x500 float", 500, 500, 8, tournament=5, p_ben=0.003, p_del=0.33,
              sigma=1.0),
        # a 2:1 torus of the replicate mix with more agents than lanes
        _grid("replicate 128x256 n48", 128, 256, 32, n=48, policy="steady"),
        # the 256-bit surface of the paper's figure (precision studies)
        _grid("wide 256x512 K4", 256, 512, 8, words=4),
        # independent replicates of uneven size and length in one batch,
        # from admission to their populations
        dict(name="batch of 16", kind="batch", runs=16, mix=4, gen_scale=200),
        # the end-state sample: 10,000 genomes of the 16.8M-agent grid
        dict(name="sample 10k of wafer", kind="sample", rows=512, cols=1024, n=32, k=10_000),
        # phylogeny of such a sample, host arrays in and out
        dict(name="tree 10k host", kind="tree", k=10_000, policy="tilted", bits=1, words=1,
             gens=1000, host=True),
        # phylogeny of a million genomes that are already on the device
        dict(name="tree 1M", kind="tree", k=1_000_000, policy="tilted", bits=1, words=1,
             gens=1000, host=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "grid", "float", "wide", "batch", "sample", "tree"])
    if kind == "batch":
        return dict(kind="batch", runs=rng.randint(6, 16), mix=rng.randint(5, 1000),
                    gen_scale=rng.randint(250, 1000))
    if kind == "sample":
        rows, cols = _log_int(rng, 16, 512), _log_int(rng, 16, 1024)
        k = min(rows * cols, _log_int(rng, 64, 16384))
        return dict(kind="sample", rows=rows, cols=cols, n=rng.choice([32, 32, 17, 48]), k=k)
    if kind == "tree":
        return dict(kind="tree", k=_log_int(rng, 500, 1_000_000),
                    policy=rng.choice(["steady", "tilted", "stretched", "hybrid"]),
                    bits=rng.choice([1, 1, 2, 4]), words=rng.choice([1, 1, 1, 2, 4]),
                    gens=rng.randint(100, 2000), host=rng.random() < 0.5)
    flt, wide = kind == "float", kind == "wide"
    # islands from 16 up to the benchmark's 524,288 (fewer where the genome is
    # larger), any aspect, odd sides among them
    islands = _log_int(rng, 16, 524_288 if kind == "grid" else 200_000)
    rows = max(1, int(math.sqrt(islands) * rng.choice([0.5, 0.7, 1.0])))
    cols = max(1, islands // rows)
    n = 32 if rng.random() < 0.6 else rng.randint(16, 32 if flt or wide else 64)
    if rows * cols * n > 16_777_216:
        rows = max(1, 16_777_216 // (cols * n))
    agents = rows * cols * n
    gens = max(1, min(_log_int(rng, 4, 512), int((5e8 if kind == "grid" else 5e7) // agents)))
    bits = rng.choice([1, 1, 2, 4])
    policy = rng.choice(["steady", "tilted", "stretched", "hybrid"] if wide else
                        ["steady", "tilted", "stretched", "hybrid", "none"])
    trial = flt or rng.random() < 0.3
    return {k: v for k, v in _grid(
        "", rows, cols, gens, n=n, tournament=5 if trial else rng.choice([2, 2, 3]),
        policy=policy, bits=bits, interval=rng.choice([1, 1, 1, 2]),
        p_ben=rng.choice([1e-3, 0.0]) if not trial else 0.003, p_del=0.33 if trial else 0.0,
        coarsen=rng.choice([1, 1, 1, 3]), words=rng.choice([2, 4]) if wide else 1,
        sigma=1.0 if flt else 0.0,
        sample=min(rows * cols, rng.choice([0, 16, 1000]))).items() if k != "name"}


def _mix(case):
    """The replicate mix: grid side uniform over {8..256}, square or 2:1,
    16-64 agents per island, steady / tilted / stretched, adaptation on or
    off, 10,000-200,000 generations divided by gen_scale."""
    r = np.random.default_rng(case["mix"])
    runs = []
    for _ in range(case["runs"]):
        side = int(r.choice([8, 16, 32, 64, 128, 256]))
        rows, cols = (side, side) if r.random() < 0.5 else (side, 2 * side)
        n = int(r.integers(16, 65))
        policy = str(r.choice(["steady", "tilted", "stretched"]))
        p_ben = 1e-3 if r.random() < 0.5 else 0.0
        gens = int(r.integers(10_000, 200_001)) // case["gen_scale"]
        runs.append((gens, dict(rows=rows, cols=cols, n=n, tournament=2, policy=policy, bits=1,
                                W=2, interval=1, p_ben=p_ben, p_del=0.0)))
    return runs


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _population(g, agents, words, flt):
    """A population some way into a run: fitnesses a few steps apart, with
    ties, and surfaces whose bits are random."""
    if flt:
        trait = torch.randn(agents, device="cuda", generator=g).view(torch.int32)
    else:
        trait = torch.randint(0, 12, (agents,), device="cuda", generator=g, dtype=torch.int32)
    half = [torch.randint(0, 2**32, (agents * words,), device="cuda", generator=g,
                          dtype=torch.int64) for _ in range(2)]
    return trait, (half[0] << 32) | half[1]


def _config(case, seed):
    kw = dict(rows=case["rows"], cols=case["cols"], n=case["n"], tournament=case["tournament"],
              policy=case["policy"], bits=case["bits"], W=case["W"], interval=case["interval"],
              p_ben=case["p_ben"], p_del=case["p_del"], coarsen=case["coarsen"],
              words=case["words"], seed=1 + seed)
    if case["sigma"] > 0:
        kw.update(fitness="float", sigma=case["sigma"])
    return kw


def prepare(case, seed):
    stream = _the_stream()
    g = _generator(seed)
    st = dict(case=case, stream=stream)
    kind = case["kind"]
    if kind == "batch":
        st["runs"] = [(gens, dict(kw, seed=1 + seed * 1000 + i))
                      for i, (gens, kw) in enumerate(_mix(case))]
        st["out"] = []
        for _, kw in st["runs"]:
            agents = kw["rows"] * kw["cols"] * kw["n"]
            st["out"].append((torch.empty(agents, dtype=torch.int32, device="cuda"),
                              torch.empty(agents, dtype=torch.int64, device="cuda")))
        return st
    if kind == "tree":
        # genomes of a population that has evolved for `gens` generations
        words, k = case["words"], case["k"]
        side = 64
        while side * side * 32 < k:
            side *= 2
        agents = side * side * 32
        with hb.Grid(stream=stream.cuda_stream, rows=side, cols=side, n=32, tournament=2,
                     policy=case["policy"], bits=case["bits"], W=2, p_ben=1e-3, words=words,
                     seed=1 + seed) as grid:
            t = torch.empty(agents, dtype=torch.int32, device="cuda")
            s = torch.empty(agents * words, dtype=torch.int64, device="cuda")
            torch.cuda.current_stream().synchronize()
            grid.run(case["gens"])
            hb.hsga_get_population(grid.handle, t, s)
            grid.sync()
        pick = torch.randperm(agents, device="cuda", generator=g)[:k]
        surf = s.view(agents, words)[pick].contiguous()
        # node arrays hold up to 2k + 1 entries; a tree's are the first n_nodes
        out = [torch.zeros(2 * k + 1, dtype=torch.int64, device="cuda"),
               torch.zeros(2 * k + 1, dtype=torch.int64, device="cuda"),
               torch.zeros(k, dtype=torch.int32, device="cuda")]
        if case["host"]:
            surf, out = surf.cpu(), [o.cpu() for o in out]
        st["surf"], st["out"] = surf, out
        torch.cuda.current_stream().synchronize()
        return st
    words = case.get("words", 1)
    agents = case["rows"] * case["cols"] * case["n"]
    if kind == "sample":
        kw = dict(rows=case["rows"], cols=case["cols"], n=case["n"], tournament=2,
                  policy="tilted", bits=1, W=2, p_ben=1e-3, seed=1 + seed)
        k = case["k"]
    else:
        kw = _config(case, seed)
        k = case["sample"]
    grid = hb.Grid(stream=stream.cuda_stream, **kw)
    t, s = _population(g, agents, words, kw.get("fitness") == "float")
    torch.cuda.current_stream().synchronize()
    hb.hsga_set_population(grid.handle, t, None if kw["policy"] == "none" else s,
                           1000 + seed % 1000)
    grid.sync()
    st["grid"] = grid
    if kind == "grid":
        st["out"] = (t, s)   # read back into the buffers that held the start
    if k:
        st["words"] = torch.empty((k, 2 + 2 * words), dtype=torch.int32, device="cuda")
        st["where"] = torch.empty((k, 2), dtype=torch.int32, device="cuda")
    torch.cuda.current_stream().synchronize()
    return st


def _run_batch(st):
    with hb.Batch(stream=st["stream"].cuda_stream) as b:
        ids = [b.add(gens, **kw) for gens, kw in st["runs"]]
        b.run(10**9)
        for rid, (t, s) in zip(ids, st["out"]):
            hb.hsga_batch_get_population(b.handle, rid, t, s)
    return st["out"]


def _run_tree(st):
    case, k = st["case"], st["case"]["k"]
    parent, time, leaf = st["out"]
    nodes = ctypes.c_uint32(0)
    status = hb.lib().hsga_reconstruct(
        st["surf"].data_ptr(), k, case["words"], hb.POLICIES[case["policy"]], case["bits"], 2,
        case["gens"], 1, parent.data_ptr(), time.data_ptr(), leaf.data_ptr(), 2 * k + 1,
        ctypes.byref(nodes), ctypes.c_void_p(st["stream"].cuda_stream))
    if status:
        raise hb.HsgaError(status, "hsga_reconstruct")
    return parent, time, leaf, nodes.value


def run(st):
    kind = st["case"]["kind"]
    if kind == "batch":
        return _run_batch(st)
    if kind == "tree":
        return _run_tree(st)
    g = st["grid"].handle
    out = ()
    if kind == "grid":
        hb.hsga_run_generations(g, st["case"]["gens"])
        t, s = st["out"]
        hb.hsga_get_population(g, t, s)
        out = (t, s)
    if "words" in st:
        hb.hsga_sample_surfaces(g, st["words"].shape[0], st["words"], st["where"])
        out += (st["words"], st["where"])
    return out


def work(case):
    """Bytes: what goes in read once, what comes out written once.  flops:
    integer operations of the Philox blocks the replications draw."""
    kind = case["kind"]
    if kind == "tree":
        k = case["k"]   # surfaces in; parent, time and leaf index out
        return dict(bytes=k * (8 * case["words"] + 36), flops=0)
    if kind == "sample":
        return dict(bytes=case["k"] * (12 + 24), flops=2 * case["k"] * OPS_PER_BLOCK)
    if kind == "batch":
        agents = sum(kw["rows"] * kw["cols"] * kw["n"] for _, kw in _mix(case))
        reps = sum(g * kw["rows"] * kw["cols"] * kw["n"] for g, kw in _mix(case))
        return dict(bytes=agents * 24, flops=reps * OPS_PER_BLOCK)
    agents = case["rows"] * case["cols"] * case["n"]
    genome = 4 + (0 if case["policy"] == "none" else 8 * case["words"])
    blocks = 1 + math.ceil(max(0, case["tournament"] - 2) / 4)
    if case["sigma"] > 0:   # the Gaussian amount of the children that mutate
        blocks += case["p_ben"] + case["p_del"]
    return dict(bytes=2 * agents * genome + case["sample"] * (16 + 16 * case["words"]),
                flops=agents * case["gens"] * blocks * OPS_PER_BLOCK)


def exact(case, seed):
    return None   # whole numbers throughout
