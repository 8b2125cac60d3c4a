"""Workloads of the walk engine, from one short query to whole-graph corpora.

A case is a dict of plain values:
  kind     "walk" (device buffers), "host" (host buffers), "batch" (a table of
           jobs, one call or a captured plan), "create" (build a graph, then
           its first walks)
  scale, edge_factor, skewed
           R-MAT graph of 2^scale nodes, edge_factor * 2^scale generated
           edges; quadrant probabilities (.57, .19, .19) or (.7, .1, .1)
  weights  "none" (h = 1), "uniform" (0, 1], "lognormal" (0, 1), "pareto1" /
           "pareto2" (tail exponent 1 / 2), "uniform8" (8-bit codes)
  algo, mode, p, q, walkers, length
           the arguments of the walk; starts are nodes that have an edge
  jobs, plan
           batch: number of jobs (their walkers spread geometrically up to
           `walkers`, their lengths between 5 and `length`) and whether they
           run as a captured plan

Graphs, weights, labels and starts are made on the GPU from the seed alone.
"""
import math

import torch

from paper_2512_00705_gb300 import flexiwalk as fw

SCHEMA = [0, 1, 2, 3, 4]  # metapath: cyclic label schema over labels 0..4
RECORD = 32               # bytes of one random access to memory


def _case(name, kind, **more):
    c = {"kind": kind, "scale": 20, "edge_factor": 16, "skewed": False, "weights": "uniform", "algo": "node2vec",
         "mode": "auto", "p": 1.0, "q": 1.0, "walkers": 1, "length": 80, "jobs": 0, "plan": False}
    c.update(more)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one small online query (a user's handful of seed nodes): launch and latency
        _case("query_small", "walk", scale=18, walkers=37, length=10, p=2.0, q=0.5),
        # a typical served query, too small to fill the GPU; odd sizes
        _case("query_mid", "walk", scale=20, walkers=5003, length=63, p=0.5, q=2.0),
        # the headline corpus: one walker per node with an edge, 80 hops; first-order (DeepWalk-like),
        # breadth-first and depth-first settings of node2vec
        _case("corpus_p1_q1", "walk", scale=22, walkers=2395919, p=1.0, q=1.0),
        _case("corpus_p4_q025", "walk", scale=20, walkers=646203, p=4.0, q=0.25),
        _case("corpus_p025_q4", "walk", scale=22, walkers=2395919, p=0.25, q=4.0),
        # heterogeneous graph: label-constrained walks from random seeds, lognormal weights
        _case("metapath", "walk", scale=21, weights="lognormal", algo="metapath", walkers=1000003, length=40),
        # second-order PageRank by sampled walks
        _case("pagerank2", "walk", scale=20, algo="pagerank2", walkers=262144, length=40),
        # heavy-tailed weights: the cost model sends many steps to the reservoir sampler
        _case("skewed_weights", "walk", scale=20, weights="pareto1", p=2.0, q=0.5, walkers=131072, length=40),
        # the reservoir sampler alone (one pass over every row, no bound needed)
        _case("reservoir_only", "walk", scale=18, mode="rvs", p=2.0, q=0.5, walkers=65536, length=20),
        # many requests of all sizes and algorithms on a skewed graph, as one captured plan
        _case("batch_mixed", "batch", scale=20, edge_factor=24, skewed=True, walkers=131072, length=80, jobs=64,
              plan=True),
        # a corpus through pinned host buffers: starts in, rows out
        _case("host_corpus", "host", scale=20, walkers=700001, length=80, p=2.0, q=0.5),
        # a graph arrives on the device: checks, preprocessing, its first walks
        _case("create_graph", "create", scale=20, walkers=4099, length=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["walk", "walk", "walk", "walk", "walk", "host", "batch", "create"])
    scale = rng.randint(12, 21)
    ef = rng.choice([4, 8, 16, 24]) if scale < 21 else rng.choice([4, 8, 16])
    c = _case(None, kind, scale=scale, edge_factor=ef, skewed=rng.random() < 0.25,
              weights=rng.choice(["uniform", "uniform", "none", "lognormal", "pareto2", "uniform8"]),
              p=rng.choice([0.25, 0.5, 1.0, 2.0, 4.0]), q=rng.choice([0.25, 0.5, 1.0, 2.0, 4.0]),
              length=_log_int(rng, 3, 120))
    if kind == "create":
        c.update(weights=rng.choice(["uniform", "none", "lognormal"]), walkers=rng.randint(100, 8000),
                 length=rng.randint(3, 30))
        return c
    if kind == "batch":
        c.update(weights=rng.choice(["uniform", "lognormal"]), jobs=rng.randint(2, 64), plan=rng.random() < 0.5,
                 length=rng.randint(10, 100))
        c["walkers"] = _log_int(rng, 100, min(200000, (1 << 26) // (c["length"] * c["jobs"])))
        return c
    hops = 1 << 26
    if kind == "walk":
        c["algo"] = rng.choice(["node2vec", "node2vec", "weighted", "metapath", "pagerank2"])
        if c["algo"] == "pagerank2":
            hops = 1 << 22
        if rng.random() < 0.2:
            c.update(weights=rng.choice(["pareto1", "pareto2"]))
        if c["algo"] != "metapath" and rng.random() < 0.2:
            c["mode"] = "rvs"
        if c["mode"] == "rvs" or c["weights"].startswith("pareto"):
            c["scale"] = min(scale, 18)
            hops = 1 << 20
    c["walkers"] = _log_int(rng, 1, max(2, hops // c["length"]))
    return c


# ---------------------------------------------------------------- inputs
def _mix(x):
    """64-bit mix of int64 values (wrapping arithmetic, logical shifts)."""
    x = x + -7046029254386353131
    x = (x ^ ((x >> 30) & 0x3FFFFFFFF)) * -4658895280553007687
    x = (x ^ ((x >> 27) & 0x1FFFFFFFFF)) * -7723592293110705685
    return x ^ ((x >> 31) & 0x1FFFFFFFF)


def _salt(seed, use):
    return ((2 * seed + 1) * 0x9E3779B97F4A7C15 * (2 * use + 1)) & ((1 << 62) - 1)


def _unit(x):
    """(0, 1) in double from the top bits of mixed int64 values."""
    return (((x >> 32) & 0xFFFFFFFF).double() + 0.5) * 2.0 ** -32


def _csr(case, seed, labels):
    """Symmetric CSR without loops or duplicates, weights and labels equal on mirrored entries."""
    dev = torch.device("cuda")
    scale, n = case["scale"], 1 << case["scale"]
    a, b, c = (0.7, 0.1, 0.1) if case["skewed"] else (0.57, 0.19, 0.19)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    m = case["edge_factor"] << scale
    src = torch.zeros(m, dtype=torch.int32, device=dev)
    dst = torch.zeros(m, dtype=torch.int32, device=dev)
    for _ in range(scale):
        r = torch.rand(m, generator=gen, device=dev)
        src.mul_(2).add_(r >= a + b)
        dst.mul_(2).add_(((r >= a) & (r < a + b)) | (r >= a + b + c))
    perm = torch.randperm(n, generator=gen, device=dev)
    src, dst = perm[src.long()], perm[dst.long()]
    keep = src != dst
    src, dst = src[keep], dst[keep]
    key = torch.unique(torch.cat([(src << scale) | dst, (dst << scale) | src]))
    del src, dst, keep, r
    row, col = key >> scale, key & (n - 1)
    offsets = torch.zeros(n + 1, dtype=torch.int32, device=dev)
    offsets[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    edge = (torch.minimum(row, col) << scale) | torch.maximum(row, col)
    del key, row
    weights = None
    if case["weights"] != "none":
        u = _unit(_mix(edge + _salt(seed, 1)))
        if case["weights"] == "lognormal":
            v = _unit(_mix(edge + _salt(seed, 2)))
            u = torch.exp(torch.sqrt(-2.0 * torch.log(u)) * torch.cos(2.0 * math.pi * v))
        elif case["weights"].startswith("pareto"):
            u = u ** (-1.0 / int(case["weights"][-1]))
        weights = u.float()
        del u
    lab = None
    if labels:
        lab = (((_mix(edge + _salt(seed, 3)) >> 32) & 0xFFFF) % len(SCHEMA)).to(torch.uint8)
    return offsets, col.int(), weights, lab, gen


def _starts(offsets, walkers, gen):
    nodes = torch.nonzero(offsets[1:] > offsets[:-1]).flatten()
    pick = torch.randint(nodes.numel(), (walkers,), generator=gen, device=nodes.device)
    return nodes[pick].int()


def _job_shapes(case):
    """(walkers, length, algo, p, q) of a batch's jobs."""
    jobs, most, longest = case["jobs"], case["walkers"], case["length"]
    settings = [("node2vec", 1.0, 1.0), ("node2vec", 4.0, 0.25), ("metapath", 1.0, 1.0), ("node2vec", 0.25, 4.0),
                ("weighted", 1.0, 1.0)]
    out = []
    for j in range(jobs):
        w = max(1, int(most * 100.0 ** (j / max(1, jobs - 1) - 1)))
        out.append((w, 5 + (37 * j) % max(1, longest - 4)) + settings[j % len(settings)])
    return out


def _needs_labels(case):
    return case["kind"] in ("batch", "create") or case["algo"] == "metapath"


def prepare(case, seed):
    offsets, cols, weights, labels, gen = _csr(case, seed, _needs_labels(case))
    if case["kind"] == "create":
        return {"case": case, "seed": seed, "csr": (offsets, cols, weights, labels),
                "starts": _starts(offsets, case["walkers"], gen)}
    graph = fw.Graph(offsets=offsets, cols=cols, weights=weights, labels=labels)
    if case["weights"] == "uniform8":
        graph.quantize_weights()
    state = {"case": case, "seed": seed, "graph": graph}
    w, length = case["walkers"], case["length"]
    if case["kind"] == "batch":
        shapes = _job_shapes(case)
        rows = torch.empty(sum(s[0] * (s[1] + 1) for s in shapes), dtype=torch.int32, device="cuda")
        starts = _starts(offsets, sum(s[0] for s in shapes), gen)
        jobs, at, out_at = [], 0, 0
        for j, (jw, jl, algo, p, q) in enumerate(shapes):
            out = rows[out_at:out_at + jw * (jl + 1)]
            jobs.append(fw.make_job(starts[at:at + jw], jl, algo, out, p=p, q=q, seed=seed + j,
                                    schema=SCHEMA if algo == "metapath" else None))
            at, out_at = at + jw, out_at + jw * (jl + 1)
        state.update(starts=starts, out=rows, jobs=jobs)
        if case["plan"]:
            state["plan"] = fw.BatchPlan(graph, jobs)
    elif case["kind"] == "host":
        state["starts"] = _starts(offsets, w, gen).cpu().pin_memory()
        state["out"] = torch.empty((w, length + 1), dtype=torch.int32, pin_memory=True)
    else:
        state["starts"] = _starts(offsets, w, gen)
        state["out"] = torch.empty((w, length + 1), dtype=torch.int32, device="cuda")
    return state


# ---------------------------------------------------------------- one pass
def run(state):
    case, seed = state["case"], state["seed"]
    if case["kind"] == "create":
        offsets, cols, weights, labels = state["csr"]
        graph = fw.Graph(offsets=offsets, cols=cols, weights=weights, labels=labels)
        hmax, hsum = graph.node_stats()
        out = {"hmax": hmax, "hsum": hsum, "label_stats": graph.label_stats(),
               "node2vec": graph.walk(state["starts"], case["length"], "node2vec", p=case["p"], q=case["q"], seed=seed),
               "metapath": graph.walk(state["starts"], case["length"], "metapath", schema=SCHEMA, seed=seed)}
        graph.close()
        return out
    if case["kind"] == "batch":
        if case["plan"]:
            state["plan"].launch()
        else:
            fw.fw_walk_batch(state["graph"].handle, state["jobs"])
        return state["out"]
    walk = state["graph"].walk_host if case["kind"] == "host" else state["graph"].walk
    return walk(state["starts"], case["length"], case["algo"], p=case["p"], q=case["q"], mode=case["mode"], seed=seed,
                schema=SCHEMA if case["algo"] == "metapath" else None, out=state["out"])


def _walk_bytes(walkers, length):
    # starts in, rows out, and one random access per hop: the neighbour taken with its weight
    return 4 * walkers + 4 * walkers * (length + 1) + RECORD * walkers * length


def work(case):
    if case["kind"] == "batch":
        return {"bytes": sum(_walk_bytes(s[0], s[1]) for s in _job_shapes(case)), "flops": 0}
    total = _walk_bytes(case["walkers"], case["length"])
    if case["kind"] == "create":
        # The CSR in (twice: checked, copied) and out, then what a graph keeps per entry: 32-byte records in row order,
        # class order (with weights) and label order with the grouped weight, 8 bytes of membership table and 1 of
        # filter; per node 32 + 8 bytes of statistics and, for eight labels, 8 * (32 + 8), a filter and a table block.
        n, e = 1 << case["scale"], 2 * (case["edge_factor"] << case["scale"])
        h = 0 if case["weights"] == "none" else 1
        total = 2 * total + e * (3 * (5 + 4 * h) + 32 * (2 + h) + 4 + 9) + n * (12 + 40 + 320 + 64)
    return {"bytes": total, "flops": 0}


# ---------------------------------------------------------------- 64-bit answers
def exact(case, seed):
    """Row statistics of a new graph in 64 bits; walks are whole numbers and have no such value."""
    if case["kind"] != "create":
        return None
    offsets, cols, weights, labels, _ = _csr(case, seed, True)
    n, kinds = offsets.numel() - 1, 8
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), (offsets[1:] - offsets[:-1]).long())
    h = torch.ones(cols.numel(), dtype=torch.float64, device="cuda") if weights is None else weights.double()
    place = row * kinds + labels.long()

    def stats(index, size):
        top = torch.zeros(size, dtype=torch.float64, device="cuda").scatter_reduce_(0, index, h, "amax")
        return top, torch.zeros(size, dtype=torch.float64, device="cuda").index_add_(0, index, h)

    hmax, hsum = stats(row, n)
    lmax, lsum = stats(place, n * kinds)
    return {"hmax": hmax, "hsum": hsum, "label_stats": torch.stack([lmax, lsum], 1).reshape(n, kinds, 2),
            "node2vec": None, "metapath": None}
