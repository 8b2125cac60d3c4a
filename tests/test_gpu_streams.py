"""Launches side by side take another shape than a launch alone (their share
of the GPU): on eight streams in turn every walk and batch has the rows that
the counting build, which keeps one shape, gives."""
import pytest

from paper_2512_00705_gb300 import flexiwalk as fw
from paper_2512_00705_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LEN = 6
WALKERS = [1, 300, 3001, 9800, 20000, 40000, 78000, 156000]  # either side of a share's warps and of the GPU's


@pytest.fixture(scope="module")
def graph():
    g = synth.workload_graph("small")
    G = fw.Graph(g)
    starts = torch.from_numpy(synth.random_starts(g.n, max(WALKERS), seed=17)).cuda()
    streams = [torch.cuda.Stream() for _ in range(8)]
    yield G, starts, streams
    G.close()


@pytest.mark.parametrize("algo,p,q", [("weighted", 1.0, 1.0), ("node2vec", 2.0, 0.5), ("node2vec", 0.25, 4.0),
                                      ("metapath", 1.0, 1.0), ("pagerank2", 1.0, 1.0)])
@pytest.mark.parametrize("mode,ratio", [("auto", 4.0), ("auto", 0.5), ("rvs", 4.0), ("exact", 4.0)])
def test_walks_on_eight_streams(graph, algo, p, q, mode, ratio):
    G, starts, streams = graph
    kw = dict(p=p, q=q, mode=mode, cost_ratio=ratio, schema=[0, 1, 2] if algo == "metapath" else None)
    sizes = [(w, k) for k, w in enumerate(WALKERS * 2)]
    outs = [torch.full((w, LEN + 1), -7, dtype=torch.int32, device="cuda") for w, _ in sizes]
    torch.cuda.synchronize()
    for w, k in sizes:
        G.walk(starts[:w], LEN, algo, seed=k, out=outs[k], stream=streams[k % 8], **kw)
    torch.cuda.synchronize()
    for w, k in sizes:
        ref = G.walk(starts[:w], LEN, algo, seed=k, flags=fw.FLAG_COUNTERS, **kw)
        assert torch.equal(outs[k], ref), (w, k)


def test_batches_on_eight_streams(graph):
    G, starts, streams = graph
    todo, outs = [], []
    for k in range(16):
        jobs = []
        for j, (algo, p, q) in enumerate([("weighted", 1.0, 1.0), ("node2vec", 2.0, 0.5), ("metapath", 1.0, 1.0),
                                          ("node2vec", 0.25, 4.0), ("pagerank2", 1.0, 1.0)]):
            w = WALKERS[(k + j) % 7]
            out = torch.full((w, LEN + 1), -7, dtype=torch.int32, device="cuda")
            kw = dict(p=p, q=q, schema=[0, 1, 2] if algo == "metapath" else None, seed=10 * k + j)
            jobs.append(fw.make_job(starts[:w], LEN, algo, out, **kw))
            outs.append((out, w, algo, kw))
        todo.append(jobs)
    torch.cuda.synchronize()
    for k, jobs in enumerate(todo):
        fw.fw_walk_batch(G.handle, jobs, stream=streams[k % 8])
    torch.cuda.synchronize()
    for out, w, algo, kw in outs:
        assert torch.equal(out, G.walk(starts[:w], LEN, algo, flags=fw.FLAG_COUNTERS, **kw))
