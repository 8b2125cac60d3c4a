"""Rows at the edges of the launch shapes: just below, at and just above every
walker count at which a variant of 3 to 7 blocks per SM has no lane (or, for
jobs that scan rows, no warp place) left and its walkers come from a queue."""
import numpy as np
import pytest

import oracle
from paper_2512_00705_gb300 import flexiwalk as fw
from paper_2512_00705_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BPS = [3, 4, 5, 7]


@pytest.fixture(scope="module", params=[2, 16])  # short rows (32 or 16 walkers per warp scan) and longer ones
def graph(request):
    g = synth.rmat(12, request.param, seed=1)
    g.h = synth.edge_weights(g, "uniform01", seed=2)
    g.labels = synth.edge_labels(g, 5, seed=3)
    G = fw.Graph(g)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    starts = torch.from_numpy(synth.random_starts(g.n, sms * 7 * 256 + 64, seed=5)).cuda()
    yield g, G, sms, starts
    G.close()


ALGOS = [("weighted", 1.0, 1.0), ("node2vec", 2.0, 0.5), ("node2vec", 0.25, 4.0), ("node2vec", 4.0, 1.0),
         ("node2vec", 0.5, 1.0), ("metapath", 1.0, 1.0), ("pagerank2", 1.0, 1.0)]


@pytest.mark.parametrize("algo,p,q", ALGOS)
@pytest.mark.parametrize("mode,ratio", [("auto", 4.0), ("auto", 8.0), ("auto", 0.5), ("rjs", 0.0), ("random", 0.0)])
def test_lanes_run_out(graph, algo, p, q, mode, ratio):
    g, G, sms, starts = graph
    kw = dict(p=p, q=q, mode=mode, cost_ratio=ratio, schema=[0, 1, 2] if algo == "metapath" else None, seed=8)
    ref = G.walk(starts, 3, algo, flags=fw.FLAG_COUNTERS, **kw)  # a walker's row does not depend on the others
    for bps in BPS:
        for more in (-1, 0, 1, 33):
            w = sms * bps * 256 + more
            assert torch.equal(G.walk(starts[:w], 3, algo, **kw), ref[:w]), w
    G.check()


@pytest.mark.parametrize("algo,p,q", ALGOS)
@pytest.mark.parametrize("mode", ["exact", "rvs"])
def test_places_run_out(graph, algo, p, q, mode):
    g, G, sms, starts = graph
    kw = dict(p=p, q=q, mode=mode, schema=[0, 1, 2] if algo == "metapath" else None, seed=8)
    ref = G.walk(starts, 2, algo, flags=fw.FLAG_COUNTERS, **kw)
    for bps in BPS:
        for wpw in (1, 4, 8, 16, 32):
            for more in (-1, 0, 1):
                w = sms * bps * 8 * wpw + more
                assert torch.equal(G.walk(starts[:w], 2, algo, **kw), ref[:w]), w
    if mode == "exact":
        few = starts[:4096].cpu().numpy()
        want, _ = oracle.walk(g, few, 2, algo, p, q, schema=kw["schema"], seed=8)
        assert np.array_equal(ref[:4096].cpu().numpy(), want)


@pytest.mark.parametrize("mode", ["exact", "rvs"])
@pytest.mark.parametrize("draws", [1, 1000, 40_000, 400_000])
def test_histograms_of_scans(graph, mode, draws):
    g, G, sms, starts = graph
    v = int(np.argmax(np.diff(g.offsets)))
    for node in (v, int(g.cols[g.offsets[v]])):
        a = G.sample_hist(node, -1, 0, "weighted", draws, mode=mode, seed=4)
        b = G.sample_hist(node, -1, 0, "weighted", draws, mode=mode, seed=4, flags=fw.FLAG_COUNTERS)
        assert int(a.sum()) == draws and torch.equal(a, b)
