"""Trial caps at the end of their range: forced eRJS with a cap near 2^31
never hands a step to eRVS, whichever kernel variant makes the trials."""
import numpy as np
import pytest

import oracle
from paper_2512_00705_gb300 import flexiwalk as fw
from paper_2512_00705_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MOST = 2**31 - 1


@pytest.fixture(scope="module", params=["pareto", "uniform"])
def graph(request):
    g = synth.workload_graph("small")
    if request.param == "pareto":  # trials together in every algorithm; on uniform weights in PageRank only
        g.h = synth.edge_weights(g, "pareto", 1.0, seed=7)
    G = fw.Graph(g)
    yield request.param, g, G
    G.close()


@pytest.mark.parametrize("algo,p,q", [("weighted", 1.0, 1.0), ("node2vec", 2.0, 0.5), ("node2vec", 0.25, 4.0),
                                      ("metapath", 1.0, 1.0), ("pagerank2", 1.0, 1.0)])
@pytest.mark.parametrize("cap,batch", [(MOST, 0), (MOST, 16), (MOST - 1, 5), (MOST - 31, 2)])
@pytest.mark.parametrize("walkers,length", [(4099, 12), (180000, 2)])
def test_a_cap_near_the_largest_integer_is_never_met(graph, algo, p, q, cap, batch, walkers, length):
    kind, g, G = graph
    starts = synth.random_starts(g.n, walkers, seed=11)
    dev = torch.from_numpy(starts).cuda()
    more = dict(p=p, q=q, schema=[0, 1, 2] if algo == "metapath" else None, mode="rjs", seed=3, rjs_cap=cap,
                rjs_batch=batch)
    a = G.walk(dev, length, algo, **more)
    G.reset_counters()
    b = G.walk(dev, length, algo, flags=fw.FLAG_COUNTERS, **more)
    assert G.counters()["handoffs"] == 0
    assert torch.equal(a, b)
    if algo == "weighted":
        ref, _ = oracle.walk_rjs(g, starts[:512], length, algo, seed=3, envelope="classes")
        assert np.array_equal(a[:512].cpu().numpy(), ref)
