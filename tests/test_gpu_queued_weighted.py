"""Queued weighted walks by blocks per SM: the rows do not depend on the
variant, on either side of each of its rule's lines."""
import pytest

from paper_2512_00705_gb300 import flexiwalk as fw
from paper_2512_00705_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MOST = 400_000


@pytest.fixture(scope="module")
def graph():
    g = synth.rmat(20, 16)  # 31 M entries: records well beyond L2
    g.h = synth.edge_weights(g, "uniform01", seed=2)
    G = fw.Graph(g)
    starts = torch.from_numpy(synth.random_starts(g.n, MOST, seed=4)).cuda()
    yield G, starts
    G.close()


@pytest.mark.parametrize("walkers", [155_649, 194_560, 194_561, 300_000, MOST])  # turns of 4 and of 5 blocks per SM
@pytest.mark.parametrize("length", [15, 16])
@pytest.mark.parametrize("mode,flags", [("auto", 0), ("rjs", 0), ("auto", fw.FLAG_UNWEIGHTED)])
def test_rows_of_queued_weighted_walks(graph, walkers, length, mode, flags):
    G, starts = graph
    a = G.walk(starts[:walkers], length, "weighted", mode=mode, flags=flags, seed=6)
    b = G.walk(starts[:walkers], length, "weighted", mode=mode, flags=flags | fw.FLAG_COUNTERS, seed=6)
    assert torch.equal(a, b)


def test_rows_of_a_batch(graph):
    G, starts = graph
    jobs, outs = [], []
    for j, (w, length) in enumerate([(160_000, 20), (900, 7), (220_000, 40)]):
        out = torch.full((w, length + 1), -7, dtype=torch.int32, device="cuda")
        jobs.append(fw.make_job(starts[:w], length, ["weighted", "node2vec", "node2vec"][j], out, p=1.0, q=1.0, seed=j))
        outs.append((out, w, length))
    fw.fw_walk_batch(G.handle, jobs)
    for j, (out, w, length) in enumerate(outs):
        ref = G.walk(starts[:w], length, ["weighted", "node2vec", "node2vec"][j], p=1.0, q=1.0, seed=j, flags=fw.FLAG_COUNTERS)
        assert torch.equal(out, ref)
