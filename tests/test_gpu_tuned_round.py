"""Trials per round after tuning: a tuned result may say that the launch's own
rule is the fastest (batch=0), and one that names 2 trials means 2."""
import numpy as np
import pytest

from paper_2512_00705_gb300 import flexiwalk as fw
from paper_2512_00705_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,shown", [(0, 2), (2, 2), (5, 5)])
def test_a_cached_shape_is_installed(tmp_path, batch, shown):
    g = synth.workload_graph("small")
    G = fw.Graph(g)
    cache = str(tmp_path / "shape.txt")
    G.autotune("node2vec", p=0.5, q=2.0, method=2, cache_path=cache)
    line = open(cache).read().splitlines()[0]
    with open(cache, "w") as f:
        f.write(line.rsplit("r=", 1)[0] + "r=11 lane=16 batch=%d budget=0.5\n" % batch)
    assert G.autotune("node2vec", p=0.5, q=2.0, method=2, cache_path=cache) == pytest.approx(11.0)  # not in the sweep
    a = fw.ALGO["node2vec"]
    assert (G.info["lane_max_degrees"][a], G.info["rjs_batches"][a], G.info["trial_budgets"][a]) == (16, shown, 0.5)
    assert len(open(cache).read().splitlines()) == 1
    starts = torch.from_numpy(np.arange(g.n, dtype=np.int32)).cuda()
    x = G.walk(starts, 20, "node2vec", p=0.5, q=2.0, seed=4)
    y = G.walk(starts, 20, "node2vec", p=0.5, q=2.0, seed=4, cost_ratio=11.0, lane_max_degree=16, trial_budget=0.5,
               rjs_batch=batch)
    assert torch.equal(x, y)
    G.close()
