"""The first use of every launch variant may be inside a stream capture: a
plan in a process that has launched no walk yet gives the rows of fw_walk."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
import torch
from paper_2512_00705_gb300 import flexiwalk as fw
from paper_2512_00705_gb300 import synth

algo, mode, ratio, weights, walkers = sys.argv[1], sys.argv[2], float(sys.argv[3]), sys.argv[4], int(sys.argv[5])
njobs = int(sys.argv[6])
g = synth.workload_graph("small")
if weights == "pareto":
    g.h = synth.edge_weights(g, "pareto", 1.0, seed=7)
G = fw.Graph(g)
starts = torch.from_numpy(synth.random_starts(g.n, walkers, seed=3)).cuda()
kw = dict(p=0.5, q=2.0, mode=mode, cost_ratio=ratio, schema=[0, 1, 2] if algo == "metapath" else None)
outs = [torch.full((walkers, 4), -7, dtype=torch.int32, device="cuda") for _ in range(njobs)]
torch.cuda.synchronize()
plan = fw.BatchPlan(G, [fw.make_job(starts, 3, algo, o, seed=j, **kw) for j, o in enumerate(outs)])
plan.launch()
torch.cuda.synchronize()
for j, o in enumerate(outs):
    assert torch.equal(o, G.walk(starts, 3, algo, seed=j, **kw)), j
print("same rows")
"""


@pytest.mark.parametrize("algo,mode,ratio,weights,walkers", [
    ("node2vec", "auto", 0.5, "uniform", 200_000),    # queued, short eRVS rows scanned at once
    ("node2vec", "auto", 4.0, "uniform", 200_000),    # queued
    ("weighted", "auto", 4.0, "pareto", 200_000),     # queued, trials together
    ("pagerank2", "auto", 4.0, "uniform", 500),       # spread, trials together
    ("metapath", "rvs", 4.0, "uniform", 5_000),       # eRVS only
    ("weighted", "exact", 4.0, "uniform", 5_000)])    # exact only
@pytest.mark.parametrize("njobs", [1, 2])
def test_a_plan_before_any_walk(algo, mode, ratio, weights, walkers, njobs):
    r = subprocess.run([sys.executable, "-c", CHILD, algo, mode, str(ratio), weights, str(walkers), str(njobs)], cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.strip() == "same rows"
