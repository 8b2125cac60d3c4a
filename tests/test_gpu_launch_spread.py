"""Launch shapes: few walkers are spread over the resident warps (no queue),
more walkers than lanes come from the queue; the rows are the same."""
import numpy as np
import pytest

import oracle
from paper_2512_00705_gb300 import flexiwalk as fw
from paper_2512_00705_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LEN = 3


@pytest.fixture(scope="module")
def walks():
    g = synth.workload_graph("small")
    G = fw.Graph(g)
    lanes = torch.cuda.get_device_properties(0).multi_processor_count * 4 * 256  # 4 resident blocks of 256 threads
    most = lanes + 33
    starts = synth.random_starts(g.n, most, seed=5)
    yield g, G, lanes, starts
    G.close()


@pytest.mark.parametrize("where", ["one", "block", "warps", "warps+1", "half", "lanes-1", "lanes", "lanes+1", "lanes+33"])
@pytest.mark.parametrize("mode", ["exact", "rvs"])
def test_rows_do_not_depend_on_the_launch_shape(walks, where, mode):
    g, G, lanes, starts = walks
    w = {"one": 1, "block": 31, "warps": lanes // 32, "warps+1": lanes // 32 + 1, "half": lanes // 2 + 7,
         "lanes-1": lanes - 1, "lanes": lanes, "lanes+1": lanes + 1, "lanes+33": lanes + 33}[where]
    dev = torch.from_numpy(starts[:w]).cuda()
    out = G.walk(dev, LEN, "node2vec", p=2.0, q=0.5, mode=mode, seed=9).cpu().numpy()
    if mode == "exact":
        ref, _ = oracle.walk(g, starts[:w], LEN, "node2vec", 2.0, 0.5, seed=9)
    else:  # the counting build takes its walkers from the queue at every size
        ref = G.walk(dev, LEN, "node2vec", p=2.0, q=0.5, mode=mode, seed=9, flags=fw.FLAG_COUNTERS).cpu().numpy()
    assert np.array_equal(out, ref)
    G.check()


def test_small_batch_spreads_each_job(walks):
    g, G, lanes, starts = walks
    jobs, outs = [], []
    for j, w in enumerate([1, 63, 700, 5]):
        dev = torch.from_numpy(starts[:w]).cuda()
        out = torch.full((w, LEN + 1), -7, dtype=torch.int32, device="cuda")
        jobs.append(fw.make_job(dev, LEN, "node2vec", out, p=2.0, q=0.5, mode="exact", seed=j))
        outs.append((w, out, dev))
    fw.fw_walk_batch(G.handle, jobs)
    for j, (w, out, _) in enumerate(outs):
        ref, _ = oracle.walk(g, starts[:w], LEN, "node2vec", 2.0, 0.5, seed=j)
        assert np.array_equal(out.cpu().numpy(), ref)


@pytest.mark.parametrize("p,q", [(2.0, 0.5), (0.25, 4.0), (1.0, 4.0)])
@pytest.mark.parametrize("mode,flags,shape", [("rvs", 0, {}), ("rvs", 0, {"lane_max_degree": 64, "rjs_batch": 3}),
                                              ("rvs", fw.FLAG_RVS_NOJUMP, {"lane_max_degree": 33}),
                                              ("rvs", 0, {"lane_max_degree": 1}), ("rvs", fw.FLAG_RVS_NOJUMP, {}),
                                              ("rvs", fw.FLAG_UNWEIGHTED, {"lane_max_degree": 1}),
                                              ("auto", 0, {"cost_ratio": 8.0}),
                                              ("rjs", 0, {"rjs_cap": 1, "lane_max_degree": 40})])
@pytest.mark.parametrize("quantized", [False, True])
def test_lane_scans_in_step_with_trials_equal_whole_lane_scans(p, q, mode, flags, shape, quantized):
    """node2vec's short eRVS rows: scanned one position per trial round by the
    queued kernel (which the counting build is), at once by the spread one."""
    g = synth.workload_graph("small")
    G = fw.Graph(g)
    if quantized:
        G.quantize_weights()
    starts = torch.arange(g.n, dtype=torch.int32, device="cuda")
    a = G.walk(starts, 20, "node2vec", p=p, q=q, mode=mode, seed=3, flags=flags, **shape)
    b = G.walk(starts, 20, "node2vec", p=p, q=q, mode=mode, seed=3, flags=flags | fw.FLAG_COUNTERS, **shape)
    assert torch.equal(a, b)
    assert G.counters()["rvs_steps"] > 0
    G.close()


@pytest.fixture(scope="module")
def skewed():
    g = synth.workload_graph("small")
    g.h = synth.edge_weights(g, "pareto", 1.0, seed=7)
    G = fw.Graph(g)
    yield g, G
    G.close()


@pytest.mark.parametrize("algo,p,q", [("weighted", 1.0, 1.0), ("node2vec", 2.0, 0.5), ("node2vec", 0.25, 4.0),
                                      ("metapath", 1.0, 1.0), ("pagerank2", 1.0, 1.0)])
@pytest.mark.parametrize("mode,shape", [("auto", {}), ("rjs", {"rjs_cap": 61}), ("rjs", {"rjs_cap": 9, "rjs_batch": 4}),
                                        ("rjs", {"rjs_cap": 1 << 30})])
@pytest.mark.parametrize("walkers,length", [(4099, 12), (155700, 2)])
def test_trials_together_equal_a_lanes_own(skewed, algo, p, q, mode, shape, walkers, length):
    """Heavy-tailed weights: steps of many failed trials are tried by the whole
    warp, except in the counting build."""
    g, G = skewed
    starts = torch.from_numpy(synth.random_starts(g.n, walkers, seed=11)).cuda()
    schema = [0, 1, 2] if algo == "metapath" else None
    a = G.walk(starts, length, algo, p=p, q=q, schema=schema, mode=mode, seed=3, **shape)
    b = G.walk(starts, length, algo, p=p, q=q, schema=schema, mode=mode, seed=3, flags=fw.FLAG_COUNTERS, **shape)
    assert torch.equal(a, b)


@pytest.mark.parametrize("mode", ["rvs", "exact"])
def test_scanning_jobs_queue_behind_one_walker_per_warp(walks, mode):
    g, G, lanes, starts = walks
    w = lanes // 32 * 3 + 5
    dev = torch.from_numpy(starts[:w]).cuda()
    a = G.walk(dev, 6, "node2vec", p=2.0, q=0.5, mode=mode, seed=9)
    b = G.walk(dev, 6, "node2vec", p=2.0, q=0.5, mode=mode, seed=9, flags=fw.FLAG_COUNTERS)
    assert torch.equal(a, b)


@pytest.mark.parametrize("mode,shape", [("auto", {"cost_ratio": 0.5}), ("rjs", {"rjs_cap": 3}), ("auto", {"cost_ratio": 1.5})])
@pytest.mark.parametrize("p,q", [(2.0, 0.5), (0.25, 4.0)])
def test_whole_scans_of_rare_reservoir_steps(walks, mode, shape, p, q):
    """node2vec queues with a small cost ratio scan short rows at once, the counting build one position per trial."""
    g, G, lanes, starts = walks
    dev = torch.from_numpy(starts).cuda()
    a = G.walk(dev, 4, "node2vec", p=p, q=q, mode=mode, seed=5, **shape)
    b = G.walk(dev, 4, "node2vec", p=p, q=q, mode=mode, seed=5, flags=fw.FLAG_COUNTERS, **shape)
    assert torch.equal(a, b)
