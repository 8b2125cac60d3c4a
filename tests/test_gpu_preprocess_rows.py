"""Per-row preprocessing at the edges of its row-length classes (a warp, a
block of 8 warps, a block of 32; shared or global filter and counts), against
the oracle: exact walks read the filters and tables, rejection-sampled walks
the class- and label-ordered records."""
import numpy as np
import pytest

import oracle
from paper_2512_00705_gb300 import flexiwalk as fw
from paper_2512_00705_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _stars(hubs, seed):
    """Hub k is joined to the first hubs[k] leaves and leaf i to leaf i + 1: symmetric, sorted rows, h and labels mirrored."""
    nh, leaves = len(hubs), max(hubs)
    src = [np.full(d, k) for k, d in enumerate(hubs)] + [np.arange(leaves - 1) + nh]
    dst = [np.arange(d) + nh for d in hubs] + [np.arange(1, leaves) + nh]
    a, b = np.concatenate(src), np.concatenate(dst)
    rng = np.random.default_rng(seed)
    h = np.exp(rng.standard_normal(a.size)).astype(np.float32)
    lab = rng.integers(0, 5, a.size).astype(np.uint8)
    s, t = np.concatenate([a, b]), np.concatenate([b, a])
    order = np.lexsort((t, s))
    n = nh + leaves
    off = np.zeros(n + 1, np.int32)
    off[1:] = np.cumsum(np.bincount(s, minlength=n))
    return synth.Csr(off, t[order].astype(np.int32), np.concatenate([h, h])[order], np.concatenate([lab, lab])[order])


EDGES = [1, 8, 15, 16, 17, 31, 32, 33, 255, 256, 257, 511, 2047, 2048, 2049, 5003]


@pytest.fixture(scope="module", params=[EDGES, [102395, 17], [210001, 300]], ids=["edges", "filter", "counts"])
def stars(request):
    g = _stars(request.param, len(request.param))
    dev = [torch.from_numpy(x).cuda() for x in (g.offsets, g.cols, g.h, g.labels)]
    G = fw.Graph(offsets=dev[0], cols=dev[1], weights=dev[2], labels=dev[3])
    starts = np.concatenate([np.repeat(np.arange(len(request.param)), 40), np.arange(0, g.n, max(1, g.n // 400))])
    yield g, G, starts.astype(np.int32)
    G.close()


@pytest.mark.parametrize("flags", [0, fw.FLAG_NO_TABLE, fw.FLAG_NO_BLOOM])
def test_filters_and_tables_give_the_oracles_exact_walks(stars, flags):
    g, G, starts = stars
    length = 6 if g.n < 100000 else 3
    out = G.walk(torch.from_numpy(starts).cuda(), length, "node2vec", p=2.0, q=0.5, mode="exact", seed=1, flags=flags)
    ref, _ = oracle.walk(g, starts, length, "node2vec", 2.0, 0.5, seed=1)
    assert np.array_equal(out.cpu().numpy(), ref)


@pytest.mark.parametrize("algo,schema", [("weighted", None), ("metapath", [0, 1, 2, 3, 4])])
def test_ordered_records_give_the_oracles_rejection_walks(stars, algo, schema):
    g, G, starts = stars
    out = G.walk(torch.from_numpy(starts).cuda(), 6, algo, schema=schema, mode="rjs", rjs_cap=1 << 30, seed=2)
    ref, _ = oracle.walk_rjs(g, starts, 6, algo, 1.0, 1.0, schema, seed=2, envelope="classes")
    assert np.array_equal(out.cpu().numpy(), ref)


def test_statistics_and_symmetry(stars):
    g, G, _ = stars
    row = np.repeat(np.arange(g.n), g.degrees())
    stats = G.label_stats().cpu().numpy()
    top = np.zeros((g.n, 8), np.float32)
    np.maximum.at(top, (row, g.labels), g.h)
    total = np.zeros((g.n, 8))
    np.add.at(total, (row, g.labels), g.h.astype(np.float64))
    assert np.array_equal(stats[..., 0], top)
    # FP32 sums of positive terms, at most d / 32 + 5 additions deep
    depth = g.degrees()[:, None] / 32 + 6
    assert np.all(np.abs(stats[..., 1] - total) <= depth * 2.0 ** -24 * total)
    assert G.info["symmetric"] == 1
    for spoil in ("weight", "above", "below"):  # a weight unlike its mirror's; an entry without mirror, on either side
        off, cols, h = g.offsets.copy(), g.cols.copy(), g.h.copy()
        if spoil == "weight":
            h[-1] *= 2.0
        else:
            at = off[1] - 1 if spoil == "above" else off[g.n - 1]  # (hub 0, its last leaf); (last leaf, its first neighbour)
            v = 0 if spoil == "above" else g.n - 1
            cols, h = np.delete(cols, at), np.delete(h, at)
            off[v + 1:] -= 1
        H = fw.Graph(offsets=off, cols=cols, weights=h)
        assert H.info["symmetric"] == 0
        H.close()


@pytest.mark.parametrize("where", ["inside", "equal", "first pair", "range", "weight"])
def test_device_rows_are_checked(where):
    g = _stars([300, 2, 2049], 7)
    off, cols, h = g.offsets.copy(), g.cols.copy(), g.h.copy()
    s = off[2]  # the row of 2,049 entries
    if where == "inside":
        cols[s + 1000], cols[s + 1001] = cols[s + 1001], cols[s + 1000]
    elif where == "equal":
        cols[off[3] - 1] = cols[off[3] - 2]
    elif where == "first pair":
        cols[s + 1] = cols[s]
    elif where == "range":
        cols[off[3] - 1] = g.n
    else:
        h[s] = 0.0
    with pytest.raises(fw.FlexiWalkError) as err:
        fw.Graph(offsets=torch.from_numpy(off).cuda(), cols=torch.from_numpy(cols).cuda(), weights=torch.from_numpy(h).cuda())
    assert err.value.status == -2
