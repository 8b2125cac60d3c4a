"""fw_walk_host_noalloc takes no queue counter from the graph's own pool, which
neither the device's free bytes nor the default pool's high-water mark would
show; other queued walks do."""
import ctypes

import numpy as np
import pytest

from paper_2512_00705_gb300 import flexiwalk as fw
from paper_2512_00705_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_noalloc_walk_takes_no_counter():
    lib = fw.lib()
    lib.fw_counter_allocation_count.restype = ctypes.c_uint64
    noalloc = lib.fw_walk_host_noalloc
    noalloc.restype = ctypes.c_int
    noalloc.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int32, ctypes.c_int32, ctypes.c_int32,
                        ctypes.POINTER(fw.fw_params), ctypes.c_uint64, ctypes.c_void_p, ctypes.c_void_p]
    stream = torch.cuda.current_stream().cuda_stream
    g = synth.workload_graph("small")
    G = fw.Graph(g)
    walkers, length = 400_000, 5  # more walkers than lanes: they come from a queue
    starts = synth.random_starts(g.n, walkers, seed=6)
    got = np.full((walkers, length + 1), -7, dtype=np.int32)
    for mode in ("auto", "exact", "rvs"):
        prm = fw.make_params(2.0, 0.5, mode=mode)
        before = lib.fw_counter_allocation_count()
        assert noalloc(G.handle, starts.ctypes.data, walkers, length, fw.ALGO["node2vec"], ctypes.byref(prm), 3,
                       got.ctypes.data, stream) == 0
        assert lib.fw_counter_allocation_count() == before
        want = G.walk(torch.from_numpy(starts).cuda(), length, "node2vec", p=2.0, q=0.5, mode=mode, seed=3)
        assert lib.fw_counter_allocation_count() == before + 1
        assert np.array_equal(got, want.cpu().numpy())
    G.close()
