"""A query batch does not depend on how the one before it ended: replays of
captured batches that stop before their last kernel (as a call does that fails
between its launches) are followed by whole batches on the same handle and on
the static scratch."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
from paper_2412_18008_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _drop_last_node(torch, graph):
    """Removes the graph's last node (the one without dependents)."""
    cu = C.CDLL("libcuda.so.1")
    raw = C.c_void_p(graph.raw_cuda_graph())
    count = C.c_size_t()
    assert cu.cuGraphGetNodes(raw, None, C.byref(count)) == 0
    nodes = (C.c_void_p * count.value)()
    assert cu.cuGraphGetNodes(raw, nodes, C.byref(count)) == 0
    ends = []
    for v in nodes:
        deps = C.c_size_t()
        assert cu.cuGraphNodeGetDependentNodes_v2(C.c_void_p(v), None, None, C.byref(deps)) == 0
        if deps.value == 0:
            ends.append(v)
    assert len(ends) == 1 and count.value >= 2
    assert cu.cuGraphDestroyNode(C.c_void_p(ends[0])) == 0


@pytest.mark.parametrize("name", ["geo", "wide", "core"])
@pytest.mark.parametrize("k", [7, 1000, 17_000])
def test_a_batch_after_an_unfinished_one(name, k):
    torch = pytest.importorskip("torch")
    from paper_2412_18008_gb300 import ch
    static = ch.load().ch_query_batch_static
    static.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_uint64, C.c_void_p, C.c_void_p]
    static.restype = C.c_int
    if name == "core":  # above 2048 core vertices: every query goes to the dense kernel
        g = I.random_digraph(6_000, 30_000, 1, 30, seed=160)
        gch = ch.CH.build(g, hop_limit=5, max_candidates_per_vertex=8)
        assert gch.stats()["core_vertices"] > 2048
    else:
        g = (I.geometric_knn_graph(20_003, seed=161) if name == "geo"
             else I.random_digraph(9_000, 31_000, 1, 30, seed=162, allow_loops=False))
        gch = ch.CH.build(g, hop_limit=5)
    s, t = I.random_pairs(g.n, k, seed=163)
    ds, dt = (torch.from_numpy(x.view(np.int32)).cuda() for x in (s, t))
    out = torch.empty_like(ds)

    def batch():
        stream = torch.cuda.current_stream().cuda_stream
        gch.query_batch_raw(ds.data_ptr(), dt.data_ptr(), k, out.data_ptr(), None, stream)

    def batch_static():
        stream = torch.cuda.current_stream().cuda_stream
        assert static(gch._h, ds.data_ptr(), dt.data_ptr(), k, out.data_ptr(), stream) == 0

    check = slice(0, 100)
    want = O.dijkstra_pairs(g, s[check], t[check])
    for call in (batch, batch_static):
        call()  # (whatever the first call allocates or resolves)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph):
            call()
        _drop_last_node(torch, graph)
        graph.instantiate()
        for _ in range(2):
            graph.replay()
            torch.cuda.synchronize()
            out.fill_(-2)
            call()
            torch.cuda.synchronize()
            got = out.cpu().numpy().view(np.uint32)
            assert np.array_equal(got[check], want) and not (got == 0xFFFFFFFE).any()
    gch.query_status()
