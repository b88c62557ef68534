"""Small query batches (at most one query an SM: one launch, 1024 threads a
query) against Dijkstra, and batches of different sizes in turn on one handle,
whose work counters the last kernel of each batch leaves at zero."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
from paper_2412_18008_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 33, 151, 152, 153, 700, 1, 17_000, 5, 152]  # 152 SMs; 17,000 uses labels

GRAPHS = {
    "geo": I.geometric_knn_graph(20_003, seed=120),
    "grid": I.grid_graph(40, 40, 0.10, 1, 100, seed=121),
    "hub": I.star_graph(3000),
    "chain": I.chain_graph(2),
    "saturation": I.chain_graph(40, wmin=0x7FFFFFFF, wmax=0x7FFFFFFF),
    # searches that outgrow the shared table, finished by the dense kernel
    "overflow": I.random_digraph(9_000, 31_000, 1, 30, seed=122, allow_loops=False),
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_batches_of_all_sizes_in_turn(name):
    torch = pytest.importorskip("torch")
    from paper_2412_18008_gb300 import ch
    lib = ch.load()
    static = lib.ch_query_batch_static
    static.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_uint64, C.c_void_p, C.c_void_p]
    static.restype = C.c_int
    g = GRAPHS[name]
    gch = ch.CH.build(g, hop_limit=5)
    for j, k in enumerate(SIZES):
        s, t = I.random_pairs(g.n, k, seed=123 + j)
        check = slice(0, 200)
        want = O.dijkstra_pairs(g, s[check], t[check])
        assert np.array_equal(gch.query(s, t)[check], want), k
        ds, dt = (torch.from_numpy(x.view(np.int32)).cuda() for x in (s, t))
        out = torch.empty_like(ds)
        assert static(gch._h, ds.data_ptr(), dt.data_ptr(), k, out.data_ptr(), None) == 0
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().view(np.uint32)[check], want), k
        one = gch.query_one_to_many(int(s[0]), dt).cpu().numpy().view(np.uint32)[check]
        assert np.array_equal(one, O.dijkstra_pairs(g, np.full_like(s[check], s[0]), t[check])), k
    ds = torch.tensor([g.n, 0, 1], dtype=torch.int32).cuda()
    got = gch.query(ds, torch.zeros_like(ds)).cpu().numpy().view(np.uint32)
    with pytest.raises(ch.CHError) as ei:
        gch.query_status()
    assert ei.value.code == ch.CH_EINVAL
    assert got[0] == 0xFFFFFFFF and got[1] == 0
    assert got[2] == O.dijkstra_pairs(g, np.array([1], np.uint32), np.array([0], np.uint32))[0]
