"""Large query batches, which are answered through hub labels: against
Dijkstra and against the same pairs in batches small enough to be searched."""
import numpy as np
import pytest

import oracle as O
from paper_2412_18008_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LARGE = 1 << 14  # the smallest batch that uses labels (above 80 sqrt(n) for these sizes)


def _ch():
    from paper_2412_18008_gb300 import ch
    return ch


def _searched(gch, s, t):
    return np.concatenate([gch.query(s[i:i + 9000], t[i:i + 9000]) for i in range(0, s.size, 9000)])


def _chain_to_infinity():
    # distances reach 2^32 - 1 after two links: saturated sums are INF
    return I.chain_graph(40, wmin=0x7FFFFFFF, wmax=0x7FFFFFFF)


GRAPHS = {
    # name: (graph, the labels' case)
    "geo_few": I.geometric_knn_graph(30_011, seed=110),           # endpoints below the labelled vertices
    "geo_many": I.geometric_knn_graph(1_500, seed=111),           # more queries than vertices: every endpoint labelled
    "two_vertices": I.chain_graph(2),
    "saturation": _chain_to_infinity(),
    "unreachable": I.random_digraph(6_000, 7_000, 1, 30, seed=112),
    "wide_labels": I.random_digraph(2_500, 7_500, 1, 30, seed=113),     # labels outgrow a warp's table
    "too_wide": I.random_digraph(9_000, 31_000, 1, 30, seed=114, allow_loops=False),  # and a block's
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_label_batches_match_searches(name):
    ch, g = _ch(), GRAPHS[name]
    gch = ch.CH.build(g, hop_limit=5)
    for k, seed in ((LARGE, 115), (LARGE + 4_321, 116)):
        s, t = I.random_pairs(g.n, k, seed=seed)
        t[:50] = s[:50]
        d = gch.query(s, t)
        gch.query_status()
        assert np.array_equal(d, _searched(gch, s, t))
        assert np.array_equal(d[:300], O.dijkstra_pairs(g, s[:300], t[:300]))


def test_labels_count_their_work():
    # (that the labels, not the searches, answered a batch)
    ch, g = _ch(), GRAPHS["geo_many"]
    gch = ch.CH.build(g, hop_limit=5)
    s, t = I.random_pairs(g.n, LARGE, seed=117)
    gch.query_work()
    gch.query(s, t)
    assert gch.query_work()[0] <= 2 * g.n  # each vertex's two labels once


def test_label_batch_options(tmp_path):
    torch = pytest.importorskip("torch")
    ch, g = _ch(), GRAPHS["geo_few"]
    gch = ch.CH.build(g, hop_limit=5, composite=True)
    k = LARGE
    s, t = I.random_pairs(g.n, k, seed=118)
    want = _searched(gch, s, t)
    ds, dt = (torch.from_numpy(x.view(np.int32)).cuda() for x in (s, t))
    # one source; a captured batch, replayed on new inputs; a loaded hierarchy
    one = gch.query_one_to_many(int(s[0]), dt).cpu().numpy().view(np.uint32)
    assert np.array_equal(one, _searched(gch, np.full_like(s, s[0]), t))
    out = torch.empty_like(ds)
    with gch.query_graph(ds, dt, out) as qg:
        for _ in range(2):
            qg.launch()
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy().view(np.uint32), want)
            ds, dt = ds.copy_(ds.flip(0)), dt.copy_(dt.flip(0))
            want = want[::-1]
    path = str(tmp_path / "h.bin")
    gch.save(path)
    loaded = ch.CH.load(path)
    assert np.array_equal(loaded.query(s, t), gch.query(s, t))
    # ids out of range
    s2 = s.copy()
    s2[7] = g.n
    got = gch.query(torch.from_numpy(s2.view(np.int32)).cuda(), torch.from_numpy(t.view(np.int32)).cuda())
    with pytest.raises(ch.CHError) as ei:
        gch.query_status()
    assert ei.value.code == ch.CH_EINVAL
    got = got.cpu().numpy().view(np.uint32)
    keep = np.arange(k) != 7
    assert got[7] == 0xFFFFFFFF and np.array_equal(got[keep], _searched(gch, s, t)[keep])
