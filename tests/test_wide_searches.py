"""Hierarchies without a core whose searches outgrow the 2^11-slot tables, and
for many pairs the 2^12-slot ones: every level may be the one that overflows,
while the block's other warps are still at its top."""
import numpy as np
import pytest

import oracle as O
from paper_2412_18008_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _ch():
    from paper_2412_18008_gb300 import ch
    return ch


@pytest.fixture(scope="module", params=["some_2_11", "all_2_11", "some_2_12"])
def wide(request):
    n, m, seed = {"some_2_11": (2_600, 8_000, 150), "all_2_11": (5_000, 17_000, 151),
                  "some_2_12": (9_000, 31_000, 152)}[request.param]
    g = I.random_digraph(n, m, 1, 30, seed=seed, allow_loops=False)
    s, t = I.random_pairs(g.n, 3_000, seed=153)
    return _ch().CH.build(g, hop_limit=5), s, t, O.dijkstra_pairs(g, s, t)


@pytest.mark.parametrize("cfg", [(lay, thr, 1, 0, 0) for lay in (0, 1) for thr in (128, 256)]
                         + [(1, 256, 1, 1, 0), (1, 128, 1, 1, 40), (1, 256, 1, 1, 40), (1, 256, 0, 1, 1 << 20)])
def test_batches(wide, cfg):
    gch, s, t, want = wide
    default = gch.query_config()
    gch.set_query_config(*cfg)
    for _ in range(3):  # persistent blocks go on to other queries after an overflow
        assert np.array_equal(gch.query(s, t), want)
    assert np.array_equal(gch.query(s, t, want_settled=True)[0], want)
    assert np.array_equal(gch.query(s[:100], t[:100]), want[:100])  # a block of 1024 threads a query
    gch.set_query_config(*default)


@pytest.mark.parametrize("blocks", [0, 5])
def test_server(wide, blocks):
    gch, s, t, want = wide
    ks = np.ones(s.size, np.uint32)
    with _ch().Server(gch, blocks=blocks, ring=1024, pool=1 << 14) as sv:
        for _ in range(3):
            ans, _, _ = sv.replay(s, ks, t, np.zeros(s.size, np.uint64))
            assert np.array_equal(ans, want)
