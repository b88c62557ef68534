"""Which batches are answered through hub labels: deep hierarchies (many levels
for their size) are searched until a batch is large enough to pay for the levels'
merges; above that line their labels outgrow the warps' tables and, for the wider
one, the blocks' too, and queries without labels go through both table sizes of
the searches."""
import numpy as np
import pytest

import oracle as O
from paper_2412_18008_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _launches(ch, gch, s, t):
    before = ch.kernel_launches()
    d = gch.query(s, t)
    return d, ch.kernel_launches() - before


@pytest.mark.parametrize("n,m,seed,small", [(2_500, 7_500, 113, 1), (9_000, 31_000, 114, 1), (9_000, 31_000, 114, 0)])
def test_deep_hierarchies(n, m, seed, small):
    from paper_2412_18008_gb300 import ch
    g = I.random_digraph(n, m, 1, 30, seed=seed, allow_loops=False)
    gch = ch.CH.build(g, hop_limit=5)
    gch.set_query_config(1, 256, small, 1, 50)
    levels = gch.stats()["rounds"]
    assert 224 * levels > 17_000
    k = 224 * levels
    s, t = I.random_pairs(g.n, k, seed=170)
    below, calls = _launches(ch, gch, s[:17_000], t[:17_000])
    assert calls <= 3  # two table sizes and the dense kernel
    just_below, calls = _launches(ch, gch, s[:-1], t[:-1])
    assert calls <= 3
    labels, calls = _launches(ch, gch, s, t)
    assert calls > levels
    gch.query_status()
    assert np.array_equal(labels[:-1], just_below) and np.array_equal(labels[:17_000], below)
    assert np.array_equal(labels[-300:], O.dijkstra_pairs(g, s[-300:], t[-300:]))
