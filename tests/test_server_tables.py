"""How the query server shares out its work: the targets of a request go to
different blocks while pairs take long."""
import numpy as np
import pytest

from paper_2412_18008_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_targets_of_a_request_are_not_served_one_after_another():
    # 32 blocks, pairs of tens of microseconds, everything due at once: the 32
    # targets of a request start as blocks free up, within about a pair's time,
    # so their request takes about two pairs' time; with four positions at a time
    # for a block it would be about five
    from paper_2412_18008_gb300 import ch
    g = I.geometric_knn_graph(30_000, seed=180)
    gch = ch.CH.build(g, hop_limit=5)
    ks = np.array([1, 32] * 200, np.uint32)
    src, _ = I.random_pairs(g.n, ks.size, seed=181)
    targets, _ = I.random_pairs(g.n, int(ks.sum()), seed=182)
    with ch.Server(gch, blocks=32, ring=1024, pool=1 << 14) as sv:
        for _ in range(2):
            ans, _, svc = sv.replay(src, ks, targets, np.zeros(src.size, np.uint64))
    one, many = np.median(svc[0::2]), np.median(svc[1::2])
    assert many <= 3.2 * one, (one, many)
    assert np.array_equal(ans, gch.query(np.repeat(src, ks), targets))
