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


def test_tables_by_what_the_searches_need():
    # six blocks an SM on 2^11-slot tables where the searches fit them, else three
    from paper_2412_18008_gb300 import ch
    near = ch.CH.build(I.geometric_knn_graph(30_000, seed=183), hop_limit=5)
    wide = ch.CH.build(I.random_digraph(9_000, 31_000, 1, 30, seed=184, allow_loops=False), hop_limit=5)
    blocks = []
    for gch in (near, wide):
        s, t = I.random_pairs(gch.stats()["n"], 2_000, seed=185)
        for _ in range(2):
            with ch.Server(gch, ring=4096, pool=1 << 14) as sv:
                blocks.append(sv.blocks)
                ans, _, _ = sv.replay(s, np.ones(s.size, np.uint32), t, np.zeros(s.size, np.uint64))
            assert np.array_equal(ans, gch.query(s, t))
    assert blocks[0] == blocks[1] == 2 * blocks[2] == 2 * blocks[3]


def test_fewer_blocks_when_memory_is_short():
    # device memory left for three blocks an SM but not for six
    torch = pytest.importorskip("torch")
    from paper_2412_18008_gb300 import ch
    gch = ch.CH.build(I.chain_graph(140_000, seed=186), hop_limit=5)
    s, t = I.random_pairs(140_000, 2_000, seed=187)
    want = gch.query(s, t)
    with ch.Server(gch, ring=4096, pool=1 << 14) as sv:
        blocks = sv.blocks
    scratch = blocks * 9 * (1 << 17) * 4
    ch.trim_memory()
    free = torch.cuda.mem_get_info()[0]
    held = torch.empty(free - scratch * 3 // 4, dtype=torch.uint8, device="cuda")
    try:
        with ch.Server(gch, ring=4096, pool=1 << 14) as sv:
            assert 2 * sv.blocks == blocks
            ans, _, _ = sv.replay(s, np.ones(s.size, np.uint32), t, np.zeros(s.size, np.uint64))
    finally:
        del held
        torch.cuda.empty_cache()
    assert np.array_equal(ans, want)
