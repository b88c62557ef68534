"""Builds whose witness searches change tiers from round to round, against the
oracle: phases that start at the warp tier (more than 64 sources an SM) or at the
middle block tier (128 or 512 threads a block), with the big tier behind it, left
out (hardly any source outgrew the middle one) or in its place (most did)."""
import functools

import numpy as np
import pytest

import oracle as O
from paper_2412_18008_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _union(a, b):
    (s0, t0, w0), (s1, t1, w1) = a.edges(), b.edges()
    return I.csr_from_edges(a.n + b.n, np.concatenate([s0, s1 + a.n]), np.concatenate([t0, t1 + a.n]),
                            np.concatenate([w0, w1]))


@functools.lru_cache(maxsize=None)
def _graph(name):
    if name == "near":  # warp tier, then ever fewer sources; no big balls until late
        return I.geometric_knn_graph(14_000, seed=200)
    wide = I.random_digraph(4_000, 14_000, 1, 1000, seed=201)
    if name == "wide_many":
        return I.random_digraph(12_000, 60_000, 1, 1000, seed=203)
    if name == "wide":  # most balls outgrow the middle tier
        return wide
    return _union(I.geometric_knn_graph(12_000, seed=202), wide)


MODES = {"plain": (dict(), dict()),
         "memo": (dict(witness_memo_limit=1 << 30), dict(memo=1 << 30)),
         "prune": (dict(witness_memo_limit=1 << 30, witness_prune=True), dict(memo=1 << 30, prune=True)),
         "level_work": (dict(witness_level_work=2_000), dict(level_work=2_000))}


@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("name", ["near", "wide", "wide_many", "both"])
def test_builds_that_change_tiers(name, mode):
    from paper_2412_18008_gb300 import ch
    from tests.test_gpu_parity import assert_same_hierarchy
    g = _graph(name)
    gpu, cpu = MODES[mode]
    och = O.build_ch(g, 5, cmax=64, threads=True, **cpu)
    with ch.CH.build(g, hop_limit=5, max_candidates_per_vertex=64, **gpu) as gch:
        assert_same_hierarchy(gch, och)
