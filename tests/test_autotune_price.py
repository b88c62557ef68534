"""ch_build_autotune prices a hierarchy's queries by what answers a batch of the
sample's size: hub labels above their line, searches below it."""
import pytest

from paper_2412_18008_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sample,labels", [(8_000, False), (20_000, True)])
def test_sample_is_answered_as_any_batch(sample, labels):
    from paper_2412_18008_gb300 import ch
    g = I.geometric_knn_graph(20_000, seed=195)

    def build():
        before = ch.kernel_launches()
        h = ch.CH.build(g, hop_limit=5)
        return h, ch.kernel_launches() - before

    build()[0].close()
    h, alone = build()
    rounds = h.stats()["rounds"]
    before = ch.kernel_launches()
    tuned, rows, _ = ch.CH.build_autotune(g, hop_limits=(5,), route_degs=(0,), sample=sample)
    more = ch.kernel_launches() - before - alone
    assert tuned.stats()["rounds"] == rounds and rows[0]["query_ms"] > 0
    assert (more > 2 * rounds) == labels and (labels or more <= 7)  # a warm-up and a timed batch
