"""Hub labels take device memory only while there is plenty: a large batch on a
nearly full device is searched, and labels come back with the memory."""
import numpy as np
import pytest

from paper_2412_18008_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_labels_leave_the_device_its_memory():
    torch = pytest.importorskip("torch")
    from paper_2412_18008_gb300 import ch
    n = 1_000_000
    gch = ch.CH.build(I.chain_graph(n, seed=190), hop_limit=5)
    levels = gch.stats()["rounds"]
    s, t = I.random_pairs(n, 100_000, seed=191)
    ch.trim_memory()
    arena = 2 * n * 384 * 8
    before = torch.cuda.mem_get_info()[0]
    held = torch.empty(before - 2 * arena, dtype=torch.uint8, device="cuda")
    try:
        launches = ch.kernel_launches()
        searched = gch.query(s, t)
        assert ch.kernel_launches() - launches <= 3
        assert torch.cuda.mem_get_info()[0] > 3 * arena // 2
    finally:
        del held
        torch.cuda.empty_cache()
    launches = ch.kernel_launches()
    labels = gch.query(s, t)
    assert ch.kernel_launches() - launches > levels
    assert np.array_equal(labels, searched)
