"""Row offsets where four sorted destinations are read at a time: edge counts around multiples of four, empty rows at
both ends and between, one row holding all edges. Against the counts of the destinations (integers: equal)."""
import numpy as np
import pytest

import paper_1709_03565_gb300 as skis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 7, 8, 1023, 1024, 1025, 100_003])
@pytest.mark.parametrize("rows", ["first", "last", "middle", "spread"])
def test_offsets(m, rows):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 5001
    rng = np.random.default_rng(m)
    dst = {"first": np.zeros(m), "last": np.full(m, n - 1), "middle": rng.integers(2000, 2004, m),
           "spread": rng.integers(0, n, m)}[rows].astype(np.int32)
    src = ((dst + rng.integers(1, n, m)) % n).astype(np.int32)
    g = skis.skis_load_graph(n, src, dst, None, skis.SKIS_W_WC)
    want = np.concatenate([[0], np.cumsum(np.bincount(dst, minlength=n))])
    assert np.array_equal(skis.skis_graph_export(g)["off"], want)
    g.close()
