"""Greedy max-coverage where its argmax changes form: the candidate pool (1024 vertices) holding every vertex, running
out and being refilled, and too many ties for a pool (rounds by segments of 256 vertices). Seeds, cumulative coverage
and estimates against the oracle's plain greedy."""
import numpy as np
import pytest

import oracle
import paper_1709_03565_gb300 as skis
import synth

pytestmark = pytest.mark.gpu

REL = 1e-12  # FP64 estimates of exact integers


@pytest.mark.parametrize("ris", [False, True])
@pytest.mark.parametrize("n,m,T,k", [
    (40, 200, 3000, 40),        # every vertex chosen; fewer than a pool pays for
    (1000, 8000, 500, 1000),    # every vertex fits the pool; Delta runs out long before k
    (1025, 8000, 5000, 1025),   # one vertex outside the pool
    (5000, 40000, 200, 1500),   # few samples: thousands of ties at Delta 0 and 1
    (6000, 60000, 60000, 2500),  # refills
    (4200, 30000, 3000, 4096), (4200, 30000, 3000, 4097)  # results copied back together or one by one
])
def test_greedy_seeds_over_pool_refills_and_ties(n, m, T, k, ris):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, dst = synth.chunglu(n, m, 2.3, n)
    g = skis.skis_load_graph(n, src, dst, weight_model=skis.SKIS_W_WC)
    o = oracle.OracleGraph(n, src, dst, model=oracle.W_WC)
    seed = 0x6EED + T
    s = skis.skis_sketch_create(g, seed)
    if ris:
        skis.skis_sketch_set_option(s, skis.SKIS_OPT_SAMPLER, 1)
    skis.skis_sample(s, T)
    sd, sc, se = skis.skis_greedy_maxcover(s, k)
    od, oc, oe = oracle.OracleSketch(o, seed, T, ris=ris).greedy(k)
    assert np.array_equal(sd, od) and np.array_equal(sc, oc)
    np.testing.assert_allclose(se, oe, rtol=REL, atol=0)
    sd2, sc2, se2 = skis.skis_greedy_maxcover(s, k)  # nothing is left over from the first call
    assert np.array_equal(sd2, sd) and np.array_equal(sc2, sc) and np.array_equal(se2, se)
    s.close()
    g.close()
