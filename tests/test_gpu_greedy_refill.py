"""Greedy where the winner lies outside the candidate pool round after round: every sample holds one of the pool's vertices
and the next winner covers them all, so that the pool is empty of gain after each round and is filled again. Seeds,
coverage and estimates against the oracle's plain greedy."""
import numpy as np
import pytest

import oracle
import paper_1709_03565_gb300 as skis

pytestmark = pytest.mark.gpu

REL = 1e-12  # FP64 estimates of exact integers


@pytest.mark.parametrize("groups,leaves,T,k", [(3, 1100, 40_000, 8), (40, 300, 60_000, 60), (2, 5000, 30_000, 5)])
@pytest.mark.parametrize("ris", [False, True])
def test_refill_after_every_round(groups, leaves, T, k, ris):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    # a group: a hub with a live edge to each of its leaves (a leaf's sample is the leaf and the hub); the leaves' own
    # counts are close together, so a hub's round empties a pool of its leaves' gains
    per = leaves + 1
    n = groups * per
    hubs = np.arange(groups) * per
    src = np.repeat(hubs, leaves).astype(np.int32)
    dst = (np.repeat(hubs, leaves) + np.tile(np.arange(1, per), groups)).astype(np.int32)
    tau = np.full(len(src), 0xFFFFFFFF, np.uint32)
    tau[dst % 7 == 3] = 1 << 30  # some leaves are drawn less often
    g = skis.skis_load_graph(n, src, dst, tau, skis.SKIS_W_EXPLICIT_TAU)
    o = oracle.OracleGraph(n, src, dst, weights=tau, model=oracle.W_TAU)
    s = skis.skis_sketch_create(g, 0x9F)
    if ris:
        skis.skis_sketch_set_option(s, skis.SKIS_OPT_SAMPLER, 1)
    skis.skis_sample(s, T)
    sd, sc, se = skis.skis_greedy_maxcover(s, k)
    od, oc, oe = oracle.OracleSketch(o, 0x9F, T, ris=ris).greedy(k)
    assert np.array_equal(sd, od) and np.array_equal(sc, oc)
    np.testing.assert_allclose(se, oe, rtol=REL, atol=0)
    s.close()
    g.close()
