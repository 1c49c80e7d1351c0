"""A sketch grown by further calls: its samples against the oracle (integers and sets: equal) when the arena grows ahead
of a call, when that was too little and the call takes several passes, and after a call whose surplus samples were
dropped, which must not count as members of the ones that were kept."""
import numpy as np
import pytest

import oracle
import paper_1709_03565_gb300 as skis
from test_gpu_parity import assert_samples_equal

pytestmark = pytest.mark.gpu


def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("lt", [False, True])
def test_second_call_of_several_passes(lt):
    _cuda()
    n = 20_000  # a path: the sample of source v has v + 1 members
    src, dst = np.arange(n - 1, dtype=np.int32), np.arange(1, n, dtype=np.int32)
    tau = np.full(n - 1, 0xFFFFFFFF, np.uint32)
    g = (skis.skis_load_graph_lt if lt else skis.skis_load_graph)(n, src, dst, tau, skis.SKIS_W_EXPLICIT_TAU)
    o = oracle.OracleGraph(n, src, dst, weights=tau, model=oracle.W_TAU, lt=lt)
    T, seed = 3000, next(x for x in range(1000) if o.sample_ids(x, np.arange(1, dtype=np.uint64))["len"][0] < 40)
    s = skis.skis_sketch_create(g, seed)
    skis.skis_sample(s, 1)  # a short one: what follows has 10,000 members a sample
    skis.skis_sample(s, T - 1)
    assert skis.skis_sketch_stats(s)["last_passes"] > 1
    skis.skis_sample(s, 500)
    ora = o.sample_ids(seed, np.arange(T + 500, dtype=np.uint64))
    assert_samples_equal(skis.skis_sketch_export(s, 0, T + 500), ora)
    assert skis.skis_sketch_stats(s)["entries"] == ora["len"].sum()
    s.close()
    g.close()


def test_samples_after_a_call_that_dropped_most_of_its_own():
    _cuda()
    n = 4000
    rng = np.random.default_rng(3)
    src, dst = rng.integers(0, n, 20_000).astype(np.int32), rng.integers(0, n, 20_000).astype(np.int32)
    src, dst = src[src != dst], dst[src != dst]
    g = skis.skis_load_graph(n, src, dst, weight_model=skis.SKIS_W_WC)
    o = oracle.OracleGraph(n, src, dst, model=oracle.W_WC)
    s = skis.skis_sketch_create(g, 0xD20)
    kept, _ = skis.skis_sample_to_size(s, 1, 60_000)
    assert kept == 1
    T = 1 + 20_000
    skis.skis_sample(s, T - 1)
    assert skis.skis_sketch_stats(s)["arena_capacity"] < 100_000_000  # 60,000 samples' room, and what 20,000 more have
    assert_samples_equal(skis.skis_sketch_export(s, 0, T), o.sample_ids(0xD20, np.arange(T, dtype=np.uint64)))
    s.close()
    g.close()
