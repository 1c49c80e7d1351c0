"""One sketch sampled again after an option changed its slots: the samples that outgrow a slot's queue, before and after,
against the oracle (integers and sets: equal)."""
import numpy as np
import pytest

import oracle
import paper_1709_03565_gb300 as skis
from test_gpu_parity import assert_samples_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("changes", [
    ((skis.SKIS_OPT_CTA_SLOTS, 2), (skis.SKIS_OPT_CTA_SLOTS, 300)),
    ((skis.SKIS_OPT_CTA_THREADS, 512), (skis.SKIS_OPT_CTA_THREADS, 256)),
    ((skis.SKIS_OPT_CTA_QUEUE_CAP, 64), (skis.SKIS_OPT_CTA_SLOTS, 1))])
def test_outgrown_samples_after_the_slots_changed(changes):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 2000
    src, dst = np.arange(1, n, dtype=np.int32), np.zeros(n - 1, np.int32)  # every edge live: n members or two
    src, dst = np.concatenate([src, dst[:1]]), np.concatenate([dst, src[:1]])
    tau = np.full(n, 0xFFFFFFFF, np.uint32)
    g = skis.skis_load_graph(n, src, dst, tau, skis.SKIS_W_EXPLICIT_TAU)
    o = oracle.OracleGraph(n, src, dst, weights=tau, model=oracle.W_TAU)
    seed, per = 0x5107, 700
    s = skis.skis_sketch_create(g, seed)
    for k, v in ((skis.SKIS_OPT_THREAD_MAX_DEG, 0), (skis.SKIS_OPT_WARP_MAX_COINS, 1), (skis.SKIS_OPT_CTA_QUEUE_CAP, 32)):
        skis.skis_sketch_set_option(s, k, v)
    skis.skis_sample(s, per)
    for k, v in changes:
        skis.skis_sketch_set_option(s, k, v)
        skis.skis_sample(s, per)
    T = per * (1 + len(changes))
    ora = o.sample_ids(seed, np.arange(T, dtype=np.uint64))
    assert (ora["len"] > 64).sum() > T // 4
    assert_samples_equal(skis.skis_sketch_export(s, 0, T), ora)
    s.close()
    g.close()
