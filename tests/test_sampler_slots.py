"""The sampler's slots when options change between two calls on one sketch: no launch has more blocks than the slots that
are allocated (each block works in a slot of its own). On the host, with no GPU (fake_cuda)."""
import pytest

import fake_cuda
import paper_1709_03565_gb300 as skis

N = 100_000


def _check(s, first):
    """Grids of the CTA-tier launches from record `first` on against the slots' buffers; how many there were."""
    slots = s.value("cta_slots_alloc")
    assert s.bytes("bitmaps") >= slots * s.value("bitmap_words") * 4
    assert s.bytes("queues") >= slots * s.value("queue_cap") * 4
    assert s.bytes("slot_clean") >= slots * 4
    tier = [(name, grid) for name, grid, _ in s.launches()[first:] if "k_iis_cta" in name or "k_lt_long" in name]
    assert all(grid <= slots for _, grid in tier), (tier, slots)
    if s.value("big_slots"):
        assert s.value("big_slots") <= slots and s.bytes("big_queues") >= s.value("big_slots") * N * 4
    return len(tier)


@pytest.mark.parametrize("lt", [False, True])
@pytest.mark.parametrize("opt,value", [(skis.SKIS_OPT_CTA_SLOTS, 2), (skis.SKIS_OPT_CTA_SLOTS, 5000),
                                       (skis.SKIS_OPT_CTA_THREADS, 512), (skis.SKIS_OPT_CTA_QUEUE_CAP, 1 << 20)])
def test_the_pass_for_outgrown_samples_keeps_to_the_slots_there_are(lt, opt, value):
    s = fake_cuda.Sketch(N, lt=lt)
    s.option(skis.SKIS_OPT_CTA_QUEUE_CAP, 32)
    s.script((0, 1000, 20))  # 20 samples outgrow a slot
    assert s.sample(5000) == skis.SKIS_OK
    assert s.value("big_slots") > 0 and _check(s, 0) >= 2
    s.option(opt, value)
    first = len(s.launches())
    s.script((0, 1000, 20))
    assert s.sample(5000) == skis.SKIS_OK
    assert _check(s, first) >= 2
    s.close()
