"""A sampling call that could not grow the member arena, or failed past its first pass in another way, leaves the arena's
cursor where the samples end: the next call is not refused, nor grows the arena, for what the failed one had asked for.
On the host, with no GPU (fake_cuda)."""
import pytest

import fake_cuda
import paper_1709_03565_gb300 as skis


@pytest.mark.parametrize("lt", [False, True])
@pytest.mark.parametrize("before", [0, 1000])
def test_the_cursor_returns_to_the_samples_end(before, lt):
    s = fake_cuda.Sketch(5000, lt=lt, limit=16 << 30)
    used = 0
    if before:
        s.script((0, 7777, 0))
        assert s.sample(before) == skis.SKIS_OK
        used = 7777
    for _ in range(3):
        s.script(*[(900, 1 << 36, 0)] * 200)  # the samples of a pass would take 256 GiB, whatever the arena holds
        assert s.sample(1000) == skis.SKIS_ERR_ARENA_FULL
        assert s.value("T") == before
        assert s.fk.fk_cursor(s.s) == used
    s.script((0, 500, 0))
    assert s.sample(100) == skis.SKIS_OK
    assert s.value("T") == before + 100 and s.fk.fk_cursor(s.s) == used + 500
    s.close()


def test_after_the_pass_for_outgrown_samples_failed():
    s = fake_cuda.Sketch(1 << 20)
    s.option(skis.SKIS_OPT_CTA_QUEUE_CAP, 32)
    s.option(skis.SKIS_OPT_CTA_SLOTS, 4)
    assert s.sample(10) == skis.SKIS_OK
    s.script((0, 3000, 5))
    s.fk.fk_fail_at(1, 1)  # the n-entry queues
    assert s.sample(10) == skis.SKIS_ENOMEM
    s.fk.fk_fail_at(0, 0)
    assert s.fk.fk_cursor(s.s) == 0 and s.value("T") == 10
    s.script((0, 3000, 5))
    assert s.sample(10) == skis.SKIS_OK
    assert s.fk.fk_cursor(s.s) == 3000 and s.value("T") == 20
    s.close()
