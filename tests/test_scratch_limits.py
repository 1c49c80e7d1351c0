"""Sampling on a device without room for the whole of the default scratch: the call takes less instead of failing, down to
what a split of 608 CTA-tier slots within 8 GB and an arena of 8 members a sample need in all. On the host, with no GPU
(fake_cuda)."""
import pytest

import fake_cuda
import paper_1709_03565_gb300 as skis
from test_failed_allocations import sampler_buffers


def _plain(n, count, lt):
    """Bytes of that split, of the samples' headers and lists and of the members' counts."""
    per_slot = 4 * min(n, 1 << 20) + 4 * ((n + 31) // 32)
    slots = min(152 * (2 if lt else 4), max(1, (8 << 30) // per_slot))
    tables = 152 * 256 * (2048 + 1024 + 1024) * 4 if lt else 0
    return (28 + 64) * count + 4 * max(8 * count, 1 << 20) + slots * per_slot + tables + 4 * n + 4096


@pytest.mark.parametrize("lt", [False, True])
@pytest.mark.parametrize("n,count", [(3000, 100), (3000, 5_000_000), (1_000_000, 10_000_000), (1 << 25, 1_000_000),
                                     (1 << 28, 1000)])
def test_less_scratch_where_there_is_less_room(n, count, lt):
    s = fake_cuda.Sketch(n, lt=lt)
    s.fk.fk_start(s.fk.fk_used() + (280 << 30))
    at = s.fk.fk_used()
    assert s.sample(count) == skis.SKIS_OK and s.value("lean") == 0
    full = s.fk.fk_used() - at
    s.fk.skis_sketch_free(s.s)
    for room in sorted({_plain(n, count, lt), (full + _plain(n, count, lt)) // 2, full - 1, full}):
        if room > full:
            continue
        s.fk.fk_start(at + room)
        assert s.fk.skis_sketch_create(fake_cuda.ctypes.byref(s.s), s.g, 1, 0, None) == 0
        for more in (count, count // 3):  # the second within what is left of the first's room
            if more != count:
                s.fk.fk_start(at + room + 92 * more + (8 << 30))
            first = len(s.launches())
            assert s.sample(more) == skis.SKIS_OK, (room, full)
            assert (s.value("lean") == 0) == (room == full)
            sampler_buffers(s, more, lt, n, first)
        s.fk.skis_sketch_free(s.s)
    s.s = None
    s.close()


def test_a_call_that_never_fits_leaves_the_sketch_as_it_was():
    s = fake_cuda.Sketch(3000)
    assert s.sample(1 << 38) == skis.SKIS_ENOMEM
    assert s.value("lean") == 0
    assert s.sample(1000) == skis.SKIS_OK and s.value("lean") == 0
    sampler_buffers(s, 1000, False, 3000, 0)
    s.close()


def test_the_arena_grows_by_doubling_where_its_whole_demand_has_no_room():
    s = fake_cuda.Sketch(3000, limit=3 << 30)
    # 300M entries wanted at 1.125 of it and the chunks' ends, beside what is held: too much; 134M and then 268M fit
    s.fk.fk_start(s.fk.fk_used() + 1_900_000_000)
    s.script((900, 300_000_000, 0), (900, 300_000_000, 0), (0, 1000, 0))
    assert s.sample(1_000_000) == skis.SKIS_OK
    assert s.value("T") == 1_000_000
    s.close()
