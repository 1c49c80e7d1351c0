"""How far a sketch's member arena grows ahead of a further call: by the members its samples have had, as far as the
reserved entries tell (a warp leaves the end of its chunk unused). On the host, with no GPU (fake_cuda)."""
import pytest

import fake_cuda
import paper_1709_03565_gb300 as skis

GIB = 1 << 28  # arena entries of a GiB


# (samples, entries reserved) of the calls before: a few members a sample, and all that the warps can leave unused (512
# entries a warp of the first tier, 2048 one of the second, a warp for every sample up to 8 a block)
@pytest.mark.parametrize("lt,calls", [
    (False, [(1, 2560)]), (False, [(1, 2560)] * 20), (False, [(3, 7690), (100, 209_000)]), (False, [(5000, 10_060_000)]),
    (True, [(1, 514)]), (True, [(1, 514)] * 20), (True, [(3, 1550), (100, 4300)]), (True, [(5000, 90_000)])])
def test_unused_chunk_ends_are_not_taken_for_members(calls, lt):
    s = fake_cuda.Sketch(1000, lt=lt)
    for count, reserved in calls:
        s.script((0, reserved, 0))
        assert s.sample(count) == skis.SKIS_OK
    s.script((0, 1000, 0))
    assert s.sample(10_000_000) == skis.SKIS_OK
    assert s.value("arena_cap") <= 2.2 * GIB  # the room a first call of this size takes, and what was there
    s.close()


@pytest.mark.parametrize("members,low,high", [(4, 4e7, 22e7), (75, 75e7, 105e7), (2000, 2e10, 2.6e10)])
def test_known_sizes_are_grown_for(members, low, high):
    reserved = members * 1_000_000 + 6_000_000  # fewer unused than the warps can leave
    s = fake_cuda.Sketch(1000, limit=300 << 30, arena=reserved)
    s.script((0, reserved, 0))
    assert s.sample(1_000_000) == skis.SKIS_OK and s.value("arena_cap") == reserved
    s.script((0, 1000, 0))
    assert s.sample(10_000_000) == skis.SKIS_OK
    assert low <= s.value("arena_cap") <= high
    s.close()


def test_growth_beyond_any_memory_is_left_to_the_pass():
    s = fake_cuda.Sketch(1000, limit=40 << 30)
    s.script((0, 90_000_000, 0))
    assert s.sample(10) == skis.SKIS_OK  # 9 million members a sample (or so it seems)
    cap = s.value("arena_cap")
    s.script((0, 1000, 0))
    assert s.sample(200_000) == skis.SKIS_OK
    assert s.value("arena_cap") >= cap
    s.close()
