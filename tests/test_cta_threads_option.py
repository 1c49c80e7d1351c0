"""SKIS_OPT_CTA_THREADS: a size that was asked for is the size of every CTA-tier block, with 1024 threads of them an SM;
without the option the library chooses by pass. On the host, with no GPU (fake_cuda)."""
import pytest

import fake_cuda
import paper_1709_03565_gb300 as skis


def _tier(s, count):
    first = len(s.launches())
    assert s.sample(count) == skis.SKIS_OK
    return [(grid, block) for name, grid, block in s.launches()[first:] if "k_iis_cta" in name]


@pytest.mark.parametrize("count", [100, 10_000, 1_000_000])
def test_block_sizes(count):
    s = fake_cuda.Sketch(5000)
    chosen = _tier(s, count)
    assert (1216, 128) in chosen
    s.option(skis.SKIS_OPT_CTA_THREADS, 256)
    assert _tier(s, count) == [(608, 256)]
    s.option(skis.SKIS_OPT_CTA_THREADS, 512)
    assert _tier(s, count) == [(304, 512)]
    s.option(skis.SKIS_OPT_CTA_THREADS, 256)
    s.option(skis.SKIS_OPT_CTA_SLOTS, 700)
    s.script((0, 0, 5))  # outgrown samples: the same blocks
    assert set(_tier(s, count)) == {(700, 256)}
    s.close()


def test_refused_sizes():
    s = fake_cuda.Sketch(100)
    for value in (0, 1, 64, 128, 1024):
        assert s.fk.skis_sketch_set_option(s.s, skis.SKIS_OPT_CTA_THREADS, value) == skis.SKIS_EINVAL
    s.close()
