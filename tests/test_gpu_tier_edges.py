"""Samples whose sizes and shapes sit at the edges of the deeper sampling tiers: every edge is live, so a sample is its
source's ancestor set and its size is known. The warp tier keeps 256 members in shared memory and 1536 in all (4096 on
graphs of 24,576 vertices and more), batches 32 rows and joins 32 live edges at a time; the CTA tier holds 512 rows of
a level in shared memory. All against the
oracle, sample by sample (integers and sets: equal)."""
import numpy as np
import pytest

import oracle
import paper_1709_03565_gb300 as skis
from test_gpu_parity import assert_samples_equal

pytestmark = pytest.mark.gpu


def _star(n):  # one row of n - 1 in-edges
    return np.arange(1, n), np.zeros(n - 1)


def _path(n):  # n - 1 levels of one row each; sources at every depth, so samples of every size up to n
    return np.arange(1, n), np.arange(n - 1)


def _tree(n):  # levels of 1, 2, 4, ... rows of two edges
    i = np.arange(1, n)
    return i, (i - 1) // 2


def _broom(n):  # a level of (n - 1) / 2 rows of one edge each
    h = (n - 1) // 2
    mid = np.arange(1, h + 1)
    return np.concatenate([mid, mid + h]), np.concatenate([np.zeros(h), mid])


SHAPES = {"star": _star, "path": _path, "tree": _tree, "broom": _broom}
TIERS = {"default": {}, "warp": {skis.SKIS_OPT_THREAD_MAX_DEG: 0},
         "cta": {skis.SKIS_OPT_THREAD_MAX_DEG: 0, skis.SKIS_OPT_WARP_MAX_COINS: 1},
         "cta-hub": {skis.SKIS_OPT_THREAD_MAX_DEG: 0, skis.SKIS_OPT_WARP_MAX_COINS: 1, skis.SKIS_OPT_CTA_HUB_QUADS: 2,
                     skis.SKIS_OPT_CTA_THREADS: 512}}


@pytest.mark.parametrize("tier", sorted(TIERS))
@pytest.mark.parametrize("shape,size,n", [
    ("star", 33, 33), ("star", 257, 257), ("star", 258, 258), ("star", 1536, 1536), ("star", 1537, 1537),
    ("path", 300, 300), ("path", 1600, 1600), ("tree", 256, 256), ("tree", 1537, 1537), ("broom", 1027, 1027),
    ("broom", 2501, 2501), ("star", 1537, 24_575), ("star", 4096, 24_576), ("star", 4097, 24_576),
    ("broom", 4095, 24_576), ("broom", 4097, 24_576), ("path", 1700, 24_576)])
@pytest.mark.parametrize("bucket", [False, True])
def test_sizes_at_the_tiers_edges(shape, size, n, tier, bucket):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, dst = (np.ascontiguousarray(x, dtype=np.int32) for x in SHAPES[shape](size))
    tau = np.full(len(src), 0xFFFFFFFF, np.uint32)
    g = skis.skis_load_graph(n, src, dst, tau, skis.SKIS_W_EXPLICIT_TAU)
    o = oracle.OracleGraph(n, src, dst, weights=tau, model=oracle.W_TAU)
    T, seed = 2000, 0xED6E + size
    s = skis.skis_sketch_create(g, seed)
    skis.skis_sketch_set_option(s, skis.SKIS_OPT_FIRST_STEP, 1 if bucket else 0)
    for k, v in TIERS[tier].items():
        skis.skis_sketch_set_option(s, k, v)
    skis.skis_sample(s, T)
    ora = o.sample_ids(seed, np.arange(T, dtype=np.uint64), bucket=bucket)
    assert shape not in ("star", "path") or ora["len"].max() >= size - 4  # a sample of (nearly) everything is among them
    assert_samples_equal(skis.skis_sketch_export(s, 0, T), ora)
    s.close()
    g.close()


# the CTA tier's block size goes by the samples of the pass and of the tier: 24 and 96 an SM are the lines
@pytest.mark.parametrize("per_sm,more", [(1, -1), (24, 0), (24, 1), (96, 0), (96, 1), (130, 0)])
@pytest.mark.parametrize("hub_quads", [2, 0])
def test_cta_block_sizes(per_sm, more, hub_quads):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 700
    rng = np.random.default_rng(5)
    src = np.concatenate([rng.integers(1, n, 3000), np.arange(1, n)]).astype(np.int32)
    dst = np.concatenate([rng.integers(1, n, 3000), np.zeros(n - 1)]).astype(np.int32)
    keep = src != dst
    src, dst = src[keep], dst[keep]
    tau = rng.integers(1 << 28, 1 << 31, len(src)).astype(np.uint32)
    g = skis.skis_load_graph(n, src, dst, tau, skis.SKIS_W_EXPLICIT_TAU)
    o = oracle.OracleGraph(n, src, dst, weights=tau, model=oracle.W_TAU)
    T, seed = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more, 0xB10C
    s = skis.skis_sketch_create(g, seed)
    for k, v in ((skis.SKIS_OPT_THREAD_MAX_DEG, 0), (skis.SKIS_OPT_WARP_MAX_COINS, 1),
                 (skis.SKIS_OPT_CTA_HUB_QUADS, hub_quads)):
        skis.skis_sketch_set_option(s, k, v)
    skis.skis_sample(s, T)
    assert_samples_equal(skis.skis_sketch_export(s, 0, T), o.sample_ids(seed, np.arange(T, dtype=np.uint64)))
    s.close()
    g.close()
