"""Coverage by the scan of a sketch in sample order: tasks of 32 to 1024 samples (by the members of a sample), ends
that are not a whole task, scans in which every member is a seed (more hits than a warp holds back, and more than the
list of 2^22), and the exact and the hashed seed filter. Against the counts of the exported samples (integers: equal)."""
import numpy as np
import pytest

import paper_1709_03565_gb300 as skis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth,T", [(3, 31), (3, 1025), (3, 200_001), (70, 1), (70, 63), (70, 65), (70, 150_000),
                                     (2100, 33), (2100, 1000)])
@pytest.mark.parametrize("n", [2100, (1 << 20) + 64])
def test_scan_counts(depth, T, n):
    # a path of always-live edges on the first `depth` vertices: sample sizes from 2 to depth
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, dst = np.arange(1, depth, dtype=np.int32), np.arange(depth - 1, dtype=np.int32)
    g = skis.skis_load_graph(n, src, dst, np.full(depth - 1, 0xFFFFFFFF, np.uint32), skis.SKIS_W_EXPLICIT_TAU)
    s = skis.skis_sketch_create(g, 11)
    skis.skis_sample(s, T)
    e = skis.skis_sketch_export(s, 0, T)
    member = np.zeros((T, depth), bool)
    member[np.repeat(np.arange(T), e["len"]), e["members"]] = True
    rng = np.random.default_rng(T)
    sets = [[depth - 1], [0], [n - 1], list(range(depth))]
    sets += [rng.choice(depth, int(rng.integers(1, min(depth, 60) + 1)), replace=False).tolist() for _ in range(66)]
    off = np.concatenate([[0], np.cumsum([len(x) for x in sets])]).astype(np.int64)
    seeds = np.concatenate(sets).astype(np.int32)
    want = [int(member[:, [v for v in x if v < depth]].any(axis=1).sum()) for x in sets]
    skis.skis_sketch_set_option(s, skis.SKIS_OPT_QUERY_INDEX, 3)
    for _ in range(2):  # the masks are zero again after the first call
        cov, _ = skis.skis_estimate(s, off, seeds)
        assert cov.tolist() == want
    s.close()
    g.close()
