"""Linear Threshold walks at the edges of the lane tiers: walks of exactly the
members that a tier holds and one more or less, walk counts that fill warps and
refills only in part, and rows whose weight is one share of 2^32, against the
oracle."""
import numpy as np
import pytest

import oracle
import paper_1709_03565_gb300 as skis
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    skis.build()
    yield


def _same(n, src, dst, T, ris, seed, w=None):
    dm, om = (skis.SKIS_W_WC, oracle.W_WC) if w is None else (skis.SKIS_W_EXPLICIT_P, oracle.W_P)
    g = skis.skis_load_graph_lt(n, src, dst, w, dm)
    o = oracle.OracleGraph(n, src, dst, weights=w, model=om, lt=True)
    s = skis.skis_sketch_create(g, seed)
    if ris:
        skis.skis_sketch_set_option(s, skis.SKIS_OPT_SAMPLER, 1)
    skis.skis_sample(s, T)
    dev = skis.skis_sketch_export(s, 0, T)
    ora = o.sample_ids(seed, np.arange(T, dtype=np.uint64), ris=ris)
    assert np.array_equal(dev["len"].astype(np.int64), ora["len"])
    for k in ("src", "coins", "members"):
        assert np.array_equal(dev[k], ora[k]), k
    s.close()
    g.close()
    return dev["len"]


# a walk on a cycle collects the whole cycle: a sample's length is its cycle's
@pytest.mark.parametrize("lens", [(2, 3, 4, 5), (47, 48, 49), (7, 48, 49, 64), (1023, 1024, 1025)])
@pytest.mark.parametrize("T", [1, 31, 33, 1000])
@pytest.mark.parametrize("ris", [False, True])
def test_walks_on_cycles(lens, T, ris):
    src, dst, first = [], [], 0
    for c in lens:
        ids = first + np.arange(c)
        src.append(ids)
        dst.append(first + (np.arange(c) + 1) % c)
        first += c
    got = _same(first, np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32), T, ris, 0xC1C + T)
    assert set(got.tolist()) <= set(lens)


# rows of every degree from 1 to 40 with one weight a row, and with weights of their own
@pytest.mark.parametrize("explicit", [False, True])
@pytest.mark.parametrize("ris", [False, True])
def test_row_degrees(explicit, ris):
    n = 400
    rng = np.random.default_rng(17)
    src, dst = [], []
    for v in range(n):
        d = 1 + v % 40
        src.append(rng.choice(np.delete(np.arange(n), v), d, replace=False))
        dst.append(np.full(d, v))
    src, dst = np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)
    w = None
    if explicit:
        w = synth.uniform_p(len(dst), 5, 0.05, 1.0) / np.bincount(dst, minlength=n)[dst] * 0.999
    _same(n, src, dst, 20_000, ris, 0xDE6, w)
