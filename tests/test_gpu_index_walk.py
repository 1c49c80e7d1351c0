"""Coverage through the inverted index where a seed's sample list is cut into chunks of 256: lists of exactly one
chunk, one entry more, many chunks, and more chunks than the walk's queue holds. Against the counts of the exported
samples (integers: equal) and the scan of the sketch."""
import numpy as np
import pytest

import paper_1709_03565_gb300 as skis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [256, 257, 512, 100_000])
def test_list_lengths_at_the_chunk_edges(T):
    # vertex 0's only in-neighbour is 1 and so on along a path of always-live edges, so vertex n - 1 is in every
    # sample and the others in fewer
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 70
    src, dst = np.arange(1, n, dtype=np.int32), np.arange(n - 1, dtype=np.int32)
    g = skis.skis_load_graph(n, src, dst, np.full(n - 1, 0xFFFFFFFF, np.uint32), skis.SKIS_W_EXPLICIT_TAU)
    s = skis.skis_sketch_create(g, 11)
    skis.skis_sample(s, T)
    e = skis.skis_sketch_export(s, 0, T)
    member = np.zeros((T, n), bool)
    member[np.repeat(np.arange(T), e["len"]), e["members"]] = True
    rng = np.random.default_rng(T)
    sets = [[n - 1], [0], [n - 1, 0], list(range(n))] + [rng.choice(n, k, replace=False).tolist() for k in range(1, 62)]
    off = np.concatenate([[0], np.cumsum([len(x) for x in sets])]).astype(np.int64)
    seeds = np.concatenate(sets).astype(np.int32)
    want = [int(member[:, x].any(axis=1).sum()) for x in sets]
    assert want[0] == T  # a list of T entries
    for mode in (1, 2, 1):
        skis.skis_sketch_set_option(s, skis.SKIS_OPT_QUERY_INDEX, mode)
        cov, _ = skis.skis_estimate(s, off, seeds)
        assert cov.tolist() == want
    s.close()
    g.close()


def test_more_chunks_than_the_queue_holds():
    # a server whose slots take 64 seeds: 64 requests for vertices in all of 2.2M samples queue 64 x 8593 chunks, more
    # than the 524,352 places
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, T = 65, 2_200_000
    src, dst = np.arange(1, n, dtype=np.int32), np.zeros(n - 1, np.int32)  # the centre of an always-live star
    g = skis.skis_load_graph(n, src, dst, np.full(n - 1, 0xFFFFFFFF, np.uint32), skis.SKIS_W_EXPLICIT_TAU)
    s = skis.skis_sketch_create(g, 12, 65 * T + (1 << 24))
    skis.skis_sample(s, T)
    srv = skis.skis_server_create(s, slots=1, max_batch=64, seed_capacity=64)
    for _ in range(2):  # the masks are zero again after the first batch
        tickets = [skis.skis_server_submit(srv, np.array([v], np.int32)) for v in range(1, n)]
        done = 0
        while done < len(tickets):
            done += len(skis.skis_server_progress(srv, wait=True))
        assert [skis.skis_server_poll(srv, t)[1] for t in tickets] == [T] * (n - 1)
    srv.close()
    s.close()
    g.close()
