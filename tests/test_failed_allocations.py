"""Any one allocation of a call fails: the call returns SKIS_ENOMEM, and the next calls on the same sketch work in buffers
that are all there and large enough. On the host, with no GPU (fake_cuda)."""
import numpy as np
import pytest

import fake_cuda
import paper_1709_03565_gb300 as skis

N = 3000


def sampler_buffers(s, count, lt, n=N, first=0):
    """The bytes the sampling kernels of a call for `count` more samples (launches from record `first` on) may touch,
    buffer by buffer."""
    T, slots = s.value("T"), s.value("cta_slots_alloc")
    want = {"ctr": 72, "status": 16, "arena": s.value("arena_cap") * 4, "h_off": 8 * T, "h_len": 4 * T, "h_src": 4 * T,
            "h_retries": 4 * T, "h_coins": 8 * T, "to_warp_ids": 8 * count, "to_cta_ids": 8 * count, "big_ids": 8 * count,
            "ovf_ids[0]": 8 * count, "ovf_ids[1]": 8 * count, "srcrec": 16 * count, "srcpick": 8 * count,
            "bitmaps": 4 * slots * s.value("bitmap_words"), "queues": 4 * slots * s.value("queue_cap"),
            "slot_clean": 4 * slots}
    if lt:
        lanes = 128 * [g for name, g, _ in s.launches()[first:] if "k_lt_mid" in name][-1]
        want.update({"lt_hash": lanes * 2048 * 4, "lt_list": lanes * 1024 * 4})
    else:
        grid = [g for name, g, _ in s.launches()[first:] if "k_iis_warp" in name][-1]
        slot_hash, slot_members = (8192, 4096) if n >= 24_576 else (4096, 1536)
        want.update({"spill_hash": 8 * grid * slot_hash * 4, "spill_queue": 8 * grid * slot_members * 4})
    for name, size in want.items():
        assert size > 0 and s.bytes(name) >= size, name
    assert all(g <= slots for name, g, _ in s.launches()[first:] if "k_iis_cta" in name or "k_lt_long" in name)


@pytest.mark.parametrize("lt", [False, True])
@pytest.mark.parametrize("before", [0, 100])
def test_sampling_after_any_allocation_failed(before, lt):
    k = 0
    while True:
        k += 1
        s = fake_cuda.Sketch(N, lt=lt)
        if before:
            assert s.sample(before) == skis.SKIS_OK
        s.fk.fk_fail_at(k, 1)
        rc = s.sample(9000)
        s.fk.fk_fail_at(0, 0)
        assert rc in (skis.SKIS_OK, skis.SKIS_ENOMEM)
        done = before + (9000 if rc == skis.SKIS_OK else 0)
        for count in (60, 7000):
            assert s.sample(count) == skis.SKIS_OK
            done += count
            assert s.value("T") == done and s.fk.fk_events(s.s)
            sampler_buffers(s, count, lt)
        allocs = s.fk.fk_allocs()
        s.close()
        if k > allocs:  # every allocation has failed once
            break


def _estimate(s, off, seeds):
    cov, est = np.zeros(len(off) - 1, np.int64), np.zeros(len(off) - 1)
    return s.fk.skis_estimate(s.s, len(off) - 1, off.ctypes.data, seeds.ctypes.data, cov.ctypes.data, est.ctypes.data,
                              skis.SKIS_MEM_HOST, None)


@pytest.mark.parametrize("mode,T", [(2, 500), (3, 500), (1, 500), (0, (1 << 20) + 1)])
def test_queries_after_any_allocation_failed(mode, T):
    off, seeds = np.array([0, 2, 5], np.int64), np.arange(5, dtype=np.int32)
    for k in range(1, 40):
        s = fake_cuda.Sketch(N)
        s.option(skis.SKIS_OPT_QUERY_INDEX, mode)
        assert s.sample(T) == skis.SKIS_OK
        s.fk.fk_fail_at(k, 1)
        rc = _estimate(s, off, seeds)
        s.fk.fk_fail_at(0, 0)
        if rc == skis.SKIS_OK:
            s.close()
            assert k > 5
            return
        assert rc == skis.SKIS_ENOMEM
        for more in (0, 40):
            assert s.sample(more) == skis.SKIS_OK
            assert _estimate(s, off, seeds) == skis.SKIS_OK
            now = s.value("T")
            want = {"qmask": 8 * N, "qbits": 4 * ((N + 31) // 32), "qcov": 65 * 8, "qstatus": 16}
            if mode in (0, 3):
                want.update({"touched": 4 * now, "ntouched": 24, "hits": 8 << 22, "smask": 8 * now})
            if mode == 1:
                want.update({"smask": 8 * now})
            for name, size in want.items():
                assert s.bytes(name) >= size, (name, k)
            assert s.fk.fk_first_bad(s.s) == 2 ** 64 - 1  # no query of an earlier call
        s.close()
    assert False, "the call never ran out of allocations"
