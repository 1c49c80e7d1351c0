"""Greedy, queries, the inverted index and a server on a device that the sampler's scratch has filled: the scratch is given
back before the call is refused, and taken again by the next sampling call. On the host, with no GPU (fake_cuda)."""
import ctypes

import numpy as np
import pytest

import fake_cuda
import paper_1709_03565_gb300 as skis

N, T = 1_000_000, 2_000_000


def _greedy(s):
    seeds = np.zeros(10, np.int32)
    return s.fk.skis_greedy_maxcover(s.s, 10, seeds.ctypes.data, None, None, None)


def _estimate(mode):
    def call(s):
        s.option(skis.SKIS_OPT_QUERY_INDEX, mode)
        off, seeds = np.array([0, 2, 5], np.int64), np.arange(5, dtype=np.int32)
        cov, est = np.zeros(2, np.int64), np.zeros(2)
        return s.fk.skis_estimate(s.s, 2, off.ctypes.data, seeds.ctypes.data, cov.ctypes.data, est.ctypes.data,
                                  skis.SKIS_MEM_HOST, None)
    return call


def _server(s):
    srv = ctypes.c_void_p()
    rc = s.fk.skis_server_create(ctypes.byref(srv), s.s, 2, 64, 4096)
    if rc == skis.SKIS_OK:
        s.fk.skis_server_free(srv)
    return rc


@pytest.mark.parametrize("call", [_greedy, _estimate(2), _estimate(3), _estimate(1), _server])
def test_the_scratch_makes_room(call):
    s = fake_cuda.Sketch(N)
    assert s.sample(T) == skis.SKIS_OK and s.bytes("queues") > 0
    s.fk.fk_start(s.fk.fk_used() + 100_000)  # no room but the scratch's
    assert call(s) == skis.SKIS_OK
    assert s.bytes("queues") == 0 and s.bytes("arena") > 0
    s.fk.fk_start(280 << 30)
    assert s.sample(100) == skis.SKIS_OK and s.value("lean") == 0
    assert s.bytes("queues") >= 4 * s.value("cta_slots_alloc") * s.value("queue_cap") > 0
    assert call(s) == skis.SKIS_OK
    s.close()


def test_no_room_at_all_is_still_refused():
    s = fake_cuda.Sketch(N)
    assert s.sample(1000) == skis.SKIS_OK
    s.fk.fk_fail_at(1, 1)
    assert _greedy(s) == skis.SKIS_ENOMEM and _estimate(2)(s) == skis.SKIS_ENOMEM and _server(s) == skis.SKIS_ENOMEM
    s.fk.fk_fail_at(0, 0)
    assert s.sample(1000) == skis.SKIS_OK and _greedy(s) == skis.SKIS_OK
    s.close()
