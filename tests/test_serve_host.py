"""The server's host side where the runtime refuses a launch: the request is
refused, nothing of it is published, and every admitted request is answered."""
import ctypes as C

import numpy as np
import pytest

import fake_runtime
import paper_2507_17094_gb300 as A


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    return fake_runtime.load(tmp_path_factory.mktemp("serve_host"))


@pytest.mark.parametrize("busy", [0, 1])
def test_a_refused_launch_publishes_nothing(L, busy):
    """With a busy stream the launches before the refused one are still queued
    and read what the host has published when they start."""
    d, k = 8, 4
    ix, srv, X = C.c_void_p(), C.c_void_p(), np.zeros((64, d), np.float32)
    G = np.zeros((64, 4), np.uint32)
    assert L.ann_index_create(0, A.F32, 64, d, 4, X.ctypes.data, G.ctypes.data, 0, None, 0, None, 1, 1,
                              C.byref(ix)) == 0
    p = A.make_params(k=k, itopk=16, max_iters=8)
    cfg = A.binding.ServerConfig(capacity=32, max_requests=8, max_params=p, streams=1)
    assert L.ann_server_create(ix, C.byref(cfg), None, C.byref(srv)) == 0
    fail, busy_now = C.c_int.in_dll(L, "fake_fail_launches"), C.c_int.in_dll(L, "fake_busy")
    results = []

    def submit(rid, nq):
        results.append((np.empty((nq, k), np.uint32), np.empty((nq, k), np.float32)))
        return L.ann_server_submit(srv, rid, np.zeros((nq, d), np.float32).ctypes.data, nq, C.byref(p),
                                   results[-1][0].ctypes.data, results[-1][1].ctypes.data)

    def finished():
        L.fake_run_serve()
        out, n, ids = (A.binding.Completion * 8)(), C.c_uint32(), []
        assert L.ann_server_poll(srv, out, 8, C.byref(n)) == 0
        return [out[i].req_id for i in range(n.value)]

    assert submit(1, 3) == 0
    busy_now.value = busy
    assert submit(2, 4) == 0
    fail.value = 1
    assert submit(3, 5) != 0
    assert sorted(finished()) == [1, 2]
    busy_now.value = 0
    assert submit(4, 2) == 0 and submit(5, 6) == 0
    assert sorted(finished()) == [4, 5]
    assert L.ann_server_in_flight(srv) == 0
    assert L.ann_server_destroy(srv) == 0 and L.ann_index_free(ix) == 0
