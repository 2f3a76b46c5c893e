"""Two host threads with an object each: a kernel's limit of dynamic shared
memory belongs to the kernel, so what one thread's call sets must leave the
other's launches possible. Run without a GPU: the stand-in runtime refuses a
launch beyond its kernel's limit, and lets a second object's whole call happen
between any call's setting of a limit and what follows it."""
import ctypes as C

import numpy as np
import pytest

import fake_runtime
import paper_2507_17094_gb300 as A


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    return fake_runtime.load(tmp_path_factory.mktemp("limits"))


def f32(*shape):
    return np.zeros(shape, np.float32)


def network(L, out, device=0):
    h = C.c_void_p()
    assert L.ann_mlp_create(device, 16, 16, 16, out, 64, C.byref(h)) == 0
    return h


def train(L, out):
    h, x, y = network(L, out), f32(64, 16), np.zeros(64, np.uint32)
    return lambda: L.ann_mlp_train_step(h, x.ctypes.data, y.ctypes.data, 64, 1e-3, 0.9, 0.999, 1e-8, 0.0, None, None)


def prune(L, K):
    knn, graph = np.zeros((300, K), np.uint32), np.zeros((300, 64), np.uint32)
    return lambda: L.ann_graph_prune(knn.ctypes.data, 300, K, 64, graph.ctypes.data, None)


def knn(L, n, d):
    x, ids = f32(n, d), np.zeros((n, 16), np.uint32)
    return lambda: L.ann_knn_exact(x.ctypes.data, n, d, 16, ids.ctypes.data, None)


def index(L, d, n=64):
    ix, x, g = C.c_void_p(), f32(n, d), np.zeros((n, 16), np.uint32)
    assert L.ann_index_create(0, A.F32, n, d, 16, x.ctypes.data, g.ctypes.data, 0, None, 0, None, 1, 1,
                              C.byref(ix)) == 0
    return ix


def search(L, d, nq):
    ix, q, p = index(L, d), f32(nq, d), A.make_params(k=4, itopk=64, search_width=4)
    ids, dists = np.zeros((nq, 4), np.uint32), f32(nq, 4)
    return lambda: L.ann_search(ix, q.ctypes.data, nq, C.byref(p), None, 0, ids.ctypes.data, dists.ctypes.data, None,
                                None)


def serve(L, d):
    ix, srv, p = index(L, d), C.c_void_p(), A.make_params(k=4, itopk=64, search_width=4)
    cfg = A.binding.ServerConfig(capacity=64, max_requests=8, max_params=p, streams=1)
    q, ids, dists = f32(2, d), np.zeros((2, 4), np.uint32), f32(2, 4)
    assert L.ann_server_create(ix, C.byref(cfg), None, C.byref(srv)) == 0

    def call():
        st = L.ann_server_submit(srv, 1, q.ctypes.data, 2, C.byref(p), ids.ctypes.data, dists.ctypes.data)
        out, n = (A.binding.Completion * 8)(), C.c_uint32()
        L.fake_run_serve()
        assert L.ann_server_poll(srv, out, 8, C.byref(n)) == 0
        return st
    return call


@pytest.mark.parametrize("make,large,small", [
    (train, (40_000,), (13_000,)), (prune, (256,), (130,)), (knn, (2000, 500), (1500, 200)), (knn, (500, 500), (400, 100)),
    (search, (960, 4), (64, 4)), (search, (960, 5000), (64, 5000)), (serve, (960,), (64,))])
def test_one_calls_limit_leaves_the_others_launch_possible(L, make, large, small):
    ours, others = make(L, *large), make(L, *small)
    assert ours() == 0 and others() == 0          # each on its own
    statuses = []
    hook = C.CFUNCTYPE(None)(lambda: statuses.append(others()))
    at = C.c_void_p.in_dll(L, "fake_after_limit")
    at.value = C.cast(hook, C.c_void_p).value
    try:
        status = ours()
    finally:
        at.value = None
    assert statuses and not any(statuses), L.ann_last_error()
    assert status == 0, L.ann_last_error()


@pytest.mark.parametrize("rows", [8, 64])
def test_a_network_on_a_second_device(L, rows):
    """The limit belongs to the device, too: networks on two devices of one
    process, forward, training and prediction, the second after the first."""
    for device in (0, 1, 0):
        h, x = network(L, 2000, device), f32(64, 16)
        logits, y = f32(64, 2000), np.zeros(64, np.uint32)
        seeds, pmax = np.zeros((64, 8), np.uint32), f32(64)
        assert L.ann_mlp_forward(h, x.ctypes.data, rows, logits.ctypes.data, None) == 0, L.ann_last_error()
        assert L.ann_mlp_train_step(h, x.ctypes.data, y.ctypes.data, rows, 1e-3, 0.9, 0.999, 1e-8, 0.0, None, None) == 0
        assert L.ann_mlp_predict(h, x.ctypes.data, rows, 8, 0.0, seeds.ctypes.data, pmax.ctypes.data, None) == 0
        assert L.ann_mlp_free(h) == 0
