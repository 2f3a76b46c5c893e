"""The pool that temporaries come from: one per device, bounded, not used under
capture, done without when it is refused, and given back when memory is short
(host code over a stand-in runtime); and on the GPU calls from several threads
and streams at once."""
import ctypes as C
import threading

import numpy as np
import pytest

import fake_runtime


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    return fake_runtime.load(tmp_path_factory.mktemp("temporaries"))


def test_one_bounded_pool_per_device_that_is_given_back(L):
    word = lambda name, t=C.c_ulonglong: t.in_dll(L, "fake_" + name)
    X, ids = np.zeros((1500, 16), np.float32), np.zeros((1500, 8), np.uint32)
    knn = lambda: L.ann_knn_exact(X.ctypes.data, 1500, 16, 8, ids.ctypes.data, None)
    word("capturing", C.c_int).value = 1
    assert knn() == 0 and word("pools").value == 0               # a node of the graph
    word("capturing", C.c_int).value = 0
    assert knn() == 0 and knn() == 0
    assert word("pools").value == 1 and word("temporaries").value == 2
    assert 0 < word("pool_keep").value <= 64 << 20
    L.fake_set_device(1)
    assert knn() == 0 and word("pools").value == 2 and word("temporaries").value == 3
    L.fake_set_device(0)
    word("no_temporaries", C.c_int).value = 1
    launches = word("launches").value
    assert knn() == 0 and word("launches").value == launches + 1   # the plain kernel alone
    word("no_temporaries", C.c_int).value = 0
    knn_ids, graph = np.zeros((64, 8), np.uint32), np.zeros((64, 4), np.uint32)
    assert word("trims").value == 0
    word("no_memory", C.c_int).value = 1
    assert L.ann_graph_prune(knn_ids.ctypes.data, 64, 8, 4, graph.ctypes.data, None) == 2
    word("no_memory", C.c_int).value = 0
    assert word("trims").value == 2


@pytest.mark.gpu
def test_threads_and_streams_at_once():
    """Eight threads, a stream each, lists of different sizes: the same as one
    after another, and what stays reserved is bounded."""
    torch = pytest.importorskip("torch")
    import paper_2507_17094_gb300 as A
    assert torch.cuda.is_available()
    A.build()
    g = torch.Generator(device="cuda").manual_seed(3)
    sets = [torch.randn((1024 + 613 * i, 24 + 8 * i), device="cuda", generator=g) for i in range(8)]
    want = [A.knn_exact(x, 16).cpu() for x in sets]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    got, errors = [[] for _ in sets], []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for r in range(12):
                    got[i].append(A.knn_exact(sets[i], 16))
                    if r % 5 == i % 5:
                        torch.cuda.current_stream().synchronize()
                torch.cuda.current_stream().synchronize()
        except Exception as e:   # noqa: BLE001
            errors.append(e)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sets))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for w, lists in zip(want, got):
        assert len(lists) == 12 and all(torch.equal(x.cpu(), w) for x in lists)
    # most of a workspace of hundreds of megabytes goes back at the synchronisation
    x = torch.randn((40_000, 32), device="cuda", generator=g)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    out = A.knn_exact(x, 32)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= (80 << 20) + out.numel() * 4
