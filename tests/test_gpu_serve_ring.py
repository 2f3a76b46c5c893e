"""The serving ring under pressure: more requests than the ring and its records
hold, so that slots and records are reused and queries wrap around, with one
stream and several, and a minimum of queries per warp. Every answer equals the
same search on its own."""
import numpy as np
import pytest

from workloads import build_graph, ghost_sample

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def index():
    import paper_2507_17094_gb300 as A
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    A.build()
    rng = np.random.default_rng(2)
    X = rng.standard_normal((3000, 40)).astype(np.float32)
    S = ghost_sample(3000, 80, 1)
    ix = A.Index(X, build_graph(X, 16, 32, "exact"), storage=A.F16, ghost_ids=S,
                 ghost_graph=build_graph(X[S], 8, 16, "exact", n_bridge=0))
    yield ix
    ix.close()


@pytest.mark.parametrize("capacity,records,streams,per_warp,most", [
    (1, 1, 1, 0, 1), (61, 3, 2, 0, 61), (257, 9, 4, 0, 40), (257, 64, 3, 5, 7), (5000, 40, 4, 0, 900)])
def test_reused_slots_and_records(index, capacity, records, streams, per_warp, most):
    import paper_2507_17094_gb300 as A
    rng = np.random.default_rng(capacity + most)
    params = dict(k=5, itopk=16, max_iters=24, entry=1, dgs_discard=0.5, rerank=1, seed=4)
    srv = A.Server(index, capacity=capacity, max_requests=records, max_params=dict(params, k=8), streams=streams,
                   queries_per_warp=per_warp)
    requests = [rng.standard_normal((int(rng.integers(1, most + 1)), 40)).astype(np.float32) for _ in range(120)]
    done, i = {}, 0
    for _ in range(2_000_000):
        while i < len(requests) and srv.submit(i, requests[i], **dict(params, k=1 + i % 8)):
            i += 1
        for rid, ids, dists, _lat in srv.poll():
            done[rid] = (ids, dists)
        if len(done) == len(requests):
            break
    assert len(done) == len(requests) and srv.in_flight() == 0
    for r in range(0, len(requests), 7):
        ids, dists, _ = index.search(torch.from_numpy(requests[r]).cuda(), **dict(params, k=1 + r % 8))
        assert np.array_equal(done[r][0], ids.cpu().numpy().view(np.uint32))
        assert np.array_equal(done[r][1], dists.cpu().numpy())
    srv.close()
