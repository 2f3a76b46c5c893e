"""Distances from shared memory for every split of a row over its lanes: 16 rows
a round on lane pairs, 8 or 4 rows on four lanes each, and a block's rows, at
the dimensions where the 16-byte units of row and query end, for every storage.
All of them run the same FP32 operations, so the results are equal bit for bit
to each other and to the oracle's."""
import numpy as np
import pytest

import oracle as O
from workloads import build_graph, ghost_sample

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DIMS = [1, 3, 4, 7, 8, 9, 15, 16, 17, 24, 31, 32, 33, 63, 65, 100, 128, 161, 256, 387]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2507_17094_gb300 as A
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    A.build()


@pytest.mark.parametrize("d", DIMS)
@pytest.mark.parametrize("storage", [0, 1, 2])
def test_equals_the_oracle(d, storage, monkeypatch):
    import paper_2507_17094_gb300 as A
    rng = np.random.default_rng(d)
    n, nq, nref = 400, 1200, 24
    X = rng.standard_normal((n, d)).astype(np.float32)
    S = ghost_sample(n, 40, 1)
    G = build_graph(X, 16, 32, "exact")
    Gg = build_graph(X[S], 8, 16, "exact", n_bridge=0)
    Q = rng.standard_normal((nq, d)).astype(np.float32)
    params = dict(k=8, itopk=24, max_iters=30, entry=1, dgs_discard=0.5, rerank=int(storage != 0), seed=3, qid_base=2)
    ix = A.Index(X, G, storage=storage, ghost_ids=S, ghost_graph=Gg)
    o_ids, o_d, _ = O.search(O.OracleIndex(X, G, storage, S, Gg), Q[:nref], **params)
    q = torch.from_numpy(Q).cuda()
    first = None
    for rows in (16, 8, 4, 0):
        monkeypatch.setenv("ANN_STAGE_ROWS", str(rows))
        ids, dists, _ = ix.search(q, **params)
        ids, dists = ids.cpu().numpy().view(np.uint32), dists.cpu().numpy()
        assert np.array_equal(ids[:nref], o_ids) and np.array_equal(dists[:nref], o_d), rows
        first = first or (ids, dists)
        assert np.array_equal(ids, first[0]) and np.array_equal(dists, first[1]), rows
    ids, dists, _ = ix.search(q[:100], **params)        # a block per query
    assert np.array_equal(ids.cpu().numpy().view(np.uint32), first[0][:100])
    assert np.array_equal(dists.cpu().numpy(), first[1][:100])
    ix.close()
