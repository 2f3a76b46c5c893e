"""The search of small batches (a block per query) and of larger ones (a warp
per query) against the oracle at the sizes where either can go wrong: both
sides of the batch size that divides them, every storage, one and several
parents, queues of one entry to the largest, lists and rows of every padding,
direction words beyond those held in registers, a visited table that resets."""
import numpy as np
import pytest

import oracle as O
from workloads import build_graph, ghost_sample

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2507_17094_gb300 as A
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    A.build()


_made = {}


def data(n, d, degree):
    if (n, d, degree) not in _made:
        rng = np.random.default_rng(n + d + degree)
        X = rng.standard_normal((n, d)).astype(np.float32)
        S = ghost_sample(n, max(40, n // 20), 1)
        _made[n, d, degree] = (X, build_graph(X, degree, min(2 * degree, n - 2), "exact"), S,
                               build_graph(X[S], 8, 16, "exact", n_bridge=0),
                               rng.standard_normal((4000, d)).astype(np.float32))
    return _made[n, d, degree]


CASES = [
    # n, d, degree, storage, queries, parameters
    (1500, 33, 16, 0, 1, dict(k=1, itopk=1, max_iters=3, entry=0)),
    (1500, 33, 16, 1, 7, dict(k=5, itopk=7, max_iters=24, entry=1, rerank=1, dgs_discard=0.5)),
    (1500, 33, 13, 2, 65, dict(k=10, itopk=33, max_iters=48, entry=1, rerank=1, dgs_discard=0.3, search_width=3)),
    (1500, 96, 64, 0, 153, dict(k=10, itopk=129, max_iters=90, entry=1, dgs_discard=0.75, ghost_search_width=4)),
    (1500, 96, 64, 2, 40, dict(k=10, itopk=64, max_iters=80, entry=0, dgs_min_match=0.55, search_width=2)),
    (1500, 300, 32, 1, 33, dict(k=10, itopk=32, max_iters=48, entry=1, dgs_discard=0.5, rerank=1)),
    (1500, 768, 24, 1, 20, dict(k=20, itopk=64, max_iters=64, entry=1, dgs_discard=0.5, rerank=1, search_width=2)),
    (1500, 516, 20, 0, 20, dict(k=20, itopk=40, max_iters=64, entry=1, dgs_discard=0.25, dgs_reexpand=1)),
    (1500, 4, 8, 2, 90, dict(k=3, itopk=16, max_iters=32, entry=1, dgs_discard=0.5, rerank=1)),
    (6000, 24, 64, 0, 30, dict(k=50, itopk=512, max_iters=400, entry=1, ghost_itopk=300, search_width=8)),
    (1500, 33, 16, 0, 4000, dict(k=10, itopk=32, max_iters=48, entry=1, dgs_discard=0.5)),
    (1500, 96, 64, 1, 3000, dict(k=10, itopk=64, max_iters=80, entry=1, dgs_discard=0.5, rerank=1)),
    (1500, 300, 32, 2, 1500, dict(k=10, itopk=100, max_iters=80, entry=0, dgs_discard=0.5, search_width=2)),
]


@pytest.mark.parametrize("n,d,degree,storage,nq,params", CASES)
def test_equals_the_oracle(n, d, degree, storage, nq, params):
    import paper_2507_17094_gb300 as A
    X, G, S, Gg, Q = data(n, d, degree)
    params = dict(params, seed=9, qid_base=5)
    ix = A.Index(X, G, storage=storage, ghost_ids=S, ghost_graph=Gg)
    oi = O.OracleIndex(X, G, storage, S, Gg)
    ids, dists, st = ix.search(torch.from_numpy(Q[:nq]).cuda(), stats=True, **params)
    torch.cuda.synchronize()
    ix.sync()
    o_ids, o_d, o_st = O.search(oi, Q[:nq], **params)
    assert np.array_equal(ids.cpu().numpy().view(np.uint32), o_ids)
    assert np.array_equal(dists.cpu().numpy(), o_d)
    st = A.binding.stats_to_numpy(st)
    exact = st["hash_resets"] == 0            # a reset lets rows be evaluated again
    for f in ("iters", "parents", "dgs_parents", "ghost_iters", "ghost_parents", "ghost_vec_rows", "rerank_rows"):
        assert np.array_equal(st[f], o_st[f]), f
    assert np.array_equal(st["vec_rows"][exact], o_st["vec_rows"][exact])
    ix.close()


@pytest.mark.parametrize("nq", [3, 1800])
def test_given_seeds_and_the_judge(nq):
    import paper_2507_17094_gb300 as A
    X, G, S, Gg, Q = data(1500, 33, 16)
    rng = np.random.default_rng(nq)
    given = rng.integers(0, len(S), size=(nq, 4)).astype(np.uint32)
    given[::5, 0] = O.INVALID
    given[1::7, 2] = len(S) + 3
    ix = A.Index(X, G, storage=1, ghost_ids=S, ghost_graph=Gg)
    oi = O.OracleIndex(X, G, 1, S, Gg)
    for params in (dict(entry=2, ghost_judge=float(40.0), ghost_max_iters_given=1, ghost_max_iters=9),
                   dict(entry=3, num_seeds=0)):
        params = dict(params, k=10, itopk=24, max_iters=30, dgs_discard=0.5, seed=3)
        ids, dists, _ = ix.search(torch.from_numpy(Q[:nq]).cuda(),
                                  given=torch.from_numpy(given.view(np.int32)).cuda(), **params)
        o_ids, o_d, _ = O.search(oi, Q[:nq], given_seeds=given, **params)
        assert np.array_equal(ids.cpu().numpy().view(np.uint32), o_ids)
        assert np.array_equal(dists.cpu().numpy(), o_d)
    ix.close()
