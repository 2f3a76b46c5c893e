"""Graph pruning against the builder's oracle at the sizes where its tables
and counting change: each number of 32-entry words of a list, lists with
repeated, invalid and out-of-range entries, buckets of offers around the size
that is ranked in shared memory."""
import numpy as np
import pytest

from oracle import INVALID
from oracle import graph as OG

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2507_17094_gb300 as A
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    A.build()


def prune(knn, degree):
    import paper_2507_17094_gb300 as A
    return A.graph_prune(torch.from_numpy(knn.view(np.int32)).cuda(), degree).cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("n,K,degree", [(70, 1, 1), (90, 31, 2), (140, 32, 32), (150, 33, 17), (160, 64, 64),
                                        (200, 65, 9), (230, 96, 64), (220, 129, 128), (300, 161, 31),
                                        (320, 200, 100), (330, 256, 128)])
def test_each_list_width(n, K, degree):
    rng = np.random.default_rng(n + K)
    knn = np.stack([rng.permutation(np.delete(np.arange(n), u))[:K] for u in range(n)]).astype(np.uint32)
    assert np.array_equal(prune(knn, degree), OG.prune(knn, degree))


@pytest.mark.parametrize("hubs", [1, 2, 40])
def test_buckets_around_the_counted_size(hubs):
    """Node h < hubs is the first neighbour of about 96 others, give or take
    one per hub, so that buckets just below, at and above the counted size (and
    one of 400) occur; the lists' tails are invalid."""
    rng = np.random.default_rng(hubs)
    n, K, degree = 4200, 12, 10
    knn = np.full((n, K), INVALID, np.uint32)
    at = hubs
    for h in range(hubs):
        size = 400 if hubs == 1 else 96 - hubs // 2 + h
        for u in range(at, at + size):
            knn[u, 0] = h
        at += size
    for u in range(n):
        extra = rng.permutation(n)[:8]
        extra = [v for v in extra if v != u and v != knn[u, 0]][:6]
        first = 0 if knn[u, 0] == INVALID else 1
        knn[u, first:first + len(extra)] = extra
    assert np.array_equal(prune(knn, degree), OG.prune(knn, degree))


def test_repeated_ids_and_a_regular_id_set():
    """Lists with repeated entries (the smallest rank counts), and ids spaced
    so that multiplicative hashing is at its worst (differences that are powers
    of two)."""
    rng = np.random.default_rng(3)
    n, K, degree = 300, 70, 32
    knn = np.stack([rng.permutation(n)[:K] for _ in range(n)]).astype(np.uint32)
    knn[::3, 40:] = knn[::3, :30]
    assert np.array_equal(prune(knn, degree), OG.prune(knn, degree))
    n, K = 1 << 10, 128
    step = (np.arange(K, dtype=np.uint64) << 3).astype(np.uint32)
    knn = (np.arange(n, dtype=np.uint32)[:, None] + step[None, :]) % n
    assert np.array_equal(prune(knn, 64), OG.prune(knn, 64))


def test_lists_no_multiplier_keeps_apart():
    """Lists of 128 ids that collide in 4,096 slots under each of the 64
    multipliers tried (about one random list in 7,000), each listing others."""
    rng = np.random.default_rng(11)
    n, K, degree = 20_000, 128, 40
    muls, mul = [], 2654435761
    for _ in range(64):
        muls.append(mul)
        mul = ((mul * 1664525 + 1013904223) & 0xFFFFFFFF) | 1
    hard = []
    for _ in range(200):
        lists = rng.integers(200, n, size=(2000, K), dtype=np.uint32)
        lists = lists[[len(np.unique(r)) == K for r in lists]]
        for m in muls:
            slots = np.sort((lists * np.uint32(m)) >> np.uint32(20), axis=1)
            lists = lists[(slots[:, 1:] == slots[:, :-1]).any(axis=1)]
        hard += list(lists)
        if len(hard) >= 4:
            break
    assert hard
    knn = np.full((n, K), INVALID, np.uint32)
    for u, row in enumerate(hard):
        knn[u] = row
        for w in row[:20]:                     # their lists share many of its ids
            knn[w] = rng.permutation(row)
    assert np.array_equal(prune(knn, degree), OG.prune(knn, degree))
