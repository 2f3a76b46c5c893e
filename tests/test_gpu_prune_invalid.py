"""Invalid entries in the pruned lists and in their neighbours' lists: they are
no edges, so they have no detours, whichever way a list's entries are looked
up (a table of ranks, a scan where no multiplier keeps the ids apart, probing
for long lists). Node 0 lists nodes whose own lists repeat its ids or hold
invalid entries at low ranks."""
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


def apart(row, muls):
    return [len(np.unique((row * np.uint32(m)) >> np.uint32(20))) == len(row) for m in muls]


@pytest.mark.parametrize("lookup,valid,K", [("scan", 126, 128), ("table", 126, 128), ("table", 40, 50),
                                            ("probing", 150, 180)])
def test_invalid_entries_have_no_detours(lookup, valid, K):
    import paper_2507_17094_gb300 as A
    n, degree = 20_000, 40
    muls, mul = [], 2654435761
    for _ in range(64):
        muls.append(mul)
        mul = ((mul * 1664525 + 1013904223) & 0xFFFFFFFF) | 1
    rng = np.random.default_rng(622)     # one of whose lists collides under every multiplier
    if lookup == "scan":
        lists = rng.integers(200, n, size=(2000, valid), dtype=np.uint32)
        row = next(r for r in lists if len(np.unique(r)) == valid and not any(apart(r, muls)))
    else:
        row = rng.permutation(np.arange(200, n, dtype=np.uint32))[:valid]
        assert lookup == "probing" or any(apart(row, muls))
    knn = np.full((n, K), INVALID, np.uint32)
    knn[0, :valid] = row
    for w in row[:20]:
        knn[w, :valid] = rng.permutation(row)
    want = OG.prune(knn, degree)
    got = A.graph_prune(torch.from_numpy(knn.view(np.int32)).cuda(), degree).cpu().numpy().view(np.uint32)
    assert np.array_equal(got, want)
