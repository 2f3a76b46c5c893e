"""The filtered kNN lists at the ends of FP32's range: where distances overflow
(all of them infinite, so the order is by id), where squares fall among the
subnormal numbers and lose bits, and at scales the filter still takes. The ids
are those of the definition."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2507_17094_gb300 as A
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    A.build()


def reference(X, K, rows):
    """The K other nodes nearest to each of the given rows by (distance, id),
    infinite distances among them. The fused multiply-add is formed in FP64
    (the square is exact there) and rounded to FP32."""
    q = X[rows]
    acc = torch.zeros((len(rows), X.shape[0]), dtype=torch.float32, device=X.device)
    for i in range(X.shape[1]):
        df = (q[:, i:i + 1] - X[None, :, i]).double()
        acc = (acc.double() + df * df).float()
    key = (acc.view(torch.int32).long() << 32) | torch.arange(X.shape[0], device=X.device)
    key[torch.arange(len(rows), device=X.device), rows] = torch.iinfo(torch.int64).max
    return (torch.topk(key, K, dim=1, largest=False).values & 0xFFFFFFFF).to(torch.int32)


def points(kind, n, d, g):
    x = torch.rand((n, d), device="cuda", generator=g) * 2 - 1
    if kind == "signs":                      # every distance between different rows overflows
        return torch.where(x > 0, 1.5, -1.5) * 2.0 ** 60
    if kind == "wide":                       # some sums of squares overflow, some do not
        return x * 2e18
    if kind == "outlier":                    # one row sets the scale, the others' squares are subnormal
        x *= 2.0 ** -74
        x[5, 0] = 1.5 * 2.0 ** -60
        return x
    return x * kind                          # a power of two


@pytest.mark.parametrize("n,d,K,kind", [
    (1500, 128, 20, "signs"), (2000, 256, 33, "wide"), (1500, 64, 24, "outlier"), (1500, 40, 16, 2.0 ** -66),
    (1500, 40, 16, 2.0 ** -55), (1500, 40, 16, 2.0 ** -50), (1500, 40, 16, 2.0 ** -49), (1500, 40, 16, 2.0 ** 50),
    (1500, 40, 16, 2.0 ** 51), (1500, 40, 16, 2.0 ** 56), (1500, 40, 16, 2.0 ** 61),
])
def test_lists_at_the_ends_of_the_range(n, d, K, kind):
    import paper_2507_17094_gb300 as A
    g = torch.Generator(device="cuda").manual_seed(n + d + K)
    X = points(kind, n, d, g)
    rows = torch.arange(0, n, 7, device="cuda")
    assert torch.equal(A.knn_exact(X, K)[rows], reference(X, K, rows))
