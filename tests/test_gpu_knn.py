"""The filtered kNN lists against the definition (FP32, one fused multiply-add
per element in index order, ordered by (distance, id)): the ids are equal, at
the edges of the filter's tiles, ranges and row blocks, for inputs whose
distances tie, whose buffers overflow and which its operands cannot bound."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2507_17094_gb300 as A
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    A.build()


def reference(X, K, rows):
    """The K nearest of the given rows. The fused multiply-add is formed in
    FP64 (the square is exact there) and rounded to FP32."""
    q = X[rows]
    acc = torch.zeros((len(rows), X.shape[0]), dtype=torch.float32, device=X.device)
    for i in range(X.shape[1]):
        df = (q[:, i:i + 1] - X[None, :, i]).double()
        acc = (acc.double() + df * df).float()
    acc[torch.arange(len(rows), device=X.device), rows] = float("inf")
    key = (acc.view(torch.int32).long() << 32) | torch.arange(X.shape[0], device=X.device)
    key[acc.isnan()] = torch.iinfo(torch.int64).max
    return (torch.topk(key, K, dim=1, largest=False).values & 0xFFFFFFFF).to(torch.int32)


def points(kind, n, d, g):
    x = torch.randn((n, d), device="cuda", generator=g)
    if kind == "integer":                       # many equal distances, exact in FP16
        return (40.0 * x + 120.0).clamp(0, 255).round()
    if kind == "clusters":                      # ordered by cluster: a column range is not a sample of X
        return x + 4.0 * torch.randn((16, d), device="cuda", generator=g).repeat_interleave(-(-n // 16), 0)[:n]
    if kind == "offset":                        # far from the origin: the centring matters
        return x + 1000.0
    if kind == "few":                           # 40 distinct rows: every list overflows
        return x[torch.randint(0, 40, (n,), device="cuda", generator=g)].contiguous()
    if kind == "outlier":                       # one row sets the scale of the operands
        x[3] *= 1e6
    if kind == "tiny":                          # squares below the smallest normal number
        return x * 1e-25
    if kind == "unaligned":                     # rows not on 16-byte boundaries
        return torch.randn(n * d + 1, device="cuda", generator=g)[1:].view(n, d)
    return x


@pytest.mark.parametrize("n,d,K,kind", [
    (1023, 64, 32, "normal"), (1024, 64, 32, "normal"), (1025, 33, 1, "normal"), (1153, 100, 256, "normal"),
    (2048, 128, 64, "integer"), (5003, 7, 17, "integer"), (4099, 96, 96, "clusters"), (3000, 96, 32, "offset"),
    (2500, 32, 48, "few"), (3001, 64, 32, "outlier"), (1500, 40, 16, "tiny"), (2100, 64, 32, "unaligned"),
    (9731, 580, 16, "normal"), (19585, 65, 128, "normal"), (38913, 48, 64, "clusters"),
])
def test_filtered_lists_equal_the_definition(n, d, K, kind):
    import paper_2507_17094_gb300 as A
    g = torch.Generator(device="cuda").manual_seed(n + d + K)
    X = points(kind, n, d, g)
    got = A.knn_exact(X, K)
    rows = torch.unique(torch.cat([torch.randperm(n, device="cuda", generator=g)[:160],
                                   torch.tensor([0, 3, 127, 128, n - 1], device="cuda")]))
    assert torch.equal(got[rows], reference(X, K, rows))


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 1e30])
def test_values_the_operands_cannot_bound(value):
    """An unusable value in one row: every list as the plain computation has
    it (a NaN distance is never listed, an overflowing one is infinite)."""
    import paper_2507_17094_gb300 as A
    g = torch.Generator(device="cuda").manual_seed(5)
    X = torch.randn((2000, 24), device="cuda", generator=g)
    X[17, 5] = value
    rows = torch.cat([torch.arange(17, device="cuda"), torch.arange(18, 100, device="cuda")])
    assert torch.equal(A.knn_exact(X, 20)[rows], reference(X, 20, rows))
