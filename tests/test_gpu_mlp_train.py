"""The training step's products, sums and update at the sizes where their
tiles and paths change: operands read transposed with ragged edges, narrow and
wide tiles, column sums of partial chunks, rows of logits in shared memory and
too long for it; and an epoch against its steps one by one."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2507_17094_gb300 as A
    assert torch.cuda.is_available()
    A.build()


def make(d, h1, h2, out, seed):
    import paper_2507_17094_gb300 as A
    rng = np.random.default_rng(seed)
    shapes = ((h1, d), (h1,), (h2, h1), (h2,), (out, h2), (out,))
    m = M.MLP(*((rng.standard_normal(s) * (np.sqrt(2.0 / s[-1]) if len(s) == 2 else 0.1)).astype(np.float32)
                for s in shapes))
    g = A.MLP(d, h1, h2, out, 2048)
    g.set_params(m.W1, m.b1, m.W2, m.b2, m.W3, m.b3)
    return m, g


@pytest.mark.parametrize("d,h1,h2,out,n", [
    (8, 8, 8, 8, 8), (72, 136, 72, 1016, 1032), (24, 200, 264, 8, 64), (96, 64, 192, 20_000, 264),
    (16, 24, 16, 51_208, 16), (40, 512, 512, 640, 2048)])
def test_gradients_vs_oracle(d, h1, h2, out, n):
    """Relative Frobenius norm 1e-2: the hidden activations and gradients are
    rounded to BF16 on both sides, and where the two sums straddle a rounding
    boundary they differ by 2^-8 of the value."""
    m, g = make(d, h1, h2, out, n)
    rng = np.random.default_rng(n + 1)
    X = rng.standard_normal((n, d)).astype(np.float32)
    y = rng.integers(0, out, n).astype(np.uint32)
    loss = torch.zeros(1, device="cuda")
    g.train_step(torch.from_numpy(X).cuda(), torch.from_numpy(y.view(np.int32)).cuda(), lr=0.0, loss=loss)
    g.sync()
    want = M.gradients(m, X, y.astype(np.int64))
    for k, got in zip(M.LAYERS, g.get(1)):
        err = np.linalg.norm(got.astype(np.float64) - want[k])
        assert err <= 1e-2 * np.linalg.norm(want[k]) + 1e-12, k
    assert abs(loss.item() - M.loss(m, X, y.astype(np.int64))) <= 1e-2 * abs(loss.item())
    g.close()


def mix64(x):
    k = (1 << 64) - 1
    z = (x + 0x9E3779B97F4A7C15) & k
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & k
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & k
    return z ^ (z >> 31)


@pytest.mark.parametrize("n,batch", [(1000, 256), (40, 8), (2600, 1024)])
def test_an_epoch_equals_its_steps(n, batch):
    """Two epochs take the rows in the documented order, in batches cut to a
    multiple of 8: the parameters equal those of the steps made one by one."""
    _, a = make(40, 72, 136, 600, 1)
    _, b = make(40, 72, 136, 600, 1)
    rng = np.random.default_rng(n)
    X = torch.from_numpy(rng.standard_normal((n, 40)).astype(np.float32)).cuda()
    y = torch.from_numpy(rng.integers(0, 600, n).astype(np.int32)).cuda()
    a.train_epochs(X, y, batch=batch, epochs=2, seed=7)
    for epoch in range(2):
        order, key = list(range(n)), mix64(7 ^ mix64(epoch))
        for i in range(n - 1, 0, -1):
            j = mix64(key ^ i) % (i + 1)
            order[i], order[j] = order[j], order[i]
        for at in range(0, n - 7, batch):
            rows = torch.tensor(order[at:at + min(batch, n - at) // 8 * 8], device="cuda")
            b.train_step(X[rows].contiguous(), y[rows].contiguous())
    a.sync()
    b.sync()
    for p, q in zip(a.get(0), b.get(0)):
        assert np.array_equal(p, q)
    a.close()
    b.close()


@pytest.mark.parametrize("d,h1,h2,out,n", [(24, 200, 264, 1000, 264), (96, 512, 512, 4096, 1024), (8, 8, 8, 8, 8)])
def test_overlapped_steps_are_ordered(d, h1, h2, out, n):
    """A step uses a second stream: steps one after another without a wait, on
    the default stream, on another one and as a captured graph, give the bits
    that steps with a wait after each give, and the caller's stream waits for
    all of a step's work."""
    rng = np.random.default_rng(n)
    X = torch.from_numpy(rng.standard_normal((n, d)).astype(np.float32)).cuda()
    y = torch.from_numpy(rng.integers(0, out, n).astype(np.int32)).cuda()
    steps, results = 6, []
    for mode in ("wait", "default", "stream", "graph"):
        _, g = make(d, h1, h2, out, 7)
        go = lambda: g.train_step(X, y, lr=1e-3, weight_decay=0.01)
        go()
        torch.cuda.synchronize()
        if mode == "stream":
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(steps):
                    go()
        elif mode == "graph":
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                for _ in range(steps):
                    go()
            graph.replay()
        else:
            for _ in range(steps):
                go()
                if mode == "wait":
                    torch.cuda.synchronize()
        if mode == "stream":
            torch.cuda.synchronize()
        g.sync()
        results.append([np.copy(a) for a in g.get(0)])
    for other in results[1:]:
        for a, b in zip(results[0], other):
            assert np.array_equal(a, b)
