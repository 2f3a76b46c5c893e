"""The work that a user of this library has it do, as measurable cases.

listed() are the fixed cases, draw(rng) gives further ones of the same ranges,
prepare(case, seed) makes what a program holds before the call (index, network,
server, query tensors), run(state) makes the call, work(case) counts what the
call cannot do without, and exact(case, seed) is the same result in 64 bits
where it is a computed number.

A case's "kind":
  search   one batch of queries against a resident index (Index.search, or
           Index.search_host for host arrays)
  serve    a burst of requests of mixed sizes through the continuous-batching
           server (Server.submit / Server.poll)
  predict  the learned entry's prediction for a batch of queries (MLP.predict)
  train    one epoch of the learned entry's training and the trained
           parameters (MLP.train_epochs, MLP.get)
  knn      exact kNN lists of a set of vectors (knn_exact)
  prune    a fixed-degree graph from kNN lists (graph_prune)
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2507_17094_gb300 as A

ELEM = {0: 4, 1: 2, 2: 1}   # bytes per stored element: FP32, FP16, E4M3


def _search(name, **kw):
    case = dict(name=name, kind="search", n=300_000, d=96, values="unit", storage=0, rerank=0, degree=64, nq=1000,
                host=False, entry=1, n_ghost=3000, k=10, itopk=64, search_width=1, max_iters=80, dgs_discard=0.5,
                ghost_itopk=64, ghost_max_iters=12, ghost_search_width=4)
    case.update(kw)
    return case


def listed():
    return [
        # an interactive lookup: one query, half-precision rows with rerank
        _search("one_query_f16", storage=1, rerank=1, nq=1),
        # a request's worth of host queries on 8-bit rows of integer descriptors
        _search("request_61_e4m3", n=400_000, d=128, values="integer", storage=2, rerank=1, degree=32, nq=61, host=True,
                n_ghost=4000, max_iters=80, ghost_itopk=128, ghost_max_iters=32),
        # the benchmark's search: 10,000 queries, a million embeddings in FP32
        _search("batch_10k_fp32", n=1_000_000, nq=10_000, n_ghost=10_000, itopk=32, max_iters=48, dgs_discard=0.75,
                ghost_itopk=32),
        # long result lists: 100 results from half-precision integer descriptors
        _search("batch_10k_k100_f16", n=1_000_000, d=128, values="integer", storage=1, rerank=1, degree=32, nq=10_000,
                n_ghost=10_000, k=100, itopk=128, max_iters=144, ghost_itopk=256, ghost_max_iters=48),
        # high recall on mid-width FP32 vectors: wide queues in both stages
        _search("batch_256d_wide_queue", n=200_000, d=256, nq=2000, n_ghost=4000, itopk=256, max_iters=272,
                ghost_itopk=512, ghost_max_iters=64, ghost_search_width=8),
        # text-embedding width, an odd batch
        _search("batch_768d_f16", n=120_000, d=768, storage=1, rerank=1, nq=3001, n_ghost=1200),
        # online serving: many small requests at once
        dict(_search("serve_small_requests", n=500_000, storage=1, rerank=1, degree=32, n_ghost=5000, itopk=64,
                     max_iters=80, ghost_itopk=256, ghost_max_iters=48, ghost_search_width=8), kind="serve",
             requests=200, most=64, nq=0),
        # the learned entry: prediction for a benchmark batch, one training epoch
        dict(name="entry_predict", kind="predict", nq=10_000, d=96, hidden=512, out=10_000, top=8),
        dict(name="entry_train", kind="train", nq=16_384, d=96, hidden=512, out=10_000, batch=1024),
        # graph construction: a ghost set, a shard, and the pruning of a large list
        dict(name="knn_ghost_set", kind="knn", n=10_000, d=96, knn_k=32, values="unit"),
        dict(name="knn_shard", kind="knn", n=120_000, d=128, knn_k=64, values="integer"),
        dict(name="prune_500k", kind="prune", n=500_000, d=96, knn_k=96, degree=64, values="unit"),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search"] * 5 + ["serve", "predict", "train", "knn", "prune"])
    values = rng.choice(["unit", "integer"])
    if kind in ("search", "serve"):
        d = rng.choice([32, 64, 96, 100, 128, 200, 256, 300, 384, 768, 960])
        n = min(_spread(rng, 30_000, 1_000_000), 200_000_000 // d)
        degree = rng.choice([16, 32, 48, 64])
        itopk = rng.choice([16, 32, 33, 64, 100, 128, 256])
        storage = rng.randrange(3)
        nq = _spread(rng, 1, 10_000)
        # no more row bytes than the largest listed batch gathers
        nq = max(1, min(nq, 1_600_000_000 // (itopk * degree * d)))
        entry = rng.choice([0, 1, 1, 1])
        c = _search("", n=n, d=d, values=values, storage=storage, rerank=int(storage > 0 and rng.random() < 0.8),
                    degree=degree, nq=nq, host=rng.random() < 0.3, entry=entry, n_ghost=max(500, n // 100),
                    k=min(itopk, rng.choice([1, 10, 20, 100])), itopk=itopk, search_width=rng.choice([1, 1, 1, 2, 4]),
                    max_iters=itopk + 16, dgs_discard=rng.choice([0.0, 0.25, 0.5, 0.75]),
                    ghost_itopk=rng.choice([32, 64, 128, 256]), ghost_max_iters=rng.choice([12, 16, 32, 48]),
                    ghost_search_width=rng.choice([1, 2, 4, 8]))
        del c["name"]
        if kind == "serve":
            c.update(kind="serve", requests=_spread(rng, 4, 200), most=_spread(rng, 2, 64), nq=0, host=False,
                     itopk=min(itopk, 64), k=min(c["k"], 10), max_iters=80, search_width=1, d=min(d, 256))
        return c
    if kind == "predict":
        return dict(kind=kind, nq=_spread(rng, 1, 10_000), d=8 * rng.randint(4, 32), hidden=rng.choice([128, 256, 512]),
                    out=8 * _spread(rng, 64, 1250), top=rng.choice([1, 4, 8]))
    if kind == "train":
        batch = 8 * _spread(rng, 16, 128)
        return dict(kind=kind, nq=batch * rng.randint(1, 16), d=8 * rng.randint(4, 32),
                    hidden=rng.choice([128, 256, 512]), out=8 * _spread(rng, 64, 1000), batch=batch)
    if kind == "knn":
        d = rng.choice([32, 64, 96, 100, 128, 200, 256, 300])
        n = min(_spread(rng, 2000, 100_000), int(100_000 * math.sqrt(128 / d)))
        return dict(kind=kind, n=n, d=d, knn_k=rng.choice([16, 32, 48, 64, 96]), values=values)
    knn_k = rng.choice([32, 48, 64, 96])
    return dict(kind="prune", n=_spread(rng, 5000, 500_000), d=rng.choice([32, 64, 96]), knn_k=knn_k,
                degree=min(knn_k, rng.choice([16, 24, 32, 64])), values=values)


# ------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


class _Points:
    """A mixture of equal-sized Gaussian clusters (about 1,000 points each):
    unit-length vectors from touching anisotropic clusters (embeddings), or
    integers in [0, 255] (image descriptors)."""

    def __init__(self, g, n, d, values):
        self.g, self.n, self.d, self.values = g, n, d, values
        self.c = max(2, n // 1000)
        u = torch.rand((self.c, d), device="cuda", generator=g)
        if values == "unit":
            self.centers = 10.0 * u
            self.sigma = 0.5 + 3.5 * torch.rand((self.c, d), device="cuda", generator=g)
        else:
            self.centers = 255.0 * u
            self.sigma = torch.full((self.c, d), 16.0, device="cuda")

    def at(self, labels):
        out = torch.empty((labels.shape[0], self.d), device="cuda")
        for a in range(0, labels.shape[0], 1 << 18):
            lab = labels[a:a + (1 << 18)]
            x = torch.randn((lab.shape[0], self.d), device="cuda", generator=self.g)
            x = self.centers[lab] + self.sigma[lab] * x
            out[a:a + (1 << 18)] = (torch.nn.functional.normalize(x, dim=1) if self.values == "unit"
                                    else x.clamp(0, 255).round())
        return out

    def base(self):
        """The points in random order, and each cluster's members (padded with -1)."""
        perm = torch.randperm(self.n, device="cuda", generator=self.g)
        m = -(-self.n // self.c)
        members = torch.full((self.c * m,), -1, dtype=torch.int64, device="cuda")
        members[:self.n] = perm
        members = members.view(m, self.c).t().contiguous()
        labels = torch.empty(self.n, dtype=torch.int64, device="cuda")
        lab = torch.arange(self.c, device="cuda")[:, None].expand_as(members)
        labels[members[members >= 0]] = lab[members >= 0]
        return self.at(labels), members, labels

    def queries(self, nq):
        return self.at(torch.randint(0, self.c, (nq,), device="cuda", generator=self.g)).contiguous()


def _cluster_knn(x, members, knn_k):
    """Each point's nearest neighbours within its cluster (int32 n x K)."""
    out = torch.empty((x.shape[0], knn_k), dtype=torch.int32, device="cuda")
    m = members.shape[1]
    step = max(1, (1 << 25) // (m * m))
    for a in range(0, members.shape[0], step):
        mem = members[a:a + step]
        p = x[mem.clamp(min=0)]
        sq = (p * p).sum(dim=2)
        dist = sq[:, :, None] + sq[:, None, :] - 2.0 * torch.bmm(p, p.transpose(1, 2))
        dist.masked_fill_((mem < 0)[:, None, :], float("inf"))
        dist.diagonal(dim1=1, dim2=2).fill_(float("inf"))
        at = torch.topk(dist, knn_k, dim=2, largest=False).indices
        near = torch.gather(mem[:, None, :].expand(-1, m, -1), 2, at).to(torch.int32)
        out[mem[mem >= 0]] = near[mem >= 0]
    return out


def _with_bridges(g, graph, n):
    """The last eighth of every list points to random nodes (what keeps a
    graph over strongly clustered points connected)."""
    nb = max(1, graph.shape[1] // 8)
    graph[:, -nb:] = torch.randint(0, n, (graph.shape[0], nb), device="cuda", generator=g).to(torch.int32)
    return graph


def _host(t):
    a = t.cpu().numpy()
    return a.view(np.uint32) if a.dtype == np.int32 else a


def _index(case, g, points):
    x, members, _ = points.base()
    knn = _cluster_knn(x, members, min(members.shape[1] - 2, case["degree"] + case["degree"] // 2))
    graph = _with_bridges(g, A.graph_prune(knn, case["degree"]), case["n"])
    ghost = torch.sort(torch.randperm(case["n"], device="cuda", generator=g)[:case["n_ghost"]]).values
    near = torch.cdist(x[ghost], x[ghost]).fill_diagonal_(float("inf")).topk(32, dim=1, largest=False).indices
    ghost_graph = _with_bridges(g, A.graph_prune(near.to(torch.int32), 16), case["n_ghost"])
    return A.Index(_host(x), _host(graph), storage=case["storage"], ghost_ids=_host(ghost.to(torch.int32)),
                   ghost_graph=_host(ghost_graph), keep_fp32=bool(case["rerank"]) or case["storage"] == 0)


def _network(case, seed):
    """A learned-entry network over `out` ghost points whose logits follow the
    closeness of the hidden features, as training leaves them, or (train) its
    He-normal start; with the queries and their labels."""
    g = _gen(seed)
    d, h, out = case["d"], case["hidden"], case["out"]
    points = _Points(g, max(2000, out), d, "unit")
    ghosts, x = points.queries(out), points.queries(case["nq"])
    w1 = torch.randn((h, d), device="cuda", generator=g) * math.sqrt(2.0 / d)
    w2 = torch.randn((h, h), device="cuda", generator=g) * math.sqrt(2.0 / h)
    b1, b2, b3 = (torch.zeros(k, device="cuda") for k in (h, h, out))
    mean, inv_std = ghosts.mean(dim=0), 1.0 / ghosts.std(dim=0)
    if case["kind"] == "train":
        w3 = torch.randn((out, h), device="cuda", generator=g) * math.sqrt(2.0 / h)
    else:
        f = torch.relu(torch.relu(((ghosts - mean) * inv_std) @ w1.t()) @ w2.t())
        w3 = f * (2.0 * math.sqrt(h) / f.square().sum(dim=1, keepdim=True).sqrt().clamp(min=1e-6))
        w3 = w3 / math.sqrt(h) * 3.0
    labels = None
    if case["kind"] == "train":
        labels = torch.cat([torch.cdist(q, ghosts).argmin(dim=1) for q in x.split(4096)]).to(torch.int32)
    return x, labels, [w1, b1, w2, b2, w3, b3], (mean, inv_std)


def _lists(case, seed):
    g = _gen(seed)
    return _Points(g, case["n"], case["d"], case["values"]).base()


def _params(case):
    names = ("k", "itopk", "search_width", "max_iters", "dgs_discard", "entry", "ghost_itopk", "ghost_max_iters",
             "ghost_search_width", "rerank")
    return {k: case[k] for k in names}


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("search", "serve"):
        g = _gen(seed)
        points = _Points(g, case["n"], case["d"], case["values"])
        ix = _index(case, g, points)
        params = dict(_params(case), seed=seed)
        if kind == "search":
            q = points.queries(case["nq"])
            return {"kind": kind, "index": ix, "queries": q.cpu().numpy() if case["host"] else q, "params": params}
        sizes = np.random.default_rng(case["requests"]).integers(1, case["most"] + 1, case["requests"]).tolist()
        q = points.queries(sum(sizes)).cpu().numpy()
        at = np.cumsum([0] + sizes)
        srv = A.Server(ix, capacity=16_384, max_requests=256, max_params=params)
        return {"kind": kind, "server": srv, "params": params,
                "requests": [q[a:b] for a, b in zip(at[:-1], at[1:])]}
    if kind in ("predict", "train"):
        x, labels, weights, norm = _network(case, seed)
        mlp = A.MLP(case["d"], case["hidden"], case["hidden"], case["out"],
                    max_batch=case.get("batch", 8 * -(-case["nq"] // 8)))
        mlp.set_params(*(w.cpu().numpy() for w in weights))
        mlp.set_input_norm(*(v.cpu().numpy() for v in norm))
        return {"kind": kind, "mlp": mlp, "x": x, "labels": labels, "case": case}
    x, members, _ = _lists(case, seed)
    if kind == "knn":
        return {"kind": kind, "x": x, "K": case["knn_k"]}
    return {"kind": kind, "knn": _cluster_knn(x, members, case["knn_k"]), "degree": case["degree"]}


# --------------------------------------------------------------------- call
def _serve(srv, requests, params):
    done, i = {}, 0
    while len(done) < len(requests):
        while i < len(requests) and srv.submit(i, requests[i], **params):
            i += 1
        for rid, ids, dists, _ in srv.poll():
            done[rid] = (ids, dists)
    return (np.concatenate([done[j][0] for j in range(len(requests))]),
            np.concatenate([done[j][1] for j in range(len(requests))]))


def run(state):
    kind = state["kind"]
    if kind == "search":
        if isinstance(state["queries"], np.ndarray):
            return state["index"].search_host(state["queries"], **state["params"])
        ids, dists, _ = state["index"].search(state["queries"], **state["params"])
        return ids, dists
    if kind == "serve":
        return _serve(state["server"], state["requests"], state["params"])
    if kind == "predict":
        return state["mlp"].predict(state["x"], P=state["case"]["top"])
    if kind == "train":
        losses = state["mlp"].train_epochs(state["x"], state["labels"], batch=state["case"]["batch"], epochs=1, seed=5)
        return [losses] + state["mlp"].get(0)
    if kind == "knn":
        return A.knn_exact(state["x"], state["K"])
    return A.graph_prune(state["knn"], state["degree"])


# --------------------------------------------------------------------- cost
def work(case):
    kind = case["kind"]
    if kind in ("search", "serve"):
        # Per query: every queue entry is expanded once, each of its list's
        # kept neighbours (about half of them new to the search) is read, and
        # under direction-guided selection (the first 70% of the iterations)
        # its direction rows too; the ghost stage likewise.
        nq = case["nq"] if kind == "search" else case["requests"] * (case["most"] + 1) / 2
        d, deg, words = case["d"], case["degree"], -(-case["d"] // 32)
        row = d * ELEM[case["storage"]] + (4 if case["storage"] else 0)
        parents = min(case["itopk"], case["max_iters"] * case["search_width"])
        guided = 0.7 * parents if case["dgs_discard"] > 0 else 0.0
        rows = 0.5 * deg * (guided * (1.0 - case["dgs_discard"]) + parents - guided)
        b = parents * deg * 4 + guided * deg * words * 4
        if case["entry"] == 1:
            gp = min(case["ghost_itopk"], case["ghost_max_iters"] * case["ghost_search_width"])
            b += gp * 16 * 4
            rows += 0.5 * 16 * gp
        b += rows * row + (case["itopk"] * d * 4 if case["rerank"] else 0) + d * 4 + case["k"] * 8
        return {"bytes": nq * b, "flops": nq * rows * 3 * d}
    if kind == "predict":
        d, h, o, nq = case["d"], case["hidden"], case["out"], case["nq"]
        return {"bytes": 4 * nq * d + 2 * (d * h + h * h + h * o) + 4 * (2 * h + o) + nq * (4 * case["top"] + 4),
                "flops": 2 * nq * (d * h + h * h + h * o)}
    if kind == "train":
        d, h, o, nq = case["d"], case["hidden"], case["out"], case["nq"]
        weights, steps = d * h + h * h + h * o + 2 * h + o, -(-nq // case["batch"])
        # masters and two moments read and written each step; inputs and labels once
        return {"bytes": steps * weights * 24 + nq * (4 * d + 4) + 4 * weights,
                "flops": 6 * nq * (d * h + h * h + h * o)}
    if kind == "knn":
        n, d = case["n"], case["d"]
        return {"bytes": 4 * n * (d + case["knn_k"]), "flops": 2 * n * n * d}
    n, k = case["n"], case["knn_k"]
    return {"bytes": 4 * n * (k + case["degree"]), "flops": n * k * k}


# -------------------------------------------------------------------- exact
def _mix64(x):
    m = (1 << 64) - 1
    z = (x + 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _epoch_order(n, seed, epoch):
    order, key = list(range(n)), _mix64(seed ^ _mix64(epoch))
    for i in range(n - 1, 0, -1):
        j = _mix64(key ^ i) % (i + 1)
        order[i], order[j] = order[j], order[i]
    return order


def exact(case, seed):
    if case["kind"] not in ("predict", "train"):
        return None   # ids and the distances of the ids that a search finds
    x, labels, weights, (mean, inv_std) = _network(case, seed)
    w = [t.double() for t in weights]
    x = (x.double() - mean.double()) * inv_std.double()
    if case["kind"] == "predict":
        top = []
        for q in x.split(2048):
            z = torch.relu(torch.relu(q @ w[0].t() + w[1]) @ w[2].t() + w[3]) @ w[4].t() + w[5]
            top.append(torch.softmax(z, dim=1).max(dim=1).values)
        return [None, torch.cat(top)]
    m, v = [torch.zeros_like(t) for t in w], [torch.zeros_like(t) for t in w]
    n, batch, losses = case["nq"], case["batch"], []
    order = torch.tensor(_epoch_order(n, 5, 0), device="cuda")
    for step, rows in enumerate(order.split(batch), 1):
        q, y = x[rows], labels[rows].long()
        h1 = torch.relu(q @ w[0].t() + w[1])
        h2 = torch.relu(h1 @ w[2].t() + w[3])
        z = h2 @ w[4].t() + w[5]
        losses.append(torch.nn.functional.cross_entropy(z, y))
        dz = torch.softmax(z, dim=1)
        dz[torch.arange(len(y), device="cuda"), y] -= 1.0
        dz /= len(y)
        da2 = (dz @ w[4]) * (h2 > 0)
        da1 = (da2 @ w[2]) * (h1 > 0)
        grads = [da1.t() @ q, da1.sum(dim=0), da2.t() @ h1, da2.sum(dim=0), dz.t() @ h2, dz.sum(dim=0)]
        for i, gr in enumerate(grads):
            m[i] = 0.9 * m[i] + 0.1 * gr
            v[i] = 0.999 * v[i] + 0.001 * gr * gr
            w[i] = w[i] - 1e-3 * (m[i] / (1 - 0.9 ** step)) / ((v[i] / (1 - 0.999 ** step)).sqrt() + 1e-8)
    return [torch.stack(losses).mean().reshape(1)] + w
