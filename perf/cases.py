"""The work a user of this framework has it do, as timed cases.

Online path (what a serving program calls for every batch): entry selection by the two-tower
model, then the batched beam search, over every storage type, metric and batch size in use.
Offline path (what an index builder calls once per data set, and again whenever the data
change): the proximity graph, exact k-NN ground truth, hub clustering, the label search and the
training step of the entry model.

Data follow the framework's own synthetic laws (anisotropic Gaussian mixtures under a global
spectrum, queries shifted and reweighted), drawn on the GPU from the seed.
"""
import numpy as np
import torch

from paper_2506_15986_gb300 import ann

DEV = "cuda:0"
DTYPES = {"u8": ann.U8, "f32": ann.F32, "f16": ann.F16, "i8s": ann.I8S}


def listed():
    return [
        # the parity configuration: 100 uint8 queries from the medoid; few queries, so the
        # latency of one query's chain of steps counts
        dict(name="search_u8_100q", kind="search", dtype="u8", metric="l2", n=10_000, dim=128, R=32, nq=100,
             k=10, L=64, W=1, entry="medoid", hubs=0, l_hub=0, seeds=1, tuned=False, rerank=False, mixed=False),
        # one online query: launches and the latency of one query's steps
        dict(name="online_1q", kind="search", dtype="f32", metric="l2", n=200_000, dim=128, R=32, nq=1,
             k=10, L=64, W=4, entry="exhaustive", hubs=1024, l_hub=0, seeds=1, tuned=False, rerank=False,
             mixed=False),
        # the headline: a batch of 10,000 shifted queries, learned entry by exhaustive hub scoring,
        # the sizes the autotuner picks there (rows larger than L2)
        dict(name="search_shift_10k", kind="search", dtype="f32", metric="l2", n=400_000, dim=128, R=32,
             nq=10_000, k=10, L=93, W=4, entry="exhaustive", hubs=1024, l_hub=0, seeds=1, tuned=True,
             rerank=False, mixed=False),
        # high-dimensional rows stored as FP16, final pools reranked in FP32, k = 100
        dict(name="search_960d_f16_rerank", kind="search", dtype="f16", metric="l2", n=60_000, dim=960, R=48,
             nq=1_000, k=100, L=256, W=2, entry="medoid", hubs=0, l_hub=0, seeds=1, tuned=False, rerank=True,
             mixed=False),
        # maximum inner product, out-of-distribution queries, entry by the hub-graph walk
        dict(name="search_ip_nav", kind="search", dtype="f32", metric="ip", n=200_000, dim=200, R=32, nq=10_000,
             k=10, L=256, W=4, entry="nav", hubs=4096, l_hub=32, seeds=1, tuned=False, rerank=False, mixed=False),
        # a stream batch of 100,000 queries with per-query k and L in one persistent launch, 2-hub
        # seed sets out of 16,384 hubs
        dict(name="search_mixed_100k", kind="search", dtype="f32", metric="l2", n=200_000, dim=96, R=32,
             nq=100_000, k=100, L=512, W=4, entry="exhaustive", hubs=16_384, l_hub=0, seeds=2, tuned=False,
             rerank=False, mixed=True),
        # exact ground truth of 10,000 queries (recall measurement, label targets)
        dict(name="knn_truth", kind="knn", dtype="f32", metric="l2", n=300_000, dim=128, nq=10_000, k=10),
        # the proximity graph of one shard's rows: exact 64-NN, pruning to 32, medoid, repair
        dict(name="build_graph_50k", kind="build", dtype="f32", n=50_000, dim=128, K=64, R=32),
        # label costs of 4,096 training queries from their 64 nearest hubs each, and the label rule
        dict(name="hub_labels", kind="labels", n=200_000, dim=128, R=32, nq=4_096, M=64, hubs=1024, L=64, W=1),
        # one training step at the method's batch size
        dict(name="train_step", kind="train", dim=128, hubs=1024, batch=8192, M=64, rows=100_000),
        # flat k-means on a sample, then the hub of every cluster
        dict(name="kmeans_hubs", kind="kmeans", n=200_000, dim=128, m=65_536, hubs=1024, iters=5),
        # hierarchical balanced k-means hubs (Algorithm 2)
        dict(name="hbkm_hubs", kind="hbkm", n=60_000, dim=128, k=32, levels=2, T=10, lam=1.0),
    ]


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "search", "knn", "build", "labels", "train", "train", "kmeans",
                       "hbkm"])
    if kind == "search":
        dtype = rng.choice(["u8", "f32", "f32", "f32", "f16", "i8s"])
        metric = "l2" if dtype == "u8" else rng.choice(["l2", "l2", "ip"])
        dim = rng.choice([16, 32, 48, 64, 96, 112, 128] if dtype == "u8" else
                         [16, 64, 96, 100, 128, 128, 200, 256, 384, 960] if dtype in ("f32", "i8s") else
                         [16, 64, 96, 104, 128, 128, 200, 256, 384, 960])
        n = _log(rng, 5_000, 50_000 if dim > 400 else 200_000)
        L = _log(rng, 16, 512)
        nq = _log(rng, 1, 50_000 if dim <= 128 else 2_000 if dim > 400 else 10_000)
        entry = rng.choice(["medoid", "exhaustive", "nav"] if dim <= 512 else ["medoid"])
        R = rng.choice([16, 24, 32, 32, 48])
        return dict(kind=kind, dtype=dtype, metric=metric, n=n, dim=dim, R=R, nq=nq,
                    k=max(1, min(L, rng.choice([1, 10, 10, 100, 37]))), L=L, W=rng.randint(1, 2 if R > 32 else 4),
                    entry=entry, hubs=0 if entry == "medoid" else min(n // 4, _log(rng, 100, 16_384)),
                    l_hub=rng.choice([16, 32, 64, 96]) if entry == "nav" else 0,
                    seeds=1 if entry == "medoid" else rng.choice([1, 1, 2, 4]), tuned=rng.random() < 0.3,
                    rerank=dtype in ("f16", "i8s") and rng.random() < 0.6, mixed=rng.random() < 0.2)
    if kind == "knn":
        dtype = rng.choice(["f32", "f32", "u8"])
        return dict(kind=kind, dtype=dtype, metric="ip" if dtype == "f32" and rng.random() < 0.3 else "l2",
                    n=_log(rng, 3_000, 300_000), dim=rng.choice([16, 64, 96, 128, 200, 960] if dtype == "f32" else
                                                                [16, 48, 128]),
                    nq=_log(rng, 10, 10_000), k=rng.choice([1, 10, 32, 33, 64, 100]))
    if kind == "build":
        dtype = rng.choice(["f32", "f32", "u8"])
        return dict(kind=kind, dtype=dtype, n=_log(rng, 3_000, 50_000), dim=rng.choice([64, 96, 128, 200] if dtype == "f32"
                                                                                      else [64, 128]),
                    K=64, R=rng.choice([16, 32, 48]))
    if kind == "labels":
        return dict(kind=kind, n=_log(rng, 20_000, 200_000), dim=rng.choice([96, 128, 200]), R=32,
                    nq=_log(rng, 100, 4_096), M=rng.choice([16, 33, 64]), hubs=_log(rng, 128, 4_096),
                    L=rng.choice([32, 64]), W=1)
    if kind == "train":
        return dict(kind=kind, dim=rng.choice([64, 96, 128, 200, 512]), hubs=_log(rng, 100, 16_384),
                    batch=_log(rng, 500, 8192), M=rng.choice([16, 50, 64]), rows=rng.choice([8192, 50_000]))
    if kind == "kmeans":
        m = _log(rng, 8_000, 65_536)
        return dict(kind=kind, n=m + _log(rng, 1, 134_000), dim=rng.choice([64, 96, 128, 200]), m=m,
                    hubs=_log(rng, 64, 2_048), iters=rng.choice([3, 5]))
    k, levels = rng.choice([(32, 2), (16, 2), (8, 3), (4, 5)])
    return dict(kind="hbkm", n=_log(rng, 5_000, 60_000), dim=rng.choice([64, 96, 128, 200]), k=k, levels=levels, T=10,
                lam=rng.choice([0.5, 1.0]))


class Index:
    """An index handle that goes with its state."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        ann.ann_free_index(self.handle)


class Trainer:
    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        ann.ann_trainer_free(self.handle)


def _mixture(gen, n, dim, nq, dtype="f32", metric="l2"):
    """(base, queries) on the GPU: an anisotropic mixture under the spectrum (1 + i)^-0.5, about
    1,000 rows a component; queries from the same components moved by half a standard deviation,
    5 % of the components carrying 80 % of them.  Unit rows for the inner product; rounded and
    clipped to bytes for uint8."""
    rand = lambda *s: torch.randn(*s, generator=gen, device=DEV)  # noqa: E731
    nc = max(10, n // 1000)
    if dtype == "u8":
        c = torch.rand(nc, dim, generator=gen, device=DEV) * 192 + 32
        s = torch.full((nc, dim), 40.0, device=DEV)
    else:
        g = (1.0 + torch.arange(dim, device=DEV)) ** -0.5
        c = rand(nc, dim) * g
        s = torch.exp(0.5 * rand(nc, dim)) * g
    at = torch.randint(nc, (n,), generator=gen, device=DEV)
    base = rand(n, dim).mul_(s[at]).add_(c[at])
    hot = max(1, nc // 20)
    qa = torch.where(torch.rand(nq, generator=gen, device=DEV) < 0.8,
                     torch.randint(hot, (nq,), generator=gen, device=DEV),
                     torch.randint(nc, (nq,), generator=gen, device=DEV))
    q = rand(nq, dim).mul_(s[qa]).add_((c + 0.5 * s * rand(nc, dim))[qa])
    if dtype == "u8":
        return base.round_().clamp_(0, 255).to(torch.uint8), q.round_().clamp_(0, 255).to(torch.uint8)
    if metric == "ip":
        base, q = torch.nn.functional.normalize(base), torch.nn.functional.normalize(q)
    return base.contiguous(), q.contiguous()


def _graph(base, R, K=64):
    n, dim = base.shape
    graph = torch.empty((n, R), dtype=torch.int32, device=DEV)
    dt = ann.U8 if base.dtype == torch.uint8 else ann.F32
    med, _ = ann.ann_build_graph(base, n, dim, dt, K, R, 1.0, graph)
    return graph, med


def _tower(gen, dim):
    W1 = torch.randn(dim, 256, generator=gen, device=DEV) * (2.0 / dim) ** 0.5
    W2 = torch.randn(256, 64, generator=gen, device=DEV) * (2.0 / 256) ** 0.5
    return W1, torch.zeros(256, device=DEV), W2, torch.zeros(64, device=DEV)


def _ints(t):
    return t.to(torch.int32).contiguous()


def _prepare_search(c, gen):
    base, q = _mixture(gen, c["n"], c["dim"], c["nq"], c["dtype"], c["metric"])
    graph, med = _graph(base, c["R"], max(64, c["R"]))
    metric = ann.IP if c["metric"] == "ip" else ann.L2
    n, dim = base.shape
    rows = base
    if c["dtype"] == "f16":
        rows = base.half()
    elif c["dtype"] == "i8s":
        rows = torch.empty((n, ann.ann_i8s_row_bytes(dim)), dtype=torch.uint8, device=DEV)
        ann.ann_quantize_i8s(base, n, dim, rows)
    idx = Index(ann.ann_index_create(rows, graph, med, DTYPES[c["dtype"]], metric, n=n, dim=dim, degree=c["R"],
                                     base_f32=base if c["rerank"] else None))
    if c["hubs"]:
        # the tower's initial weights, and hub embeddings that are the tower's output on the hubs' rows
        W1, b1, W2, b2 = _tower(gen, dim)
        hubs = torch.randperm(n, generator=gen, device=DEV)[:c["hubs"]]
        x = base[hubs].float()
        emb = (torch.relu(x @ W1 + b1) @ W2 + b2).contiguous()
        ann.ann_set_entry_model(idx.handle, dim, W1, b1, W2, b2, _ints(hubs), emb, 16)
        if c["entry"] == "nav":
            ann.ann_build_hub_graph(idx.handle, 8, 16)
    d_k = d_L = None
    if c["mixed"]:
        choice = torch.tensor([1, min(10, c["k"]), c["k"]], device=DEV)
        d_k = _ints(choice[torch.randint(3, (c["nq"],), generator=gen, device=DEV)])
        lo = torch.clamp(d_k, min=min(32, c["L"]))
        d_L = _ints(lo + torch.floor(torch.rand(c["nq"], generator=gen, device=DEV) * (c["L"] + 1 - lo)))
    flags = ann.SEARCH_RERANK if c["rerank"] else 0
    knobs = {}
    if c["tuned"]:
        knobs = dict(hash_bits=-1, stage_rows=8)
        if c["entry"] != "medoid":
            flags |= ann.SEARCH_GROUP_ENTRIES
    p = ann.search_params(c["k"], c["L"], W=c["W"], d_k=d_k, d_L=d_L, n_entries=c["seeds"] if c["hubs"] else 0,
                          flags=flags, **knobs)
    nq = c["nq"]
    return dict(case=c, idx=idx, q=q, p=p, keep=(d_k, d_L),
                entry=torch.empty((nq, c["seeds"]), dtype=torch.int32, device=DEV) if c["hubs"] else None,
                ids=torch.empty((nq, c["k"]), dtype=torch.int32, device=DEV),
                dists=torch.empty((nq, c["k"]), dtype=torch.int32 if c["dtype"] == "u8" else torch.float32, device=DEV))


def prepare(case, seed):
    c = case
    gen = torch.Generator(device=DEV).manual_seed(seed)
    kind = c["kind"]
    if kind == "search":
        return _prepare_search(c, gen)
    if kind == "knn":
        base, q = _mixture(gen, c["n"], c["dim"], c["nq"], c["dtype"], c["metric"])
        return dict(case=c, base=base, q=q, ids=torch.empty((c["nq"], c["k"]), dtype=torch.int32, device=DEV),
                    dists=torch.empty((c["nq"], c["k"]), device=DEV,
                                      dtype=torch.int32 if c["dtype"] == "u8" else torch.float32))
    if kind == "build":
        base, _ = _mixture(gen, c["n"], c["dim"], 1, c["dtype"])
        return dict(case=c, base=base, graph=torch.empty((c["n"], c["R"]), dtype=torch.int32, device=DEV))
    if kind == "labels":
        base, q = _mixture(gen, c["n"], c["dim"], c["nq"])
        graph, med = _graph(base, c["R"])
        idx = Index(ann.ann_index_create(base, graph, med, ann.F32))
        hubs = torch.randperm(c["n"], generator=gen, device=DEV)[:c["hubs"]]
        shape = (c["nq"], c["M"])
        cand = torch.empty(shape, dtype=torch.int32, device=DEV)
        ann.ann_knn(base[hubs].contiguous(), c["hubs"], c["dim"], ann.F32, ann.L2, q, c["nq"], c["M"], cand,
                    torch.empty(shape, device=DEV))
        target = torch.empty((c["nq"], 1), dtype=torch.int32, device=DEV)
        ann.ann_knn(base, c["n"], c["dim"], ann.F32, ann.L2, q, c["nq"], 1, target,
                    torch.empty((c["nq"], 1), device=DEV))
        return dict(case=c, idx=idx, q=q, cand=cand, target=target, hubs=_ints(hubs),
                    evals=torch.empty(shape, dtype=torch.int32, device=DEV),
                    hops=torch.empty(shape, dtype=torch.int32, device=DEV),
                    labels=torch.empty(shape, dtype=torch.int8, device=DEV),
                    best=torch.empty(c["nq"], dtype=torch.int32, device=DEV))
    if kind == "train":
        H, D, nt, M = c["hubs"], c["dim"], c["rows"], min(c["M"], c["hubs"])
        base, q = _mixture(gen, max(10_000, H), D, nt)
        W1, b1, W2, b2 = _tower(gen, D)
        E = torch.relu(base[:H] @ W1 + b1) @ W2 + b2
        # M different listed hubs a query; about five positives among them, none for one query in
        # seven (its neighbours were never reached), the rest negative or unused
        first = torch.randint(H, (nt, 1), generator=gen, device=DEV)
        cand = (first + torch.arange(M, device=DEV) * max(1, H // M)) % H
        u = torch.rand(nt, M, generator=gen, device=DEV)
        lab = torch.where(u < 5.0 / M, 1, torch.where(u < 0.7, -1, 0))
        lab[torch.rand(nt, generator=gen, device=DEV) < 0.15] = -1
        rows = torch.randperm(nt, generator=gen, device=DEV)[:min(c["batch"], nt)]
        trainer = Trainer(ann.ann_trainer_create(D, W1, b1, W2, b2, E.contiguous(), len(rows)))
        return dict(case=c, trainer=trainer, q=q, rows=_ints(rows), cand=_ints(cand),
                    lab=lab.to(torch.int8).contiguous(), M=M, start=(W1, b1, W2, b2, E),
                    grads=[torch.empty_like(t, memory_format=torch.contiguous_format) for t in (W1, b1, W2, b2, E)])
    if kind == "kmeans":
        base, _ = _mixture(gen, c["n"], c["dim"], 1)
        rng = np.random.Generator(np.random.PCG64(seed))
        sample = np.sort(rng.choice(c["n"], size=c["m"], replace=False)).astype(np.int64)
        init = rng.permutation(c["m"])[:c["hubs"]].astype(np.int32)
        return dict(case=c, base=base, sample=sample, init=init,
                    cent=torch.empty((c["hubs"], c["dim"]), device=DEV),
                    hubs=torch.empty(c["hubs"], dtype=torch.int32, device=DEV),
                    assign=torch.empty(c["n"], dtype=torch.int32, device=DEV))
    base, _ = _mixture(gen, c["n"], c["dim"], 1)
    keys = torch.randint(-2 ** 31, 2 ** 31, (c["n"],), generator=gen, device=DEV)
    nc = c["k"] ** c["levels"]
    return dict(case=c, base=base, keys=_ints(keys), hubs=torch.empty(nc, dtype=torch.int32, device=DEV),
                cent=torch.empty((nc, c["dim"]), device=DEV), label=torch.empty(c["n"], dtype=torch.int32, device=DEV))


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "search":
        h, nq = s["idx"].handle, c["nq"]
        if c["hubs"]:
            mode = ann.ENTRY_LEARNED_NAV if c["entry"] == "nav" else ann.ENTRY_LEARNED_EXHAUSTIVE
            ann.ann_select_entries(h, s["q"], nq, mode, c["l_hub"], c["seeds"], s["entry"])
        ann.ann_search_batch(h, s["q"], nq, s["entry"], s["p"], s["ids"], s["dists"])
        return dict(ids=s["ids"], dists=s["dists"], entry=s["entry"])
    if kind == "knn":
        ann.ann_knn(s["base"], c["n"], c["dim"], DTYPES[c["dtype"]], ann.IP if c["metric"] == "ip" else ann.L2,
                    s["q"], c["nq"], c["k"], s["ids"], s["dists"])
        return dict(ids=s["ids"], dists=s["dists"])
    if kind == "build":
        med, rep = ann.ann_build_graph(s["base"], c["n"], c["dim"], DTYPES[c["dtype"]], c["K"], c["R"], 1.0, s["graph"])
        return dict(graph=s["graph"], medoid=med, repairs=rep)
    if kind == "labels":
        ann.ann_hub_costs(s["idx"].handle, s["q"], c["nq"], s["target"], s["cand"], c["M"], s["hubs"], c["L"],
                          s["evals"], s["hops"], W=c["W"])
        ann.ann_hub_labels(s["evals"], s["hops"], s["cand"], c["nq"], c["M"], 3, 15, s["labels"], s["best"])
        return dict(evals=s["evals"], hops=s["hops"], labels=s["labels"], best=s["best"])
    if kind == "train":
        t = s["trainer"].handle
        loss = ann.ann_trainer_step(t, s["q"], s["rows"], len(s["rows"]), s["cand"], s["lab"], s["M"])
        ann.ann_trainer_get(t, *s["grads"], gradients=True)
        return dict(loss=torch.tensor(loss, dtype=torch.float32), grads=s["grads"])
    if kind == "kmeans":
        obj = ann.ann_kmeans(s["base"], c["n"], c["dim"], ann.F32, s["sample"], c["hubs"], s["init"], c["iters"],
                             s["cent"])
        ann.ann_assign_hubs(s["base"], c["n"], c["dim"], ann.F32, s["cent"], c["hubs"], s["hubs"], s["assign"])
        return dict(objective=obj, centroids=s["cent"], hubs=s["hubs"], assign=s["assign"])
    ann.ann_hbkm(s["base"], c["n"], c["dim"], c["k"], c["levels"], c["lam"], c["T"], s["keys"], s["hubs"], s["cent"],
                 s["label"])
    return dict(hubs=s["hubs"], centroids=s["cent"], label=s["label"])


def work(case):
    c = case
    kind = c["kind"]
    es = {"u8": 1, "f32": 4, "f16": 2, "i8s": 1}[c.get("dtype", "f32")]
    if kind == "search":
        # a search scores about 11 rows for every place of its pool (measured over the configurations
        # here), at most all of them; with per-query L the mean place count is about half of the largest
        places = (c["L"] + min(32, c["L"])) / 2 if c["mixed"] else c["L"]
        rows = c["nq"] * min(c["n"], 11 * places)
        total = rows * c["dim"] * es + c["nq"] * (c["dim"] * (1 if c["dtype"] == "u8" else 4) + 8 * c["k"])
        if c["rerank"]:
            total += c["nq"] * c["L"] * c["dim"] * 4
        flops = 3 * rows * c["dim"]
        if c["hubs"]:
            scored = c["hubs"] if c["entry"] == "exhaustive" else min(c["hubs"], 8 * c["l_hub"])
            flops += 2 * c["nq"] * (c["dim"] * 256 + 256 * 64 + scored * 64)
        return dict(bytes=total, flops=flops)
    if kind == "knn":
        return dict(bytes=(c["n"] + c["nq"]) * c["dim"] * es + c["nq"] * c["k"] * 8,
                    flops=2 * c["n"] * c["nq"] * c["dim"])
    if kind == "build":
        return dict(bytes=c["n"] * (c["dim"] * es + 4 * c["R"]), flops=2 * c["n"] ** 2 * c["dim"])
    if kind == "labels":
        # a label search ends where its target is found, about half of a whole search
        rows = c["nq"] * c["M"] * min(c["n"], 5 * c["L"])
        return dict(bytes=rows * c["dim"] * 4 + c["nq"] * c["M"] * 13, flops=3 * rows * c["dim"])
    if kind == "train":
        B, D, H = min(c["batch"], c["rows"]), c["dim"], c["hubs"]
        tower, params = D * 256 + 256 * 64, D * 256 + 256 * 64 + 320 + H * 64
        return dict(bytes=B * (4 * D + 5 * c["M"]) + 4 * params * 8,
                    flops=6 * B * (tower + H * 64) - 2 * B * D * 256)
    if kind == "kmeans":
        return dict(bytes=(c["m"] + c["n"]) * c["dim"] * 4, flops=2 * c["hubs"] * c["dim"] * (c["m"] * c["iters"] + c["n"]))
    return dict(bytes=c["n"] * c["dim"] * 4, flops=3 * c["n"] * c["dim"] * c["levels"] * (c["T"] * c["k"] + 1))


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "knn" and c["dtype"] == "f32":
        s = prepare(c, seed)
        x, n2 = s["base"].double(), None
        if c["metric"] == "l2":
            n2 = (x * x).sum(1)
        out = []
        for q in s["q"].double().split(256):
            d = -(q @ x.T)
            if n2 is not None:
                d = 2 * d + n2 + (q * q).sum(1, keepdim=True)
            near = d.topk(c["k"], largest=False).indices
            v = x[near]
            d = ((v - q[:, None]) ** 2).sum(2) if n2 is not None else -(v * q[:, None]).sum(2)
            out.append(d.sort(1).values)
        return dict(ids=None, dists=torch.cat(out))
    if kind == "train":
        s = prepare(c, seed)
        W1, b1, W2, b2, E = p = [t.double().requires_grad_() for t in s["start"]]
        rows = s["rows"].long()
        x, cand, lab = s["q"][rows].double(), s["cand"][rows].long(), s["lab"][rows]
        full = torch.full((len(rows), c["hubs"]), -1, dtype=torch.int8, device=DEV).scatter_(1, cand, lab)
        unit = torch.nn.functional.normalize
        score = unit(torch.relu(x @ W1 + b1) @ W2 + b2) @ unit(E).T / 0.07
        lse = score.masked_fill(full == 0, -torch.inf).logsumexp(1)
        pos = full > 0
        npos = pos.sum(1)
        ok = npos > 0
        loss = (lse - (score * pos).sum(1) / npos.clamp(min=1))[ok].mean()
        grads = torch.autograd.grad(loss, p)
        return dict(loss=loss.detach(), grads=list(grads))
    if kind == "kmeans":
        s = prepare(c, seed)
        x = s["base"][torch.from_numpy(s["sample"]).to(DEV)].double()
        cent = x[torch.from_numpy(s["init"]).long().to(DEV)].clone()
        objective = []
        for _ in range(c["iters"]):
            d = torch.cat([(v * v).sum(1, keepdim=True) - 2 * v @ cent.T + (cent * cent).sum(1) for v in x.split(8192)])
            at = d.argmin(1)
            dist = ((x - cent[at]) ** 2).sum(1)
            objective.append(dist.sum())
            count = torch.bincount(at, minlength=c["hubs"])
            mean = torch.zeros_like(cent).index_add_(0, at, x) / count.clamp(min=1)[:, None]
            empty = (count == 0).nonzero().flatten()
            mean[empty] = x[dist.sort(descending=True, stable=True).indices[:len(empty)]]
            cent = mean
        return dict(objective=torch.stack(objective), centroids=cent, hubs=None, assign=None)
    # the other outputs are whole numbers, or follow a search's own choices
    return None
