"""The work that a program has this framework do, as cases that can be timed.

Four kinds of call, each through the public Python binding (hnsw.py):
  search  K-NN search of a batch on a resident index (hnsw_search_ex)
  insert  a saved graph made resident, extended by new elements and saved
          again (hnsw_upload_index, hnsw_reserve, hnsw_insert,
          hnsw_index_to_blob)
  train   training of the learned-stop network on recorded check steps
          (hnsw_stop_train: forward, backward, Adam)
  merge   the top-k merge of per-shard answers (hnsw_merge_topk)

Searches run on three resident graphs with the shapes of the framework's own
workloads (synth.py): SIFT-shaped (128 integer coordinates, squared L2, 1,000
clusters), GloVe-shaped (100 coordinates, unit vectors, cosine, Zipf-weighted
clusters) and clustered low-dimensional points (8 coordinates, squared L2).
A program that serves searches builds and uploads its graph once and keeps
it, so a graph and its resident indexes are made at their first use in a
process and shared by every state; the queries are made from the seed.
Graphs are built with one host thread, which makes them a function of the
data alone.
"""
from __future__ import annotations

import math
import struct

import numpy as np
import torch

from paper_1603_09320_gb300 import hnsw, stopnet

# elements, dimension, metric, M, efConstruction, and the distinct elements
# that a search scores per layer-0 expansion (counted with a visited set that
# forgets nothing), which sizes work()
GRAPHS = {
    "sift": dict(n=1_000_000, d=128, metric=hnsw.L2SQ, M=16, efc=100, scored=13.3),
    "glove": dict(n=400_000, d=100, metric=hnsw.COSINE, M=16, efc=100, scored=11.5),
    "lowd": dict(n=2_000_000, d=8, metric=hnsw.L2SQ, M=12, efc=100, scored=5.3),
    # the graph that insertions extend
    "sift20k": dict(n=20_000, d=128, metric=hnsw.L2SQ, M=16, efc=200, scored=14.0),
}
COORD_BYTES = {"f32": 4, "bf16": 2, "f16": 2, "fp8": 1}
INSERT_MAX, TRAIN_MAX, MERGE_MAX = 2_000, 1_000_000, 100_000


def listed():
    s = dict(kind="search", rerank=False, stop=False, host=False)
    r = dict(s, rerank=True)
    return [
        # one interactive query, plain fp32: only latency counts
        dict(s, name="sift_f32_one", graph="sift", storage="f32", n=1, k=10, ef=64),
        # a small ragged request from host buffers, as an application server sends it
        dict(r, name="sift_bf16r_77_host", graph="sift", storage="bf16", n=77, k=10, ef=50, host=True),
        # the headline batch: the smallest ef at recall@10 >= 0.95, 16-bit rows with the exact rerank
        dict(r, name="sift_bf16r_10000", graph="sift", storage="bf16", n=10_000, k=10, ef=50),
        # the same batch on plain fp32 rows
        dict(s, name="sift_f32_10000", graph="sift", storage="f32", n=10_000, k=10, ef=50),
        # a medium odd-sized batch on the smallest rows
        dict(r, name="sift_fp8r_2999", graph="sift", storage="fp8", n=2_999, k=10, ef=54),
        # the learned early stop deciding when each search ends
        dict(r, name="sift_bf16r_stop_10000", graph="sift", storage="bf16", n=10_000, k=10, ef=80, stop=True),
        # a serving request that wants many neighbours: k = 100, plain fp32, cosine
        dict(s, name="glove_f32_k100_1000", graph="glove", storage="f32", n=1_000, k=100, ef=256),
        # high recall on hard angular data: the widest beam, the largest search
        dict(r, name="glove_bf16r_wide_10000", graph="glove", storage="bf16", n=10_000, k=10, ef=498),
        # bulk look-ups of low-dimensional points, short beams
        dict(s, name="lowd_f32_100000", graph="lowd", storage="f32", n=100_000, k=10, ef=20),
        # continuous indexing: a batch of new elements into a graph loaded from a file
        dict(kind="insert", name="insert_1000", n=1_000),
        # training the learned stop on recorded check steps
        dict(kind="train", name="train_200000", n=200_000, epochs=2, batch=4096),
        # the exchange step of data-sharded search
        dict(kind="merge", name="merge_8x10000_k10", shards=8, n=10_000, k=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search"] * 7 + ["insert", "train", "merge"])
    if kind == "insert":
        return dict(kind=kind, n=_log_int(rng, 50, INSERT_MAX))
    if kind == "train":
        return dict(kind=kind, n=_log_int(rng, 5_000, TRAIN_MAX), epochs=rng.randint(1, 2),
                    batch=128 * rng.choice([8, 16, 32, 64]))
    if kind == "merge":
        k = _log_int(rng, 1, 200)
        return dict(kind=kind, shards=rng.randint(2, 32), n=_log_int(rng, 1, MERGE_MAX // k), k=k)
    graph = rng.choice(["sift", "sift", "glove", "lowd"])
    storage, rerank = rng.choice({
        "sift": [("f32", False), ("bf16", True), ("bf16", False), ("fp8", True), ("f16", True)],
        "glove": [("f32", False), ("bf16", True), ("bf16", False)],
        "lowd": [("f32", False), ("f16", True)]}[graph])
    k = rng.choice([1, 10, 10, 10, 100])
    ef = _log_int(rng, max(k, 10), 498)
    n = _log_int(rng, 1, min(100_000 if graph == "lowd" else 10_000, 2_000_000 // ef))
    return dict(kind=kind, graph=graph, storage=storage, rerank=rerank, n=n, k=k, ef=ef,
                stop=graph == "sift" and storage == "bf16" and rng.random() < 0.3, host=rng.random() < 0.2)


# ---- data --------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _points(graph, seed, n, cluster_share=0.95):
    """n points of a graph's distribution (float32, on the GPU)."""
    d = GRAPHS[graph]["d"]
    fixed, g = _gen(7), _gen(seed)
    opt = dict(device="cuda", dtype=torch.float32)
    if graph.startswith("sift"):
        centre = 255.0 * torch.rand((1000, d), generator=fixed, **opt)
        sigma = 10.0 + 30.0 * torch.rand((1000, 1), generator=fixed, **opt)
        c = torch.randint(0, 1000, (n,), generator=g, device="cuda")
        x = centre[c] + sigma[c] * torch.randn((n, d), generator=g, **opt)
        return x.clamp_(0.0, 255.0).round_()
    if graph == "glove":
        centre = torch.randn((500, d), generator=fixed, **opt)
        w = 1.0 / torch.arange(1, 501, device="cuda", dtype=torch.float64) ** 1.1
        u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        c = torch.searchsorted(torch.cumsum(w / w.sum(), 0), u).clamp_(max=499)
        x = centre[c] + 0.5 * torch.randn((n, d), generator=g, **opt)
        return x / x.square().sum(1, keepdim=True).sqrt()
    centre = torch.rand((10_000, d), generator=fixed, **opt)
    c = torch.randint(0, 10_000, (n,), generator=g, device="cuda")
    x = centre[c] + 1e-3 * torch.randn((n, d), generator=g, **opt)
    far = torch.rand((n, d), generator=g, **opt)
    return torch.where(torch.rand((n, 1), generator=g, **opt) < cluster_share, x, far)


def _levels(seed, n):
    x = np.random.Generator(np.random.Philox(key=seed)).integers(0, 2**53, size=n, dtype=np.int64)
    return (x + 1.0) / float(2**53)


# graphs and resident indexes that the process keeps
_blobs, _indexes = {}, {}


def _blob(graph):
    if graph not in _blobs:
        g = GRAPHS[graph]
        x = _points(graph, 1, g["n"]).cpu().numpy()
        _blobs[graph] = hnsw.build_graph_gpu(x, _levels(3, g["n"]), metric=g["metric"], M=g["M"],
                                             ef_construction=g["efc"], n_threads=1)
    return _blobs[graph]


def _stop_model():
    """(norm, weights) of a network that stops a search when about 20
    expansions in a row have left its k nearest as they were (feature 4 is
    log1p of that count); the other hidden units carry ordinary weights and
    cancel in the output layer."""
    w = stopnet.init_weights(0).astype(np.float64)
    w1, b1, w2 = w[:384].reshape(64, 6), w[384:448], w[448:4544].reshape(64, 64)
    w3 = w[4608:4672]
    w1[0], w2[0], w3[:] = 0.0, 0.0, 0.0
    w1[0, 4], b1[0], w2[0, 0], w3[0] = 1.0, -2.0, 1.0, 4.0
    w[4672] = -2.75
    return np.array([0.0] * 6 + [1.0] * 6, np.float32), w.astype(np.float16)


def _index(graph, storage):
    key = graph, storage
    if key not in _indexes:
        ix = hnsw.Index(_blob(graph), storage, keep_fp32=storage != "f32")
        if graph == "sift" and storage == "bf16":
            ix.set_stop_model(*_stop_model())
        _indexes[key] = ix
    return _indexes[key]


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "search":
        q = _points(case["graph"], 100 + seed, n, 0.9)
        opts = dict(k=case["k"], ef=case["ef"], rerank=case["rerank"])
        if case["stop"]:
            opts |= dict(stop_threshold=0.8, stop_period=16)
        return dict(kind=kind, ix=_index(case["graph"], case["storage"]),
                    q=q.cpu().numpy() if case["host"] else q, opts=opts)
    if kind == "insert":
        # the same level draws in another order: every seed adds as many upper-layer lists
        u = np.random.Generator(np.random.Philox(key=100 + seed)).permutation(_levels(5, n))
        return dict(kind=kind, blob=_blob("sift20k"), x=_points("sift20k", 100 + seed, n), u=u)
    g = _gen(seed)
    if kind == "train":
        # log-ratios, log-counts and labels that mostly follow the staleness
        x = torch.rand((n, 6), generator=g, device="cuda") * torch.tensor([0.5, 0.7, 3.0, 8.0, 4.0, 0.6], device="cuda")
        x[:, 2] += 4.0
        x[:, 3] += 4.0
        z = 2.0 * (x[:, 4] - 2.0) - x[:, 5] + torch.randn(n, generator=g, device="cuda")
        return dict(kind=kind, x=x, y=(z > 0).float(), w=stopnet.init_weights(seed % 1000),
                    opts=dict(epochs=case["epochs"], batch=case["batch"], seed=seed % 1000))
    # merge: each shard's k nearest, sorted, over ranges of a million ids each
    shape = (case["shards"], n, case["k"])
    d = (torch.rand(shape, generator=g, device="cuda") + 0.01).cumsum(2)  # strictly increasing
    i = torch.randint(0, 1_000_000, shape, generator=g, device="cuda", dtype=torch.int32)
    return dict(kind=kind, ids=i, dists=d, base=np.arange(case["shards"], dtype=np.uint32) * 1_000_000, k=case["k"])


def run(state):
    kind = state["kind"]
    if kind == "search":
        return state["ix"].search(state["q"], **state["opts"])
    if kind == "insert":
        ix = hnsw.Index(state["blob"], "f32")
        ix.reserve(ix.info.N + len(state["u"]))
        ix.insert(state["x"], state["u"])
        blob = ix.to_blob()
        ix.close()
        return np.frombuffer(blob, np.uint8)
    if kind == "train":
        return hnsw.stop_train(state["x"], state["y"], state["w"], **state["opts"])
    return hnsw.merge_topk(state["ids"], state["dists"], state["base"], state["k"])


def _search_work(g, row_bytes, n, ef, k, d, rerank):
    """A search expands about ef' elements and a few more on the way; each
    expansion reads a neighbour list and scores its unvisited neighbours."""
    efp = max(ef, k)
    expanded, scored = efp + 5, (efp + 5) * g["scored"]
    nbytes = scored * row_bytes + expanded * 8 * g["M"] + d * 4 + k * 8 + (efp * d * 4 if rerank else 0)
    return dict(bytes=n * nbytes, flops=n * 3 * d * (scored + (efp if rerank else 0)))


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "search":
        g = GRAPHS[case["graph"]]
        row = g["d"] * COORD_BYTES[case["storage"]] + (4 if case["storage"] == "fp8" else 0)
        return _search_work(g, row, n, case["ef"], case["k"], g["d"], case["rerank"])
    if kind == "insert":
        # the graph in and out once, and a search per new element
        g = GRAPHS["sift20k"]
        w = _search_work(g, g["d"] * 4, n, g["efc"], g["efc"], g["d"], False)
        total = (2 * g["n"] + n) * (g["d"] * 4 + 8 * g["M"])
        return dict(bytes=w["bytes"] + total, flops=w["flops"])
    if kind == "train":
        # forward, and twice that backward, over 4,480 multiply-adds a sample
        return dict(bytes=case["epochs"] * n * 28, flops=case["epochs"] * n * 3 * 2 * 4480)
    nbytes = (case["shards"] + 1) * n * case["k"] * 8
    return dict(bytes=nbytes, flops=n * case["k"] * max(1.0, math.log2(case["shards"])))


# ---- the same results in 64 bits ------------------------------------------------
def _parse(blob):
    """Arrays of an HNSWGB01 blob (layout in include/hnsw.h), on the GPU."""
    n, d, _, mmax, mmax0, top, ep = struct.unpack_from("<QIIIIII", blob, 16)
    rows = struct.unpack_from("<Q", blob, 64)[0]
    at = [128]

    def take(dtype, *shape):
        count = int(np.prod(shape))
        a = np.frombuffer(blob, dtype, count, at[0]).reshape(shape)
        at[0] += -(-a.nbytes // 16) * 16
        return a

    def ids(*shape):  # 0xFFFFFFFF becomes -1
        return torch.from_numpy(take(np.int32, *shape).copy()).cuda().long()

    x = torch.from_numpy(take(np.float32, n, d).copy()).cuda()
    level = torch.from_numpy(take(np.uint8, n).copy()).cuda().long()
    return dict(x=x, first=torch.cumsum(level, 0) - level, nbr0=ids(n, mmax0), nbr=ids(rows, mmax), top=top, ep=ep)


def _stored(x, storage):
    """Rows as an index holds them, widened to 64 bits."""
    if storage == "f32":
        return x.double()
    if storage in ("bf16", "f16"):
        return x.to(torch.bfloat16 if storage == "bf16" else torch.float16).double()
    s = x.abs().amax(1, keepdim=True) / 448.0
    s = torch.where(s > 0, s, torch.ones_like(s))
    return (x / s).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).double() * s.double()


def _search64(g, rows, q, ef, cosine):
    """Best-first search of all queries in step: ids and distances of the ef
    nearest met, each list sorted by (distance, id)."""

    def dist(qi, e):
        x = rows[e.clamp(min=0)]
        d = 1.0 - (q[qi].unsqueeze(1) * x).sum(2) if cosine else (q[qi].unsqueeze(1) - x).square().sum(2)
        return torch.where(e < 0, math.inf, d)

    n, dev = len(q), q.device
    every = torch.arange(n, device=dev)
    cur = torch.full((n,), g["ep"], device=dev)
    best = dist(every, cur.unsqueeze(1))[:, 0]
    for layer in range(g["top"], 0, -1):
        act = every
        while len(act):
            e = g["nbr"][g["first"][cur[act]] + layer - 1]
            d = dist(act, e)
            m = d.amin(1)
            i = torch.where(d == m.unsqueeze(1), e, 2**40).amin(1)
            go = (m < best[act]) | ((m == best[act]) & (i < cur[act]))
            act = act[go]
            cur[act], best[act] = i[go], m[go]
    w_d = torch.full((n, ef), math.inf, device=dev, dtype=torch.float64)
    w_i = torch.full((n, ef), 2**40, device=dev)
    done = torch.ones((n, ef), device=dev, dtype=torch.bool)  # expanded, or empty
    w_d[:, 0], w_i[:, 0], done[:, 0] = best, cur, False
    act = every
    while len(act):
        act = act[~done[act].all(1)]
        if not len(act):
            break
        at = (~done[act]).int().argmax(1)
        done[act, at] = True
        e = g["nbr0"][w_i[act, at]]
        wi = w_i[act]
        e = torch.where((e.unsqueeze(2) == wi.unsqueeze(1)).any(2), -1, e)
        d = torch.cat([w_d[act], dist(act, e)], 1)
        i = torch.cat([wi, torch.where(e < 0, 2**40, e)], 1)
        x = torch.cat([done[act], e < 0], 1)
        o = i.argsort(1)
        o = o.gather(1, d.gather(1, o).argsort(dim=1, stable=True))[:, :ef]
        w_d[act], w_i[act], done[act] = d.gather(1, o), i.gather(1, o), x.gather(1, o)
    return w_i, w_d


def exact(case, seed):
    kind = case["kind"]
    if kind == "search" and not case["stop"]:
        g, x = _parse(_blob(case["graph"])), _points(case["graph"], 100 + seed, case["n"], 0.9)
        cosine, k = GRAPHS[case["graph"]]["metric"] == hnsw.COSINE, case["k"]
        ids, dists = [], []
        for q in x.double().split(20_000):
            i, d = _search64(g, _stored(g["x"], case["storage"]), q, max(case["ef"], k), cosine)
            if case["rerank"]:
                y = g["x"].double()[i.clamp(max=len(g["x"]) - 1)]
                e = 1.0 - (q.unsqueeze(1) * y).sum(2) if cosine else (q.unsqueeze(1) - y).square().sum(2)
                d = torch.where(torch.isinf(d), math.inf, e)
                o = i.argsort(1)
                o = o.gather(1, d.gather(1, o).argsort(dim=1, stable=True))
                i, d = i.gather(1, o), d.gather(1, o)
            ids.append(torch.where(torch.isinf(d), -1, i)[:, :k])
            dists.append(d[:, :k])
        ids, dists = torch.cat(ids), torch.cat(dists)
        if case["host"]:
            return ids.cpu().numpy().astype(np.uint32), dists.cpu().numpy()
        return ids.int(), dists
    if kind == "train":  # the normalisation has a value of its own; weights and losses follow a random-order path
        x = prepare(case, seed)["x"].double()
        return torch.cat([x.mean(0), x.std(0, correction=0)]).cpu().numpy(), None, None
    if kind == "merge":
        s = prepare(case, seed)
        i = s["ids"].long() + torch.from_numpy(s["base"].astype(np.int64)).cuda().view(-1, 1, 1)
        i, d = (v.permute(1, 0, 2).reshape(case["n"], -1) for v in (i, s["dists"].double()))
        o = i.argsort(1)
        o = o.gather(1, d.gather(1, o).argsort(dim=1, stable=True))[:, :case["k"]]
        return i.gather(1, o).int(), d.gather(1, o)
    return None
