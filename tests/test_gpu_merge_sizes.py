"""The top-k merge where its read-ahead ends (4 entries of a list at a time for
k above 4, one below), with lists that end early, ties between shards, negative
and infinite distances, against a sort of the union: bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 2, 7, 32])
@pytest.mark.parametrize("n,k", [(1, 1), (3, 7), (9, 8), (11, 4), (11, 5), (70, 9), (5, 16), (4, 17), (3, 200), (2, 1024)])
def test_merge_sizes(S, n, k):
    import torch
    from paper_1603_09320_gb300 import build, hnsw as H
    build.build()
    r = np.random.default_rng(1000 * S + k)
    ids = np.full((S, n, k), 0xFFFFFFFF, np.uint32)
    ds = np.full((S, n, k), np.inf, np.float32)
    base = (np.arange(S) * 5000).astype(np.uint32)
    want_i, want_d = np.full((n, k), 0xFFFFFFFF, np.uint32), np.full((n, k), np.inf, np.float32)
    for q in range(n):
        pairs = []
        for s in range(S):
            m = int(r.integers(0, k + 1)) if (q + s) % 2 else k
            i = r.permutation(5000)[:m].astype(np.uint32)
            # one shard holds most of the nearest; few distinct values: ties
            d = r.integers(-20, 20, size=m).astype(np.float32) + (0 if s == q % S else 15)
            d[r.random(m) < 0.05] = np.inf
            o = np.lexsort((i, d))
            ids[s, q, :m], ds[s, q, :m] = i[o], d[o]
            pairs += [(float(a), int(b) + int(base[s])) for a, b in zip(d, i)]
        for j, (a, b) in enumerate(sorted(pairs)[:k]):
            want_d[q, j], want_i[q, j] = a, b
    gi, gd = H.merge_topk(torch.from_numpy(ids.view(np.int32)).cuda(), torch.from_numpy(ds).cuda(), base, k)
    assert np.array_equal(gi.cpu().numpy().view(np.uint32), want_i)
    assert np.array_equal(gd.cpu().numpy().view(np.uint32), want_d.view(np.uint32))
