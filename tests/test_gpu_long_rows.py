"""Rows above 128 coordinates, a row per warp and two rows' reads at a time,
against the oracle: full and partial rows, lists that leave odd numbers of rows,
both metrics.  Small integers: ids, distances and counters are bit-exact (fp8
rows round them: the same bits as the block-per-query kernel's)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("d,Mmax0", [(129, 13), (200, 7), (384, 16), (511, 33), (512, 12)])
def test_long_rows(d, Mmax0, metric):  # f32, bf16, f16, fp8
    import torch
    from oracle import oracle as O
    from paper_1603_09320_gb300 import build, hnsw as H
    build.build()
    r = np.random.default_rng(d)
    X = r.integers(0, 32, size=(1500, d)).astype(np.float32)
    Q = r.integers(0, 32, size=(650, d)).astype(np.float32)
    g = O.Graph.build(X, 1.0 - r.random(1500), metric=metric, M=7, Mmax=7, Mmax0=Mmax0, efC=40, mL=0.5)
    for storage in ("f32", "bf16", "f16"):
        ix = H.Index(g.to_blob(), storage)
        against_the_oracle(ix, g, Q)
        ix.close()
    ix = H.Index(g.to_blob(), "fp8")
    q = torch.from_numpy(Q[:40]).cuda()
    for ef in (20, 100):
        for a, b in zip(ix.search(q, 10, ef), ix.search(q, 10, ef, schedule=1)):
            assert torch.equal(a, b)
    ix.close()


def against_the_oracle(ix, g, Q):
    import torch
    for n, schedule in ((650, 0), (40, 1)):  # both take the warp-per-query kernel
        for k, ef in ((10, 20), (10, 100)):
            ids, ds, st = (x.cpu().numpy() for x in ix.search(torch.from_numpy(Q[:n]).cuda(), k, ef, stats=True,
                                                              schedule=schedule))
            oi, od, os_ = g.knn_search_batch(Q[:n], k, ef, stats=True)
            np.testing.assert_array_equal(ids.view(np.uint32), oi)
            np.testing.assert_array_equal(ds.astype(np.float64), od)
            np.testing.assert_array_equal(st.view(np.uint32)[:, 1:3], os_[:, 1:3])
