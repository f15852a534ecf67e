"""The block-per-query search kernel where its other test does not reach:
4-warp blocks with each size of the register list, at and around the batches
they are taken for; blocks that take several queries in turn (the visited set
refilled where W and a copy of the query lay); queries with infinities and NaN;
grouped launches at the limits.  Integer data: bit-exact against the oracle."""
import numpy as np
import pytest

from paper_1603_09320_gb300 import synth
from _graphs import oracle_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    import torch
    from paper_1603_09320_gb300 import build, hnsw
    build.build()
    g, X, blob = oracle_graph("tiny", 10_000)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    Q = np.concatenate([synth.queries("tiny", 1000)] * 2)[:4 * sms + 1]
    plain, rerank = hnsw.Index(blob, "f32"), hnsw.Index(blob, "bf16", keep_fp32=True)
    yield hnsw, g, sms, Q, {False: plain, True: rerank}
    plain.close()
    rerank.close()


def check(g, ix, Q, k, ef, **kw):
    import torch
    ids, ds, st = (x.cpu().numpy() for x in ix.search(torch.from_numpy(Q).cuda(), k, ef, stats=True, **kw))
    oi, od, os_ = g.knn_search_batch(Q, k, ef, stats=True)
    np.testing.assert_array_equal(ids.view(np.uint32), oi)
    np.testing.assert_array_equal(ds.astype(np.float64), od)
    np.testing.assert_array_equal(st.view(np.uint32)[:, 1:3], os_[:, 1:3])


@pytest.mark.parametrize("rerank", [False, True])
@pytest.mark.parametrize("ef", [100, 256, 257, 512])
def test_four_warp_blocks_with_wide_beams(setup, ef, rerank):
    _, g, sms, Q, ix = setup
    for n in (2 * sms, 2 * sms + 1, 3 * sms, 3 * sms + 1, 4 * sms, 4 * sms + 1):
        check(g, ix[rerank], Q[:n], 10, ef, rerank=rerank)


@pytest.mark.parametrize("rerank", [False, True])
@pytest.mark.parametrize("ef", [20, 200, 400])
def test_several_queries_per_block(setup, ef, rerank):
    # a visited set of 128 KB: one block per SM
    _, g, sms, Q, ix = setup
    for n in (sms, sms + 1, 2 * sms, 3 * sms):
        check(g, ix[rerank], Q[:n], 10, ef, rerank=rerank, visited_log2=15)


@pytest.mark.parametrize("rerank", [False, True])
def test_infinities_and_nan(setup, rerank):
    import torch
    _, g, sms, Q, ix = setup
    q = Q[:3 * sms].copy()
    q[0::5, 3] = np.inf
    q[1::5, 7] = -np.inf
    q[2::5, 0] = np.nan
    q[3::5] = np.finfo(np.float32).max
    t = torch.from_numpy(q).cuda()
    for ef in (10, 64, 66, 200):
        for n in (40, 2 * sms, 3 * sms):
            a = ix[rerank].search(t[:n], 10, ef, rerank=rerank, stats=True)
            b = ix[rerank].search(t[:n], 10, ef, rerank=rerank, stats=True, schedule=1)
            assert torch.equal(a[0], b[0]) and torch.equal(a[1].view(torch.int32), b[1].view(torch.int32))
            assert torch.equal(a[2][:, 1:3], b[2][:, 1:3])
        check(g, ix[rerank], q[4::5], 10, ef, rerank=rerank)  # the others are what they are alone
        oi, od = g.knn_search_batch(q[4::5][:n // 5], 10, ef)[:2]
        np.testing.assert_array_equal(a[0].cpu().numpy().view(np.uint32)[4::5][:len(oi)], oi)
        np.testing.assert_array_equal(a[1].cpu().numpy().astype(np.float64)[4::5][:len(od)], od)


@pytest.mark.parametrize("total,max_ef", [("one", 300), ("two", 60), ("two+1", 512), ("three", 500), ("four", 256)])
def test_grouped_launches(setup, total, max_ef):
    # requests of different k and ef, queued behind one that holds the only slot
    hnsw, g, sms, Q, ix = setup
    n = {"one": sms, "two": 2 * sms, "two+1": 2 * sms + 1, "three": 3 * sms, "four": 4 * sms}[total]
    g2, X2, b2 = oracle_graph("sift", 20_000)
    other = hnsw.Index(b2, "f32")
    sv = hnsw.Server(n_slots=1)
    a, b = sv.add_index(other), sv.add_index(ix[False])
    big = sv.submit(a, np.ascontiguousarray(np.tile(synth.queries("sift", 2000), (10, 1))), 10, 512)
    cut = [0, 1, n // 3, n // 2, n - 7, n]
    asked = [(1, 1), (10, 20), (33, 40), (5, max_ef), (50, 10)]
    tickets = [sv.submit(b, Q[lo:hi], k, ef) for lo, hi, (k, ef) in zip(cut, cut[1:], asked)]
    for lo, hi, (k, ef), t in zip(cut, cut[1:], asked, tickets):
        ids, ds = sv.wait(t)[:2]
        oi, od = g.knn_search_batch(Q[lo:hi], k, ef)[:2]
        np.testing.assert_array_equal(ids, oi)
        np.testing.assert_array_equal(ds.astype(np.float64), od)
    sv.wait(big)
    sv.close()
    other.close()
