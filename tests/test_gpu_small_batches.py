"""The block-per-query search kernel (small batches) and the merges into W
against the oracle, at the sizes where they can go wrong: batches at the
limits of each block size and one past them, beams at the register list's
sizes (64, 256, 512 entries) and one past them, neighbour lists of more than
32, a visited set that overflows.  Integer data: ids, distances and counters
are bit-exact."""
import numpy as np
import pytest

from paper_1603_09320_gb300 import synth
from _graphs import oracle_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    import torch
    assert torch.cuda.is_available()
    from paper_1603_09320_gb300 import build, hnsw
    build.build()
    return hnsw


def check(H, g, ix, Q, k, ef, **kw):
    import torch
    q = torch.from_numpy(Q).cuda()
    ids, ds, st = (x.cpu().numpy() for x in ix.search(q, k, ef, stats=True, **kw))
    oi, od, os_ = g.knn_search_batch(Q, k, ef, stats=True)
    np.testing.assert_array_equal(ids.view(np.uint32), oi)
    np.testing.assert_array_equal(ds.astype(np.float64), od)
    np.testing.assert_array_equal(st.view(np.uint32)[:, 1:3], os_[:, 1:3])


@pytest.mark.parametrize("k,ef", [(1, 1), (10, 33), (10, 64), (5, 65), (100, 128), (10, 256), (257, 10), (10, 512),
                                  (10, 513), (10, 1023)])
def test_beam_sizes(H, k, ef):
    g, X, blob = oracle_graph("tiny", 10_000)
    ix = H.Index(blob, "f32")
    Q = synth.queries("tiny", 700)  # more queries than one-block-each launches take
    for n in (1, 40, 700):
        check(H, g, ix, Q[:n], k, ef)
    ix.close()


def test_batch_limits_of_the_block_sizes(H):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g, X, blob = oracle_graph("sift", 20_000)
    Q = synth.queries("sift", 4 * sms + 1)
    for storage, rerank in (("f32", False), ("bf16", True), ("f16", True)):  # these store the integers exactly
        ix = H.Index(blob, storage, keep_fp32=True)
        for n in (2 * sms, 2 * sms + 1, 4 * sms, 4 * sms + 1):
            check(H, g, ix, Q[:n], 10, 50, rerank=rerank)
        ix.close()


@pytest.mark.parametrize("vlog", [5, 7])
def test_overflowing_visited_set(H, vlog):
    g, X, blob = oracle_graph("tiny", 10_000)
    ix = H.Index(blob, "f32")
    for n in (20, 700):
        check(H, g, ix, synth.queries("tiny", n), 10, 100, visited_log2=vlog)
    ix.close()


@pytest.mark.parametrize("Mmax,Mmax0", [(24, 33), (40, 64)])
def test_long_neighbour_lists(H, Mmax, Mmax0):
    # lists of more than 32 on layer 0 and on the upper layers
    from oracle import oracle as O
    p = dict(synth.params("tiny"), M=24, Mmax=Mmax, Mmax0=Mmax0, mL=0.6)
    X = synth.base("tiny", 3000)
    g = O.Graph.build(X, synth.level_uniforms("tiny", 3000), **p)
    ix = H.Index(g.to_blob(), "f32")
    Q = synth.queries("tiny", 800)
    for n in (30, 800):
        for ef in (20, 64, 200):
            check(H, g, ix, Q[:n], 10, ef)
    ix.close()


def test_fewer_reachable_than_asked(H):
    g, X, blob = oracle_graph("tiny", 200)
    ix = H.Index(blob, "f32")
    for n in (3, 700):
        check(H, g, ix, synth.queries("tiny", n), 256, 300)
    ix.close()


@pytest.mark.parametrize("name,storage", [("sift", "fp8"), ("glove", "f32"), ("glove", "bf16"), ("lowd", "f32"),
                                          ("lowd", "f16")])
def test_same_bits_as_the_warp_per_query_kernel(H, name, storage):
    # rows whose distances are rounded: the two kernels add in the same order
    import torch
    g, X, blob = oracle_graph(name, 8000 if name == "glove" else 20_000)
    ix = H.Index(blob, storage, keep_fp32=True)
    q = torch.from_numpy(synth.queries(name, 300)).cuda()
    for ef in (40, 300):
        for rerank in (False, True):
            a = ix.search(q, 10, ef, rerank=rerank, stats=True)
            b = ix.search(q, 10, ef, rerank=rerank, stats=True, schedule=1)
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
            assert torch.equal(a[2][:, 1:3], b[2][:, 1:3])
    ix.close()
