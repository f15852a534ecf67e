"""Insertion on real-valued data: the upper layers' distances are fp32 sums over
the coordinates one after another (the enter point's excepted), for the search
and for the shrink of a reverse link.  2^24 + 1 + 1 + ... added that way stays
2^24, below 2^24 + 4; added in parts it comes out above it, so the order shows
in which element a list holds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U1 = float(np.exp(-1.5))  # a level of 1 at mL = 1


def insert_last(X, metric, **kw):
    from oracle import oracle as O
    from paper_1603_09320_gb300 import build, hnsw as H
    build.build()
    n = len(X) - 1
    blob = H.build_graph(X[:n], np.full(n, U1), metric=metric, M=1, ef_construction=8, mL=1.0, heuristic=False,
                         n_threads=1, **kw)
    ix = H.Index(blob, "f32")
    ix.reserve(n + 1)
    ix.insert(X[n:], np.array([U1]))
    g = O.Graph.from_blob(ix.to_blob())
    ix.close()
    return g


def rows(d, big):
    a, b = np.ones(d, np.float32), np.zeros(d, np.float32)
    a[0] = b[0] = big
    return a, b


@pytest.mark.parametrize("d", [33, 128, 200])
def test_search_order_l2(d):
    a, b = rows(d, 4096.0)
    b[1] = 2.0  # from the origin: a 2^24, b 2^24 + 4
    far = np.zeros(d, np.float32)
    far[0] = 20000.0
    g = insert_last(np.stack([far, a, b, np.zeros(d, np.float32)]), 0, Mmax=2, Mmax0=2)
    assert g.neighbors(3, 1) == [1]


@pytest.mark.parametrize("d", [33, 128, 200])
def test_search_order_inner_product(d):
    a, b = rows(d, 2.0**24)
    b[1] = 4.0  # with ones: a 2^24, b 2^24 + 4
    g = insert_last(np.stack([np.zeros(d, np.float32), a, b, np.ones(d, np.float32)]), 1, Mmax=2, Mmax0=2)
    assert g.neighbors(3, 1) == [2]


@pytest.mark.parametrize("d", [33, 128, 200])
def test_reverse_link_order(d):
    a, b = rows(d, 4096.0)
    a[0] = -4096.0
    b[1] = 2.0
    # the origin's one place holds a (2^24) and is offered b (2^24 + 4)
    g = insert_last(np.stack([np.zeros(d, np.float32), a, b]), 0, Mmax=1, Mmax0=2)
    assert g.neighbors(2, 1) == [0]
    assert g.neighbors(0, 1) == [1]
