"""Incremental insertion at the edges of its kernels' ranges against the
oracle's batch form, byte for byte on integer data: selection flags, rows of
few, ragged and more than 128 coordinates, upper lists of up to 16, of up to 32
and of more than 32, a beam
of more than 512 entries, several upper layers and new top levels."""
import numpy as np
import pytest

from paper_1603_09320_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [
    # d, M, Mmax, Mmax0, efC, mL, heuristic, keep_pruned
    (32, 8, 8, 16, 64, 0.5, False, False),
    (32, 8, 8, 16, 64, 0.8, True, True),
    (5, 6, 7, 13, 33, 0.9, True, False),
    (130, 6, 6, 12, 40, 0.7, True, False),
    (32, 12, 24, 48, 100, 0.8, True, False),
    (32, 20, 40, 64, 600, 0.6, True, False),
    (32, 20, 40, 64, 600, 0.6, True, True),
]


@pytest.mark.parametrize("d,M,Mmax,Mmax0,efC,mL,heuristic,keep", SHAPES)
def test_insert_equals_batched_oracle(d, M, Mmax, Mmax0, efC, mL, heuristic, keep):
    from oracle import oracle as O
    from paper_1603_09320_gb300 import build, hnsw as H
    build.build()
    p = dict(M=M, Mmax=Mmax, Mmax0=Mmax0, efC=efC, mL=mL, heuristic=heuristic, keep_pruned=keep)
    N, n0 = 2600, 1400
    X = synth.rng(d).integers(0, 256, size=(N, d)).astype(np.float32)
    u = synth.uniform_open01(77, N)
    base = O.Graph.build(X[:n0], u[:n0], **p)
    og = O.Graph.new(X, **p)
    for i in range(n0):
        og.insert(i, O.level_from_u(float(u[i]), mL))
    ix = H.Index(base.to_blob(), "f32")
    ix.reserve(2 * N)  # room for the many upper-layer rows of a large mL
    for lo, hi in ((n0, n0 + 1), (n0 + 1, 1500), (1500, N)):
        ix.insert(X[lo:hi], u[lo:hi])
        og.insert_batched(lo, u[lo:hi])
    gb, ob = ix.to_blob(), og.to_blob()
    ix.close()
    if gb != ob:
        g, o = O.Graph.from_blob(gb), O.Graph.from_blob(ob)
        diff = [(i, lc) for i in range(N) for lc in range(g.level(i) + 1) if g.neighbors(i, lc) != o.neighbors(i, lc)]
        raise AssertionError(f"{len(diff)} lists differ, first {diff[:10]}")
