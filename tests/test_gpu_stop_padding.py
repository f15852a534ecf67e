"""The stop network's gradient over a last tile that is not full: the places
past the last sample add nothing, also where an infinite weight would make
their share NaN (unit 0 of the second layer reads unit 0 of the first through
it, which is zero on every sample and not on zeros)."""
import numpy as np
import pytest

from oracle import stopnet_oracle as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 95, 20_001])
def test_places_past_the_end_add_nothing(n):
    import torch
    from paper_1603_09320_gb300 import build, hnsw, stopnet
    build.build()
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, 6)).astype(np.float32)
    X[:, 0] = 1.0
    y = (rng.random(n) < 0.5).astype(np.float32)
    norm = np.array([0.0] * 6 + [1.0] * 6, np.float32)
    w = stopnet.init_weights(7)
    w1, b1, w2, b2 = w[:384].reshape(64, 6), w[384:448], w[448:4544].reshape(64, 64), w[4544:4608]
    w1[0], b1[0] = 0.0, 1.0
    w1[0, 0] = -10.0  # relu(1 - 10) on a sample, relu(1) on zeros
    w2[:, 0] = 0.0
    dead = w.copy()
    w2[0, 0] = np.inf
    dead[4544] = -1000.0  # the network that unit 0 of layer 2 never takes part in
    g, loss = hnsw.stop_grad(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), norm, w)
    a = (dead.astype(np.float64), X.astype(np.float64), y, norm[:6].astype(np.float64), norm[6:].astype(np.float64))
    go, lo = S.grad(*a), S.loss(*a)
    assert abs(loss - lo) <= 1e-4 * abs(lo)
    # fp32 sums of at most n/608 + 32 terms, as in the gradient checks elsewhere
    err = np.abs(g - go) / np.maximum(np.abs(go), 1e-2 * np.abs(go).max())
    assert err.max() <= 1e-3, err.max()
