"""The stop network's training kernels at the edges of their tiles: ragged
sample counts, one tile, more tiles than blocks; a training run is a function
of its inputs alone."""
import numpy as np
import pytest

from oracle import stopnet_oracle as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 4097, 40_001])
def test_grad_at_ragged_sizes(n):
    # fp32 sums of at most n/608 + 32 terms per thread and fp16 weights taken
    # exactly: well inside the 1e-3 that the gradient check elsewhere uses
    import torch
    from paper_1603_09320_gb300 import build, hnsw, stopnet
    build.build()
    rng = np.random.default_rng(n)
    w16 = stopnet.init_weights(7)
    X = rng.normal(size=(n, 6)).astype(np.float32) * 2 + 1
    y = (rng.random(n) < 0.5).astype(np.float32)
    norm = np.array([1.0] * 6 + [2.0] * 6, np.float32)
    g, loss = hnsw.stop_grad(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), norm, w16)
    a = (w16.astype(np.float64), X.astype(np.float64), y, norm[:6].astype(np.float64), norm[6:].astype(np.float64))
    go, lo = S.grad(*a), S.loss(*a)
    assert abs(loss - lo) <= 1e-4 * abs(lo)
    err = np.abs(g - go) / np.maximum(np.abs(go), 1e-2 * np.abs(go).max())
    assert err.max() <= 1e-3, err.max()


@pytest.mark.parametrize("n,batch", [(100, 128), (5000, 1024), (50_000, 16_384)])
def test_training_is_reproducible(n, batch):
    import torch
    from paper_1603_09320_gb300 import build, hnsw, stopnet
    build.build()
    rng = np.random.default_rng(3)
    X = torch.from_numpy(rng.normal(size=(n, 6)).astype(np.float32)).cuda()
    y = (X[:, 0] > 0).float()
    a, b = (hnsw.stop_train(X, y, stopnet.init_weights(0), epochs=3, batch=batch, seed=5) for _ in range(2))
    for u, v in zip(a, b):
        np.testing.assert_array_equal(u, v)
    x = X.double().cpu().numpy()
    np.testing.assert_allclose(a[0], np.concatenate([x.mean(0), x.std(0)]), rtol=1e-5, atol=1e-6)
