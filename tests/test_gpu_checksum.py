"""The blob checksum where the GPU computes it: graphs whose payload lies
around the sizes at which its pieces and chunks end (8 KB and 16 MB) are
accepted after the host builder's checksum, exported with the same bytes, and
refused when one byte differs."""
import numpy as np
import pytest

from paper_1603_09320_gb300 import hnsw

pytestmark = pytest.mark.gpu


# payload below the smallest that goes to the GPU, of a whole number of pieces
# (8,192 elements of 97 bytes), with tails, above one chunk
@pytest.mark.parametrize("n,d,extra", [(500, 33, 0), (8192, 16, 0), (8193, 16, 3), (3001, 37, 1), (20_011, 201, 5)])
def test_checksum(n, d, extra):
    r = np.random.default_rng(n)
    x = r.integers(0, 256, size=(n, d)).astype(np.float32)
    u = np.ones(n)  # every element on layer 0 ...
    u[:extra] = 1e-3  # ... but these
    blob = hnsw.build_graph(x, u, M=4, Mmax0=8, ef_construction=8)
    ix = hnsw.Index(blob, "f32")
    assert ix.to_blob() == blob
    ix.close()
    for at in (128, 128 + 8192 * 3 + 17, len(blob) // 2, len(blob) - 1):
        bad = bytearray(blob)
        bad[min(at, len(blob) - 1)] ^= 0x10
        with pytest.raises(hnsw.HnswError, match="checksum"):
            hnsw.Index(bytes(bad), "f32")
