"""An insertion into a graph whose header asks for more links than its lists
have places (the checksum does not cover the header) is refused before any
kernel runs; the graph itself still searches and takes a proper insertion."""
import struct

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [0, 9, 17, 65, 1 << 20])
def test_impossible_m_is_refused(M):
    from paper_1603_09320_gb300 import build, hnsw
    build.build()
    r = np.random.default_rng(1)
    x = r.integers(0, 256, size=(300, 16)).astype(np.float32)
    blob = bytearray(hnsw.build_graph(x[:250], 1.0 - r.random(250), M=8, Mmax=8, Mmax0=16, ef_construction=20))
    assert struct.unpack_from("<I", blob, 28)[0] == 8
    ok = hnsw.Index(bytes(blob), "f32")
    struct.pack_into("<I", blob, 28, M)
    ix = hnsw.Index(bytes(blob), "f32")
    u = 1.0 - r.random(50)
    for i in (ok, ix):
        i.reserve(400)
    with pytest.raises(hnsw.HnswError, match="M of the graph") as e:
        ix.insert(x[250:], u)
    assert e.value.status == 1  # HNSW_EINVAL
    ok.insert(x[250:], u)
    assert ok.info.N == 300 and ix.info.N == 250
    for i in (ok, ix):
        i.close()
