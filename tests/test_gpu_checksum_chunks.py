"""The blob checksum on the GPU where its 16 MB chunks end: payloads of one
piece (8 KB) less than a chunk, exactly one, one and a tail, one and a piece,
two, and more than two.  Exported with the host builder's checksum, and
refused when a byte differs before, at and after a chunk's end."""
import numpy as np
import pytest

from paper_1603_09320_gb300 import hnsw

pytestmark = pytest.mark.gpu

PIECE, CHUNK = 8192, 2048  # bytes; pieces


@pytest.mark.parametrize("n,d,pieces,tail", [(8184, 500, 2047, 0), (8188, 500, 2048, 0), (8452, 484, 2048, 16),
                                             (8192, 500, 2049, 0), (16376, 500, 4096, 0), (16411, 500, 4104, 6176)])
def test_checksum_across_chunks(n, d, pieces, tail):
    r = np.random.default_rng(n)
    x = r.integers(0, 256, size=(n, d)).astype(np.float32)
    blob = hnsw.build_graph(x, np.ones(n), M=4, Mmax0=12, ef_construction=8)  # every element on layer 0
    assert divmod(len(blob) - 128, PIECE) == (pieces, tail)
    ix = hnsw.Index(blob, "f32")
    assert ix.to_blob() == blob
    ix.close()
    end = 128 + PIECE * CHUNK
    ats = {128, end // 2, end - 1, end, end + 17, 128 + 2 * PIECE * CHUNK - 1, 128 + 2 * PIECE * CHUNK, len(blob) - 1}
    for at in sorted(a for a in ats if a < len(blob)):
        bad = bytearray(blob)
        bad[at] ^= 0x10
        with pytest.raises(hnsw.HnswError, match="checksum"):
            hnsw.Index(bytes(bad), "f32")


CODE = """
import ctypes as C
import numpy as np
from paper_1603_09320_gb300 import build, hnsw
build.build()
x = np.random.default_rng(0).integers(0, 256, size=(16376, 500)).astype(np.float32)
hnsw.Index(hnsw.build_graph(x, np.ones(16376), M=4, Mmax0=12, ef_construction=8), "f32").close()
cu = C.CDLL("libcuda.so.1")
dev, pool, value = C.c_int(), C.c_void_p(), C.c_uint64()
assert cu.cuDeviceGet(C.byref(dev), 0) == 0 and cu.cuDeviceGetDefaultMemPool(C.byref(pool), dev) == 0
assert cu.cuMemPoolGetAttribute(pool, 8, C.byref(value)) == 0  # CU_MEMPOOL_ATTR_USED_MEM_HIGH
print(value.value)
"""


def test_scratch_is_a_chunk_and_its_maps():
    # 16 MB of input, 4 KB of maps per 8 KB piece, a few KB beside them
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert 24 << 20 <= int(r.stdout) <= (24 << 20) + (64 << 10)
