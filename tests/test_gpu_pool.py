"""An upload, an export and a construction leave the device's memory pool as
they found it: nothing kept of their scratch, the release threshold of the
process unchanged (a fresh process, as scheduled searches raise it)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import ctypes as C
import numpy as np
from paper_1603_09320_gb300 import build, hnsw
build.build()
r = np.random.default_rng(0)
x = r.integers(0, 256, size=(20_000, 128)).astype(np.float32)
u = 1.0 - r.random(20_000)
blob = hnsw.build_graph_gpu(x, u, M=8, ef_construction=20)
ix = hnsw.Index(blob, "f32")
assert len(ix.to_blob()) > 8 << 20
ix.close()
cu = C.CDLL("libcuda.so.1")
dev, pool, value = C.c_int(), C.c_void_p(), C.c_uint64()
assert cu.cuDeviceGet(C.byref(dev), 0) == 0 and cu.cuDeviceGetDefaultMemPool(C.byref(pool), dev) == 0
for name, attr in (("threshold", 4), ("reserved", 5)):  # CU_MEMPOOL_ATTR_RELEASE_THRESHOLD, _RESERVED_MEM_CURRENT
    assert cu.cuMemPoolGetAttribute(pool, attr, C.byref(value)) == 0
    print(name, value.value)
"""


def test_upload_and_export_keep_no_device_memory():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["threshold", "0", "reserved", "0"]
