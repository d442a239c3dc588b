"""Device memory of a build per key, in a process of its own (the library's pool keeps what a build has taken).
Per key: 40 bytes of ids, keys, indices and sizes; queue entries of 16 bytes, two per l + 1 keys for light split
nodes, one per l for leaves, one per l + 1 for partial leaves; per bucket 64 bytes; the structure 0.25.  At l = 12,
b = 100: 40 + 2.5 + 1.3 + 1.2 + 0.6 + 0.3 = 45.9, and the pool's rounding.  Heavy split nodes add two queue entries
and 24 bytes of search state per node, of dozens of keys each (none in a build as large as this)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROGRAM = """
import torch
from paper_1910_06416_gb300 import inputs, recsplit as rs
n = 20000000
keys = inputs.device_splitmix64(5, n, device="cuda")
rs.Structure.build_u64(keys[:100000], 12, 100).free()
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
s = rs.Structure.build_u64(keys, 12, 100)
torch.cuda.synchronize()
print((free - torch.cuda.mem_get_info()[0]) / n)
"""


def test_bytes_per_key():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1910_06416_gb300 import build
    build.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert 40 < float(r.stdout) < 48.5, r.stdout
