"""Every entry point launches on a second device too.

A kernel's limit of dynamic shared memory belongs to a device, so a launcher
that sets it once per process fails on the next one.  Run without a GPU, in a
child process over a stand-in for the CUDA runtime (fake_cudart.c) that holds
every launch to the limit set on the current device.
"""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

CHILD = r"""
import ctypes, sys
fake, name, rows, N, K = ctypes.CDLL(sys.argv[1]), sys.argv[2], *(int(v) for v in sys.argv[3:])
from paper_2412_15803_gb300 import wq4
L = wq4.load(build_if_missing=False)
A = 1 << 40          # 16-byte aligned "device" addresses, never read
for device in (0, 1, 0, 2):
    fake.fake_set_device(device)
    before = fake.fake_launches()
    if name == "attention":
        c = wq4.wq4_kv_cache(k=A, v=2 * A, num_pages=64, n_kv_heads=8, page_size=16, head_dim=128,
                             page_table=3 * A, page_table_stride=32)
        n = L.wq4_paged_attention_workspace_bytes(rows, 32, 8, 128)
        rc = L.wq4_paged_attention(ctypes.byref(c), 4 * A, 4096, 5 * A, 6 * A, 4096, rows, 32, 0.1, 7 * A, n, None)
    else:
        rc = getattr(L, name)(A, 2 * A, 4 * A, 8 * A, N, K, rows, None)
    assert rc == 0, f"device {device}: {rc}"
    assert fake.fake_launches() == before + 1
"""


# one size of every kernel: GEMM token tiles 64, 128, 192 and 256 and a split K;
# batch 1 small and large, 2, the batched tile loop with and without a tail
# round, rows of the copy ring; attention
@pytest.mark.parametrize("name,rows,N,K", [
    ("wq4_gemm", 40, 3072, 1024), ("wq4_gemm", 100, 16384, 1024), ("wq4_gemm", 180, 28672, 1024),
    ("wq4_gemm", 2048, 28672, 4096), ("wq4_gemm", 200, 512, 14336), ("wq4_gemm", 8, 3072, 1024),
    ("wq4_gemv", 1, 2048, 2048), ("wq4_gemv", 1, 16384, 3072), ("wq4_gemv", 2, 2048, 2048), ("wq4_gemv", 2, 16384, 3072),
    ("wq4_gemv", 4, 600, 14336), ("wq4_gemv", 8, 3072, 8192), ("wq4_gemv", 24, 8192, 4096), ("wq4_gemv", 32, 128256, 4096),
    ("wq4_gemv", 5, 1003, 2080), ("wq4_gemv", 1, 1003, 2080), ("attention", 4, 0, 0)])
def test_launches_on_every_device(fake_cudart, name, rows, N, K):
    env = dict(os.environ, LD_PRELOAD=fake_cudart, PYTHONPATH=os.path.dirname(HERE))
    r = subprocess.run([sys.executable, "-c", CHILD, fake_cudart, name, str(rows), str(N), str(K)], env=env,
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
