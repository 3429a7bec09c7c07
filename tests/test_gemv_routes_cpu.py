"""Which kernel wq4_gemv launches where a rule on sizes decides: at batch 2-4
the CUDA-core kernel for few long rows and the batched one elsewhere, at batch
1-2 the copy ring or a warp per row for rows that bulk copies cannot take.

The lines are those of the dispatch rule, a size on each side; run without a
GPU over a stand-in for the CUDA runtime (fake_cudart.c), which tells the
kernel of the last launch.
"""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

CHILD = r"""
import ctypes, sys
fake = ctypes.CDLL(sys.argv[1])
from paper_2412_15803_gb300 import wq4
L = wq4.load(build_if_missing=False)
A = 1 << 40          # 16-byte aligned "device" addresses, never read

def kernel(path, batch, N, K, off=0):
    assert L.wq4_test_gemv_path(path) == 0
    assert L.wq4_gemv(A, 2 * A + off, 4 * A, 8 * A, N, K, batch, None) == 0
    return fake.fake_last_kernel()

CORES = [(2, 600, 14336), (2, 1216, 14336), (2, 1216, 8192), (2, 2048, 2048), (2, 64, 256),
         (3, 64, 2048), (3, 76, 2048), (3, 77, 2816), (3, 608, 4096), (3, 1216, 2048), (3, 1216, 14336),
         (4, 64, 2048), (4, 76, 3840), (4, 77, 4096), (4, 608, 4352), (4, 608, 14336), (4, 1216, 4096)]
BATCHED = [(2, 1217, 14336), (2, 4096, 2048), (2, 128256, 4096),
           (3, 76, 1792), (3, 77, 2560), (3, 1024, 2048), (3, 1217, 14336), (3, 64, 256),
           (4, 76, 1792), (4, 77, 3840), (4, 609, 4352), (4, 609, 14336), (4, 1217, 4096), (4, 4096, 4096)]
for c in CORES:
    assert kernel(0, *c) == kernel(2, *c) != kernel(1, *c), c
for c in BATCHED:
    assert kernel(0, *c) == kernel(1, *c) != kernel(2, *c), c
# activations beyond shared memory, batch 5 and scales off 16 bytes: the batched kernels, whatever the hook says
for c in ((3, 64, 36864), (4, 64, 28672), (5, 64, 14336)):
    assert kernel(0, *c) == kernel(1, *c) == kernel(2, *c), c
assert kernel(0, 3, 64, 14336, 2) == kernel(2, 3, 64, 14336, 2) != kernel(2, 3, 64, 14336)
# rows of odd groups at batch 1-2: the copy ring of the batched kernels (as at batch 3), or a warp per row
RING = [(1, 50000, 3104), (1, 100000, 3104), (2, 4000, 2080), (2, 1000, 8160), (2, 512, 14304)]
WARPS = [(1, 1003, 2080), (1, 40000, 3104), (1, 20000, 8160), (1, 30000, 8160), (2, 1003, 2080), (2, 3000, 2080), (2, 700, 8160)]
warps = {b: kernel(0, b, 3, 32) for b in (1, 2)}
for c in RING:
    assert kernel(0, *c) != warps[c[0]], c
for c in WARPS:
    assert kernel(0, *c) == warps[c[0]], c
"""

# launch shapes kept from call to call: the same in any order of sizes, and in a thread that kept none
SHAPES = r"""
import ctypes, random, sys, threading
fake = ctypes.CDLL(sys.argv[1])
fake.fake_last_shape.restype = ctypes.c_size_t
from paper_2412_15803_gb300 import wq4
L = wq4.load(build_if_missing=False)
A = 1 << 40
rng = random.Random(1)
sizes = [(rng.randrange(1, 40000), 256 * rng.randrange(1, 57), rng.randrange(5, 33)) for _ in range(300)]

def shapes(order):
    out = {}
    for N, K, batch in order:
        assert L.wq4_gemv(A, 2 * A, 4 * A, 8 * A, N, K, batch, None) == 0
        out[N, K, batch] = (fake.fake_last_kernel(), fake.fake_last_shape())
    return out

first = shapes(sizes)
assert len(set(first.values())) > 50
for _ in range(3):
    rng.shuffle(sizes)
    assert shapes(sizes) == first and shapes([c for c in sizes[:100] for _ in range(2)]).items() <= first.items()
other = []
t = threading.Thread(target=lambda: other.append(shapes(sizes)))
t.start()
t.join()
assert other == [first]
"""


@pytest.mark.parametrize("child", [CHILD, SHAPES], ids=["routes", "shapes"])
def test_launches(fake_cudart, child):
    env = dict(os.environ, LD_PRELOAD=fake_cudart, PYTHONPATH=os.path.dirname(HERE))
    r = subprocess.run([sys.executable, "-c", child, fake_cudart], env=env, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
