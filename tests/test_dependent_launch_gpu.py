"""Programmatic dependent launch: calls one after another, nothing waited for between.

A kernel that lets its dependents launch at its start and writes late (a
spinning writer of the test's own) stands in for a predecessor that is still
running while the next call's blocks are there already.  What each call
promises about it, against the same calls run one at a time, bit for bit.
"""
import ctypes
import subprocess

import pytest
import torch

from paper_2412_15803_gb300 import build, wq4
from paper_2412_15803_gb300.attention import PagedAttentionLayer
from paper_2412_15803_gb300.model import ModelShape

pytestmark = pytest.mark.gpu

WRITER = r"""
#include <cstdint>
#include <cuda_runtime.h>
static __device__ uint64_t now() { uint64_t t; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)); return t; }
// lets its dependents launch, waits for `ns`, then copies n words
__global__ void late_copy(uint32_t* dst, const uint32_t* src, long n, uint64_t ns)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint64_t t0 = now();
    while (now() - t0 < ns) {}
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) dst[i] = src[i];
}
extern "C" int launch_late_copy(uint32_t* dst, const uint32_t* src, long n, uint64_t ns, void* stream)
{
    late_copy<<<8, 256, 0, (cudaStream_t)stream>>>(dst, src, n, ns);
    return cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def late_copy(tmp_path_factory):
    d = tmp_path_factory.mktemp("writer")
    (d / "writer.cu").write_text(WRITER)
    subprocess.check_call([build.nvcc(), *build.ARCH, "-shared", "-cudart", "shared", "-Xcompiler", "-fPIC", "-o",
                           str(d / "writer.so"), str(d / "writer.cu")])
    f = ctypes.CDLL(str(d / "writer.so")).launch_late_copy
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long, ctypes.c_uint64, ctypes.c_void_p]

    def call(dst, src, ns=300_000):
        assert f(dst.data_ptr(), src.data_ptr(), dst.numel() * dst.element_size() // 4, ns,
                 torch.cuda.current_stream().cuda_stream) == 0
    return call


def _matrix(N, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    W = torch.randint(-2**31, 2**31, (N, K // 8), generator=g, device="cuda", dtype=torch.int32)
    return W, (0.005 + 0.015 * torch.rand((N, K // 32), generator=g, device="cuda")).half().view(torch.int16)


def _x(rows, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((rows, K), generator=g, device="cuda").half().view(torch.int16)


def _call(kind, W, s, x, y):
    f = wq4.wq4_gemm if kind == "gemm" else wq4.wq4_gemv
    f(W, s, x, y, W.shape[0], W.shape[1] * 8, x.shape[0])


def _layer(seed=1):
    return PagedAttentionLayer(ModelShape("pdl", 1, 1024, 512, 8, 2, 128, 1000), [700, 33], seed=seed)


# one kernel of each route: the batched GEMV, each token tile, K split over a cluster
GEMMS = [(2048, 1024, 8), (2048, 1024, 40), (4096, 1024, 100), (4096, 512, 180), (8192, 512, 1000), (512, 14336, 200)]


@pytest.mark.parametrize("N,K,M", GEMMS)
def test_gemm_reads_weights_that_a_running_kernel_writes(late_copy, N, K, M):
    W, s = _matrix(N, K, 1)
    W1, s1 = _matrix(N, K, 2)
    x, y = _x(M, K, 3), torch.empty((M, N), dtype=torch.int16, device="cuda")
    _call("gemm", W1, s1, x, y)
    torch.cuda.synchronize()
    ref = y.clone()
    for dst, src, rest in ((W, W1, (s, s1)), (s, s1, (W, W1))):
        rest[0].copy_(rest[1])
        dst.zero_()
        torch.cuda.synchronize()
        late_copy(dst, src)
        _call("gemm", W, s, x, y)
        torch.cuda.synchronize()
        assert torch.equal(y, ref)


# what stands between the writer and wq4_gemv
@pytest.mark.parametrize("between", ["attention", "gemm-8", "gemm-100", "gemv-1-large", "gemv-1", "gemv-8", "gemv-5-ragged"])
@pytest.mark.parametrize("batch", [1, 2, 8])
def test_gemv_reads_weights_written_two_launches_before(late_copy, between, batch):
    N, K = 8192, 2048
    W, s = _matrix(N, K, 4)
    W1, _ = _matrix(N, K, 5)
    x, y = _x(batch, K, 6), torch.empty((batch, N), dtype=torch.int16, device="cuda")
    _call("gemv", W1, s, x, y)
    torch.cuda.synchronize()
    ref = y.clone()
    if between == "attention":
        mid = _layer().run
    else:
        kind, rows, *form = between.split("-")
        n, k = (8192, 2048) if form == ["large"] else (1003, 2080) if form == ["ragged"] else (1024, 1024)
        m, ms = _matrix(n, k, 7)
        mx, my = _x(int(rows), k, 8), torch.empty((int(rows), n), dtype=torch.int16, device="cuda")
        mid = lambda: _call(kind, m, ms, mx, my)
    mid()
    torch.cuda.synchronize()
    late_copy(W, W1)
    mid()
    _call("gemv", W, s, x, y)
    torch.cuda.synchronize()
    assert torch.equal(y, ref)


# one call's y is the next one's x (the shapes of a square projection), and the
# attention between two of them
@pytest.mark.parametrize("chain", ["gemv-1", "gemv-2", "gemv-3", "gemv-8", "gemv-32", "gemm-8", "gemm-40", "gemm-100", "gemm-600"])
def test_dependent_calls_back_to_back(late_copy, chain):
    kind, rows = chain.split("-")
    rows, H = int(rows), 2048
    mats = [_matrix(H, H, 10 + i) for i in range(4)]
    for _, s in mats:
        s.view(torch.float16).mul_(0.3)
    xs = [_x(rows, H, 20)] + [torch.empty((rows, H), dtype=torch.int16, device="cuda") for _ in mats]

    def run(sync):
        for i, (W, s) in enumerate(mats):
            _call(kind, W, s, xs[i], xs[i + 1])
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()

    run(True)
    ref = [t.clone() for t in xs[1:]]
    for _ in range(5):
        for t in xs[1:]:
            t.zero_()
        src = xs[0].clone()
        xs[0].zero_()
        torch.cuda.synchronize()
        late_copy(xs[0], src, 100_000)
        run(False)
        assert all(torch.equal(a, b) for a, b in zip(xs[1:], ref))


def test_attention_between_dependent_calls(late_copy):
    layer = _layer(3)
    H = 1024
    (Wq, sq), (Wo, so) = _matrix(H, H, 30), _matrix(H, H, 31)
    x, y = _x(2, H, 32), torch.empty((2, H), dtype=torch.int16, device="cuda")
    k = layer.k.clone()

    def run():
        _call("gemv", Wq, sq, x, layer.q)
        layer.run()
        _call("gemv", Wo, so, layer.out, y)

    run()
    torch.cuda.synchronize()
    ref_a, ref = layer.out.clone(), y.clone()
    for _ in range(5):
        layer.k.zero_()
        layer.out.zero_()
        torch.cuda.synchronize()
        late_copy(layer.k, k)          # the cache itself, two launches before
        run()
        torch.cuda.synchronize()
        assert torch.equal(layer.out, ref_a) and torch.equal(y, ref)
    layer.k.zero_()
    torch.cuda.synchronize()
    late_copy(layer.k, k)              # ... and right before
    layer.run()
    torch.cuda.synchronize()
    assert torch.equal(layer.out, ref_a)
    assert wq4.wq4_device_status() == 0
