"""Waits for copies that never come: the kernel ends, flags it, and the next call is clean.

Every role of a block gives up after the same time, within the few cycles in
which it began to wait, so that the lanes and warps give up in any order: one
that left its loop alone would leave the others in a warp-wide instruction or
at a named barrier.
"""
import time

import pytest
import torch

from paper_2412_15803_gb300 import wq4
from paper_2412_15803_gb300.attention import PagedAttentionLayer
from paper_2412_15803_gb300.model import ModelShape

pytestmark = pytest.mark.gpu

PIPE_TIMEOUT = 1
GEMM_X, GEMM_W, ATTN = 1, 2, 3


def _stalled(stall, call):
    assert wq4.wq4_device_status() == 0
    try:
        wq4.wq4_test_copy_stall(stall)
        t0 = time.perf_counter()
        call()
        torch.cuda.synchronize()
        took = time.perf_counter() - t0
        flags = wq4.wq4_device_status()
    finally:
        wq4.wq4_test_copy_stall()
    assert flags == PIPE_TIMEOUT, f"status {flags:#x}"
    assert 0.4 < took < 3.0               # a few limits of 0.5 s, however many tiles follow


# (N, K, M): whole K over several tiles a block in each token tile, one tile of
# fewer token blocks than epilogue groups, K split over a cluster
@pytest.mark.parametrize("stall", [GEMM_X, GEMM_W])
@pytest.mark.parametrize("N,K,M", [(28672, 512, 600), (16384, 1024, 1000), (1024, 256, 40), (512, 14336, 200)])
def test_gemm_without_its_copies_ends(N, K, M, stall):
    g = torch.Generator(device="cuda").manual_seed(N + M)
    W = torch.randint(-2**31, 2**31, (N, K // 8), generator=g, device="cuda", dtype=torch.int32)
    s = (0.005 + 0.015 * torch.rand((N, K // 32), generator=g, device="cuda")).half().view(torch.int16)
    x = torch.randn((M, K), generator=g, device="cuda").half().view(torch.int16)
    y = torch.empty((M, N), dtype=torch.int16, device="cuda")

    def call():
        wq4.wq4_gemm(W, s, x, y, N, K, M)

    call()
    torch.cuda.synchronize()
    ref = y.clone()
    _stalled(stall, call)
    y.zero_()
    call()
    torch.cuda.synchronize()
    assert wq4.wq4_device_status() == 0
    assert torch.equal(y, ref)


# one piece a block (merged over blocks), several pieces a block with more tiles
# than ring slots, an empty sequence among them
@pytest.mark.parametrize("lens", [[4096], [9000, 0, 3000, 1] * 8])
def test_attention_without_its_tiles_ends(lens):
    layer = PagedAttentionLayer(ModelShape("stall", 1, 4096, 512, 32, 8, 128, 1000), lens, seed=3)
    layer.run()
    torch.cuda.synchronize()
    ref = layer.out.clone()
    _stalled(ATTN, layer.run)
    layer.out.zero_()
    layer.run()
    torch.cuda.synchronize()
    assert wq4.wq4_device_status() == 0
    assert torch.equal(layer.out, ref)
