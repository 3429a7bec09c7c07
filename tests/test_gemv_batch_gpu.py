"""GPU parity of wq4_gemv at batch 2-32 at the edges of its kernels' tiles,
against the fp64 oracle: every element within
|y_gpu - y_ref| <= 1e-3 * sum_k |w x| + ulp16(|y_ref|).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2412_15803_gb300 import synth, wq4

pytestmark = pytest.mark.gpu


def check(N, K, batch, s_offset=0):
    W, s = synth.matrix(11 * N + K, N, K)
    x = synth.activations(N + K + batch, batch, K)
    sd = torch.zeros(s.size + s_offset, dtype=torch.int16, device="cuda")
    sd[s_offset:] = torch.from_numpy(s.ravel().view(np.int16)).cuda()
    y = torch.full((batch + 1, N), -1, dtype=torch.int16, device="cuda")   # a guard row after the outputs
    wq4.wq4_gemv(torch.from_numpy(W.view(np.int32)).cuda(), sd[s_offset:], torch.from_numpy(x.view(np.int16)).cuda(), y,
                 N, K, batch)
    torch.cuda.synchronize()
    assert wq4.wq4_device_status() == 0
    y_ref, A, _ = oracle.gemv(W, s, x)
    got = y.cpu().numpy()
    err = np.abs(oracle.half_to_double(got[:batch].view(np.uint16)) - y_ref)
    assert np.all(err <= oracle.tolerance(y_ref, A))
    assert np.all(got[batch] == -1)


# tensor-copy kernel: one row, a tile less one, odd row counts over several
# tiles, one box of K, chunks with a tail, batches at the edges of the tiles of
# eight activation rows
@pytest.mark.parametrize("batch", [3, 8, 9, 16, 17, 24, 25, 32])
@pytest.mark.parametrize("N,K", [(1, 256), (15, 512), (17, 768), (613, 2304), (2433, 1280)])
def test_tensor_copy_shapes(N, K, batch):
    check(N, K, batch)


@pytest.mark.parametrize("N,K", [(3072, 2816), (8193, 1024)])
def test_tensor_copy_batch_two(N, K):
    check(N, K, 2)


# copy-ring kernel: scales in pairs (K % 64 == 0), at any 2-byte address (odd
# group counts, a pointer off by one), chunks of one group
@pytest.mark.parametrize("batch", [3, 8, 13, 24, 32])
@pytest.mark.parametrize("N,K,off", [(1, 32, 0), (33, 96, 0), (40, 320, 0), (129, 1056, 0), (77, 2112, 0), (70, 512, 1),
                                     (1000, 1088, 1)])
def test_copy_ring_shapes(N, K, off, batch):
    check(N, K, batch, off)


def test_copy_ring_batch_two():
    check(3001, 2144, 2)


# more rows than whole rounds of the grid: the last round in tiles of 16 rows a
# warp (25-32 activation rows, three whole rounds and more; the last tail a
# row, a part, whole; one row too many for it)
@pytest.mark.parametrize("N,K,batch", [(116737, 256, 32), (116866, 512, 27), (128255, 512, 25),
                                       (136192, 256, 32), (136193, 256, 32)])
def test_tails_of_sixteen_rows(N, K, batch):
    check(N, K, batch)


# three row tiles a warp on sixteen warps (up to eight activation rows): whole,
# the third half used, a last tile of one row
@pytest.mark.parametrize("N,K", [(5121, 3072), (6153, 1024), (28672, 512), (7201, 768)])
@pytest.mark.parametrize("batch", [3, 8])
def test_three_row_tiles(N, K, batch):
    check(N, K, batch)


# few long rows at batch 2-4 on the CUDA cores: a row, an odd count, a warp's
# second row, the largest of the rule; K of one set of groups more than 4096
@pytest.mark.parametrize("batch,N,K", [(3, 1, 2048), (3, 75, 2304), (4, 76, 2048), (3, 153, 2816), (2, 1216, 7168), (3, 1215, 4352),
                                       (4, 607, 5632), (4, 1215, 4096), (3, 64, 28672), (4, 33, 20480)])
def test_few_long_rows(batch, N, K):
    check(N, K, batch)
