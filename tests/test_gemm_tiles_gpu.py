"""GPU parity of wq4_gemm at the edges of its token tiles, K splits and row
tiles, against the fp64 oracle: every element within
|y_gpu - y_ref| <= 1e-3 * sum_k |w x| + ulp16(|y_ref|).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2412_15803_gb300 import synth, wq4

pytestmark = pytest.mark.gpu


def run(W, s, x, N, K, M):
    y = torch.full((M + 1, N), -1, dtype=torch.int16, device="cuda")   # a guard row after the outputs
    wq4.wq4_gemm(torch.from_numpy(W.view(np.int32)).cuda(), torch.from_numpy(s.view(np.int16)).cuda(),
                 torch.from_numpy(x.view(np.int16)).cuda(), y, N, K, M)
    torch.cuda.synchronize()
    y = y.cpu().numpy()
    assert np.all(y[M] == -1)
    return y[:M].view(np.uint16)


def check(N, K, M, rows=None):
    W, s = synth.matrix(5 * N + K + M, N, K)
    x = synth.activations(N + K + M, M, K)
    y = run(W, s, x, N, K, M)
    assert wq4.wq4_device_status() == 0
    rows = np.arange(N) if rows is None else rows
    y_ref, A, _ = oracle.gemv(W[rows], s[rows], x)
    err = np.abs(oracle.half_to_double(y[:, rows]) - y_ref)
    assert np.all(err <= oracle.tolerance(y_ref, A))


# tokens at the edges of the tiles (and of the GEMV kernels' 16), rows at the
# edges of the row tiles; K of one block, of an uneven split, of a deep one
@pytest.mark.parametrize("M", [1, 16, 17, 63, 65, 128, 130, 193, 257])
@pytest.mark.parametrize("N,K", [(8, 256), (136, 768), (264, 2816)])
def test_tile_edges(N, K, M):
    check(N, K, M)


@pytest.mark.parametrize("N,K,M", [(128, 8192, 40), (512, 3328, 100), (1024, 2560, 200), (640, 4096, 250)])
def test_split_k(N, K, M):
    """Few tiles and a long K: the cluster split, every token, sampled rows;
    the same bits twice."""
    rows = np.unique(np.concatenate([[0, 1, 127, N - 1], np.random.default_rng(N).integers(0, N, 20)]))
    check(N, K, M, rows)
    W, s = synth.matrix(1, N, K)
    x = synth.activations(2, M, K)
    assert np.array_equal(run(W, s, x, N, K, M), run(W, s, x, N, K, M))


def test_more_tiles_than_sms():
    """Several tiles a CTA, the last round partial, a ragged last token tile."""
    N, K, M = 8320, 512, 700
    check(N, K, M, np.unique(np.concatenate([[0, 127, 128, N - 1], np.random.default_rng(0).integers(0, N, 30)])))


@pytest.mark.parametrize("M", [5, 16, 40, 300])
@pytest.mark.parametrize("bad_row", [0, 23, 135])
def test_large_scale_is_flagged(M, bad_row):
    """One scale beyond +-8188 in any row sets bit 6 of the status word, on the
    GEMV kernels (up to 16 tokens) as on the tensor-core tiles; a scale of
    exactly 8188 does not."""
    N, K = 136, 512
    W, s = synth.matrix(3, N, K)
    x = (synth.activations(4, M, K).view(np.float16) * np.float16(1e-3)).view(np.uint16)
    s = s.copy()
    s[bad_row, K // 32 - 1] = 0x6FFF
    run(W, s, x, N, K, M)
    assert wq4.wq4_device_status() == 0
    s[bad_row, K // 32 - 1] = 0x7000
    run(W, s, x, N, K, M)
    assert wq4.wq4_device_status() == 64
