"""The in-kernel attention of the decode step at batch 1-2, whose cached keys
and values come through the weight ring: the edges of its ranges (128 tokens
at least, at most 32 of them), ring chunks (a multiple of 16 tokens) and pages,
page sizes that are no power of two, every group size up to eight (the combine
takes four query heads at a time), and page ids outside the pool, which read
as zeros and are flagged.  Checked stage by stage as the other decode-step
tests do, with the oracle's tolerances."""
import numpy as np
import pytest
import torch

import oracle
from paper_2412_15803_gb300 import synth, wq4
from paper_2412_15803_gb300.model import DecodeModel, ModelShape, StepCaches
from test_decode_step_gpu import check_logits, run_step, step_and_check

pytestmark = pytest.mark.gpu


def shape(G, Hkv=1):
    return ModelShape(f"g{G}x{Hkv}", 2, 128 * G * Hkv, 512, G * Hkv, Hkv, 128, 300)


@pytest.mark.parametrize("positions", [[127], [128], [129], [31, 32], [255, 256], [257, 1], [4095], [4097, 640]])
@pytest.mark.parametrize("page_size", [16, 48])
def test_range_chunk_and_page_edges(positions, page_size):
    model, _, _, logits = step_and_check(shape(2), positions, seed=100 + positions[0], page_size=page_size)
    check_logits(model, logits)


@pytest.mark.parametrize("G", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("positions", [[40], [900, 333]])
def test_groups(G, positions):
    model, _, _, logits = step_and_check(shape(G, 1 + G % 2), positions, seed=200 + G, page_size=64)
    check_logits(model, logits)


@pytest.mark.parametrize("Hkv", [8, 32])
def test_more_units_than_ctas_and_single_ranges(Hkv):
    """Hkv = 8: nineteen ranges of every head; 32: four, at batch 2 two."""
    for positions in ([2500], [1100, 60]):
        model, _, _, logits = step_and_check(shape(1, Hkv), positions, seed=300 + Hkv)
        check_logits(model, logits)


@pytest.mark.parametrize("bad_id", [-1, 10 ** 6])
def test_bad_pages_read_as_zeros(bad_id):
    """A cached page outside the pool gives the result of a page of zeros, and
    is flagged (bit 4); the next valid step is clean."""
    sh = shape(4)
    model = DecodeModel(sh, batch=1, seed=400, step=True)
    caches = StepCaches(sh, [500], page_size=16, seed=401)
    x = synth.activations(402, 1, sh.hidden)
    xd = torch.from_numpy(x.view(np.int16)).cuda()
    logits = torch.empty((1, sh.vocab), dtype=torch.int16, device="cuda")
    good = caches.table.clone()
    for i in (3, 4, 17):
        caches.table[0, i] = bad_id
    model.decode_step(caches, xd, logits)
    torch.cuda.synchronize()
    assert wq4.wq4_device_status() & 16
    got = logits.cpu().numpy()
    caches.table.copy_(good)
    for l in range(sh.num_layers):
        for i in (3, 4, 17):
            page = int(caches.table_host[0, i])
            caches.k[l][page].zero_()
            caches.v[l][page].zero_()
    want = run_step(model, caches, x)
    assert np.array_equal(got.view(np.uint16), want)
    assert np.all(np.isfinite(oracle.half_to_double(want)))
