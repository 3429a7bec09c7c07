"""GPU parity of paged decode attention at the edges of its work split: shares
cut at the segments' ends, shares of the flat tile list, and the change from
one to the other, against the fp64 oracle."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2412_15803_gb300 import synth, wq4

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv", [(8, 8), (24, 8), (32, 4)])
@pytest.mark.parametrize("lens", [
    [16], [129], [128 * 9 + 1], [4000],                    # one sequence: whole tiles, a tile over, many parts
    [1] * 40, [17] * 40, [300, 0, 1, 2000, 0],               # as many segments as blocks and more, empty ones
    [40, 0] * 38, [40, 0, 7] * 38, [40, 0] * 76, [40] * 77,  # as many as blocks and one sequence more (8 and 4 heads)
    [64 * k + 1 for k in range(1, 20)],                      # a fair share that no cut at the ends fits
    [2500 + 7 * k for k in range(12)],                        # large shares
])
def test_shares(Hq, Hkv, lens):
    P, D = 16, 128
    lens = np.asarray(lens, np.int32)
    pages = int(((lens + P - 1) // P).sum()) + 1
    k, v = synth.kv_cache(9, pages, Hkv, P, D)
    table = synth.page_table(9, lens, P, pages)
    q = synth.queries(9, len(lens), Hq, D)
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a).view(t)).cuda()
    kd, vd, td, qd, ld = dev(k, np.int16), dev(v, np.int16), dev(table, np.int32), dev(q, np.int16), dev(lens, np.int32)
    out = torch.full((len(lens), Hq * D), -1, dtype=torch.int16, device="cuda")
    ws = torch.zeros(wq4.wq4_paged_attention_workspace_bytes(len(lens), Hq, Hkv, D), dtype=torch.uint8, device="cuda")
    cache = wq4.kv_cache_desc(kd, vd, td, P)
    scale = 1.0 / math.sqrt(D)
    first = None
    for _ in range(2):                                      # the counters are left zero; the same bits twice
        wq4.wq4_paged_attention(cache, qd, Hq * D, ld, out, Hq * D, len(lens), Hq, scale, ws, ws.numel())
        torch.cuda.synchronize()
        got = out.cpu().numpy().view(np.uint16)
        assert first is None or np.array_equal(first, got)
        first = got.copy()
    assert wq4.wq4_device_status() == 0
    o_ref, A, _ = oracle.paged_attention(q, k, v, table, lens, scale, Hq)
    err = np.abs(oracle.half_to_double(first.reshape(len(lens), Hq, D)) - o_ref)
    assert np.all(err <= oracle.attention_tolerance(o_ref, A))
