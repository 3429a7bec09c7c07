"""Rows of a decode step that map another row's new token as a cached one (two
consecutive tokens of a sequence in one step, a page in two sequences): the
definition appends every row first, then attends, at batch 2 (whose cached
tokens are copied ahead of the appends) as at 3 and more.  Checked stage by
stage against the oracle on the caches as the step left them."""
import numpy as np
import pytest
import torch

from paper_2412_15803_gb300 import synth, wq4
from paper_2412_15803_gb300.model import DecodeModel, ModelShape, StepCaches
from test_decode_step_gpu import check_step_layer, run_step

pytestmark = pytest.mark.gpu


def _check(G, Hkv, positions, page_size, seed, edit):
    sh = ModelShape(f"shared{G}x{Hkv}", 2, 128 * G * Hkv, 512, G * Hkv, Hkv, 128, 300)
    model = DecodeModel(sh, batch=len(positions), seed=seed, step=True)
    caches = StepCaches(sh, positions, page_size=page_size, seed=seed + 1, spare_pages=3, rope_theta=10000.0)
    edit(caches.table_host)
    caches.table.copy_(torch.from_numpy(caches.table_host))
    x = synth.activations(seed + 2, len(positions), sh.hidden)
    first = None
    for _ in range(2):                        # the second step rewrites the same rows
        before = [caches.host_cache(l) for l in range(sh.num_layers)]
        logits = run_step(model, caches, x)
        assert wq4.wq4_device_status() == 0
        for l in range(sh.num_layers):
            check_step_layer(model, caches, l, before[l], u=x if l == 0 else None)
        assert first is None or np.array_equal(first, logits)
        first = logits


# consecutive tokens either way round, at the edges of blocks, pages, ring
# chunks and ranges; a token far back
@pytest.mark.parametrize("positions", [[0, 1], [15, 16], [17, 16], [127, 128], [129, 128], [300, 301], [2047, 2048], [4094, 4095],
                                       [100, 900], [900, 31]])
@pytest.mark.parametrize("page_size", [16, 48])
def test_two_tokens_of_one_sequence(positions, page_size):
    longer = int(np.argmax(positions))

    def edit(table):
        table[1 - longer] = table[longer]

    _check(2, 2, positions, page_size, 500 + positions[0], edit)


@pytest.mark.parametrize("G", [1, 3, 5, 8])
def test_groups(G):
    _check(G, 1 + G % 2, [640, 641], 16, 520 + G, lambda table: table.__setitem__(0, table[1]))


def test_page_mapped_twice():
    """Row 1 maps the page of row 0's new token at two places of its own."""
    def edit(table):
        table[1, 3] = table[1, 11] = table[0, 70 // 16]

    _check(4, 1, [70, 700], 16, 540, edit)


def test_three_rows():
    """The graph path: three consecutive tokens of one sequence."""
    def edit(table):
        table[0] = table[1] = table[2]

    _check(4, 1, [200, 201, 202], 16, 560, edit)
