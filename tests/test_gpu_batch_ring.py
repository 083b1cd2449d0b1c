"""Batch 2..8: units of different sizes in one ring, from one chunk of K to more than the output warps load at once."""
import pytest
import torch

import paper_2501_07139_b200 as P
from oracle import fq_oracle as O
from fq_testlib import GEMV_TOL, bits_of, f64_of, make_layer, to_dev, x_fp16

pytestmark = pytest.mark.gpu

# rows, columns, stored width: one chunk; a ragged second one; 12, 13 and 14 chunks (twelve are loaded at once); rows for every SM
SHAPES = [(96, 512, 8), (33, 640, 3), (64, 6144, 2), (40, 6528, 7), (32, 7168, 8), (4800, 1024, 8), (4777, 896, 2), (4768, 1024, 5)]


@pytest.mark.parametrize("batch", [2, 4, 5, 8])
@pytest.mark.parametrize("ordered", [False, True])
def test_mixed_units(batch, ordered):
    fq = P.FlexQ(len(SHAPES))
    layers = [make_layer(171, i, n, k, b) for i, (n, k, b) in enumerate(SHAPES)]
    for i, (n, k, b) in enumerate(SHAPES):
        fq.fq_pack_layer(i, *to_dev(*layers[i]), b, P.FQ_FMT_PACKED)
    xs = [x_fp16(171, i, batch, k).cuda() for i, (n, k, b) in enumerate(SHAPES)]
    want = [O.gemv(*layers[i], b, bits_of(xs[i])) for i, (n, k, b) in enumerate(SHAPES)]
    # every layer five times, small and large blobs in turn: the ring wraps at every remainder
    order = [(3 * j) % len(SHAPES) for j in range(5 * len(SHAPES))]
    ys = [torch.full((batch, SHAPES[i][0]), 7.0, dtype=torch.float16, device="cuda") for i in order]
    phases = [j // 2 for j in range(len(order))] if ordered else None
    fq.fq_gemv_stack(order, [xs[i] for i in order], ys, phases, batch)
    assert fq.fq_status() == 0
    for i, y in zip(order, ys):
        for b in range(batch):
            assert O.rel_l2(f64_of(y)[b], want[i][b]) <= GEMV_TOL
    # a layer by itself gives the same bits
    for i in range(len(SHAPES)):
        y = torch.zeros((batch, SHAPES[i][0]), dtype=torch.float16, device="cuda")
        fq.fq_gemv_batched(i, xs[i], y)
        assert torch.equal(y, ys[order.index(i)])
