"""Waits of the decode kernels that run out: the launch reports it and returns, and the context works afterwards."""
import pytest
import torch

from oracle import fq_oracle as O
from fq_testlib import GEMV_TOL, bits_of, f64_of, make_layer, to_dev, x_fp16

pytestmark = pytest.mark.gpu

SHAPES = [(256, 512), (1056, 4096), (96, 512), (512, 2304), (130, 512), (2048, 1280)]
BITS = [3, 8, 5, 4, 6, 2]
PHASES = [0, 0, 0, 1, 2, 3]


@pytest.mark.parametrize("limit", [1, 500])
@pytest.mark.parametrize("batch", [2, 4, 5, 8])
def test_ordered_stack_gives_up_and_recovers(batch, limit):
    """Limits that no wait for a phase can meet: some role gives up, and where a role does while another one has copies on their
    way, those land before the CTA leaves.  Several launches one after the other, then the status, then the right values."""
    import paper_2501_07139_b200 as P
    fq = P.FlexQ(len(SHAPES))
    layers = [make_layer(152, i, n, k, b) for i, ((n, k), b) in enumerate(zip(SHAPES, BITS))]
    for i, (l, b) in enumerate(zip(layers, BITS)):
        fq.fq_pack_layer(i, *to_dev(*l), b, P.FQ_FMT_PACKED)
    xs = [x_fp16(152, i, batch, k).cuda() for i, (n, k) in enumerate(SHAPES)]
    ys = [torch.zeros((batch, n), dtype=torch.float16, device="cuda") for n, k in SHAPES]
    order = list(range(len(SHAPES)))
    fq.fq_gemv_stack(order, xs, ys, PHASES, batch)
    assert fq.fq_status() == 0
    want = [y.clone() for y in ys]
    for i in order:
        ref = O.gemv(*layers[i], BITS[i], bits_of(xs[i]))
        assert all(O.rel_l2(f64_of(ys[i])[b], ref[b]) <= GEMV_TOL for b in range(batch))
    fq.fq_set_wait_limit_ns(limit)
    for _ in range(3):
        fq.fq_gemv_stack(order, xs, ys, PHASES, batch)
    assert fq.fq_status() == -8
    assert fq.fq_status() == 0
    fq.fq_set_wait_limit_ns(0)
    for _ in range(2):
        for y in ys:
            y.zero_()
        fq.fq_gemv_stack(order, xs, ys, PHASES, batch)
        assert fq.fq_status() == 0
        assert all(torch.equal(y, w) for y, w in zip(ys, want))
    fq.fq_destroy()
