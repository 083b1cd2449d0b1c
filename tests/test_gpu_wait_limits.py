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
@pytest.mark.parametrize("batch", [1, 2, 4, 5, 8])
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


def test_single_calls_after_a_launch_that_gave_up():
    """The counters of strips that single calls share lie where the phases' counters do: a launch that gave up leaves nothing behind."""
    import paper_2501_07139_b200 as P
    n, k = 40, 14336                                        # two strips for all CTAs
    fq = P.FlexQ(2)
    a, b = make_layer(153, 0, n, k, 4), make_layer(153, 1, 512, 512, 4)
    fq.fq_pack_layer(0, *to_dev(*a), 4, P.FQ_FMT_PACKED)
    fq.fq_pack_layer(1, *to_dev(*b), 4, P.FQ_FMT_PACKED)
    x, xb = x_fp16(153, 0, 1, k).cuda(), x_fp16(153, 1, 1, 512).cuda()
    y, first, yb = (torch.zeros((1, m), dtype=torch.float16, device="cuda") for m in (n, n, 512))
    fq.fq_gemv(0, x, first)
    assert fq.fq_status() == 0 and O.rel_l2(f64_of(first)[0], O.gemv(*a, 4, bits_of(x))[0]) <= GEMV_TOL
    for _ in range(3):
        fq.fq_set_wait_limit_ns(1)
        fq.fq_gemv_stack([1, 0], [xb, x], [yb, y], [0, 1])
        fq.fq_gemv(0, x, y)                                 # (may give up too)
        assert fq.fq_status() == -8
        fq.fq_set_wait_limit_ns(0)
        y.zero_()
        fq.fq_gemv(0, x, y)
        assert fq.fq_status() == 0 and torch.equal(y, first)
    fq.fq_destroy()
