"""Lists at batch 1 whose shares of a thread block are unusual: a blob or two of a matrix, hundreds of strips of a phase."""
import pytest
import torch

import paper_2501_07139_b200 as P
from fq_testlib import x_fp16

pytestmark = pytest.mark.gpu


def random_layer(fq, i, n, k, bits):
    g = torch.Generator(device="cuda").manual_seed(1000 * i + bits)
    w = torch.randn((n, k), device="cuda", generator=g)
    fq.fq_pack_layer(i, *P.fq_quantize_layer(w, bits), bits, P.FQ_FMT_PACKED)


# rows and columns of the layers, ops of the list, ops to a phase (0: no phases).  14336 columns are 28 blobs, as many as activation slots:
# a block that has the last blob of one op and the first ones of the next needs the same slots twice within its first items.
#   64 x one strip      : twelve blobs a block, of one op or two
#   3 x 99 strips       : two strips and a blob or two of a third one a block and phase
#   widths in turn      : slots of the next phase's activations come before those of this one are taken
LISTS = [([(32, 14336)] * 4, 64, 0), ([(3168, 14336)] * 3, 12, 3), ([(3168, 14336), (96, 512), (4800, 2048)], 24, 3), ([(640, 14336), (64, 128)], 40, 1)]


@pytest.mark.parametrize("shapes,n_ops,per_phase", LISTS)
def test_a_blob_or_two_of_a_matrix(shapes, n_ops, per_phase):
    fq = P.FlexQ(len(shapes))
    for i, (n, k) in enumerate(shapes):
        random_layer(fq, i, n, k, 2)
    order = [j % len(shapes) for j in range(n_ops)]
    xs = [x_fp16(184, j, 1, shapes[i][1]).cuda() for j, i in enumerate(order)]
    want = [fq.fq_gemv(i, x, torch.empty((1, shapes[i][0]), dtype=torch.float16, device="cuda")) for i, x in zip(order, xs)]
    phases = [j // per_phase for j in range(n_ops)] if per_phase else None
    for _ in range(20):
        ys = [torch.full_like(w, 7.0) for w in want]
        fq.fq_gemv_stack(order, xs, ys, phases)
        torch.cuda.synchronize()
        assert all(torch.equal(y, w) for y, w in zip(ys, want))
    assert fq.fq_status() == 0
    fq.fq_destroy()


def test_hundreds_of_strips_of_a_phase():
    """A phase of which every block finishes more than 255 strips; the next one reads its outputs, which are no numbers before."""
    n, k, ops = 65536, 128, 24                           # 24 x 2048 strips: 332 a block of 148
    fq = P.FlexQ(2)
    random_layer(fq, 0, n, k, 2)
    random_layer(fq, 1, 640, 14336, 4)
    x = x_fp16(185, 0, 1, k).cuda()
    want = fq.fq_gemv(0, x, torch.empty((1, n), dtype=torch.float16, device="cuda"))
    ends = [want[:, -14336:].clone(), want[:, :14336].clone()]
    after = [fq.fq_gemv(1, e, torch.empty((1, 640), dtype=torch.float16, device="cuda")) for e in ends]
    torch.cuda.synchronize()
    assert all(torch.isfinite(a).all() for a in after)
    ys = [torch.empty_like(want) for _ in range(ops)]
    last = [torch.empty_like(a) for a in after]
    for _ in range(10):
        for y in ys:
            y.fill_(float("nan"))
        fq.fq_gemv_stack([0] * ops + [1, 1], [x] * ops + [ys[-1][:, -14336:], ys[0][:, :14336]], ys + last, [0] * ops + [1, 1])
        torch.cuda.synchronize()
        assert all(torch.equal(y, want) for y in ys)
        assert all(torch.equal(a, b) for a, b in zip(last, after))
    assert fq.fq_status() == 0
    fq.fq_destroy()


def test_more_rows_than_twenty_bits_of_strips():
    """33.5 million outputs are 2^20 strips; the layer has a few more."""
    n, k, bits = (1 << 25) + 2000, 128, 2
    fq = P.FlexQ(1)
    codes = torch.randint(0, 4, (n, k), dtype=torch.uint8, device="cuda", generator=torch.Generator(device="cuda").manual_seed(7))
    scales = torch.full((n, 1), 2.0 ** -6, dtype=torch.float16, device="cuda")
    zeros = torch.ones((n, 1), dtype=torch.float16, device="cuda")
    fq.fq_pack_layer(0, codes, scales, zeros, bits, P.FQ_FMT_PACKED)
    x = x_fp16(186, 0, 1, k).cuda()
    ys = [torch.full((1, n), float("nan"), dtype=torch.float16, device="cuda") for _ in range(2)]
    fq.fq_gemv(0, x, ys[0])
    fq.fq_gemv_stack([0], [x], ys[1:], [0])
    assert fq.fq_status() == 0
    for rows in (slice(0, 70000), slice((1 << 25) - 70000, n)):
        want = ((codes[rows].double() - 1) * 2.0 ** -6) @ x[0].double()
        for y in ys:
            assert float((y[0, rows].double() - want).norm() / want.norm()) <= 1e-3
    assert torch.equal(ys[0], ys[1])
    fq.fq_destroy()
