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
    # every layer five times, small and large blobs in turn (a CTA has some 33 units: a few wraps; test_many_units has the rest)
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


# rows, columns, stored width: a CTA has 14 to 44 units of an op, so that a chunk of K has more of them than may be on their way at
# once, a batch of copies straddles the end of the ring, and marks and places are used again
LONG = [(65536, 512, 2), (160000, 128, 8), (40000, 1024, 5), (160000, 256, 2), (65504, 512, 8), (100003, 384, 3), (40000, 1152, 8)]


def _random_layer(fq, i, n, k, bits):
    g = torch.Generator(device="cuda").manual_seed(1000 * i + bits)
    codes = torch.randint(0, 1 << bits, (n, k), dtype=torch.uint8, device="cuda", generator=g)
    scales = torch.rand((n, k // 128), device="cuda", generator=g).add_(0.5).mul_(2.0 ** -9).half()
    zeros = torch.randint(0, 1 << bits, (n, k // 128), device="cuda", generator=g).half()
    fq.fq_pack_layer(i, codes, scales, zeros, bits, P.FQ_FMT_PACKED)
    return codes, scales, zeros


@pytest.mark.parametrize("batch", [2, 4, 5, 8])
@pytest.mark.parametrize("ordered", [False, True])
def test_many_units(batch, ordered):
    fq = P.FlexQ(len(LONG))
    xs, want = [], []
    for i, (n, k, bits) in enumerate(LONG):
        codes, scales, zeros = _random_layer(fq, i, n, k, bits)
        xs.append(x_fp16(172, i, batch, k).cuda())
        w = (codes.double() - zeros.double().repeat_interleave(128, 1)) * scales.double().repeat_interleave(128, 1)
        want.append(xs[i].double() @ w.T)
        del w
    # 35 ops, about 700 units and 500 finished row pairs a CTA, widths in turn
    order = [(3 * j) % len(LONG) for j in range(5 * len(LONG))]
    ys = [torch.full((batch, LONG[i][0]), 7.0, dtype=torch.float16, device="cuda") for i in order]
    phases = [j // 3 for j in range(len(order))] if ordered else None
    for _ in range(2):
        fq.fq_gemv_stack(order, [xs[i] for i in order], ys, phases, batch)
        assert fq.fq_status() == 0
        for i, y in zip(order, ys):
            error = (y.double() - want[i]).norm(dim=1) / want[i].norm(dim=1)
            assert float(error.max()) <= GEMV_TOL
            y.fill_(7.0)
    fq.fq_destroy()


@pytest.mark.parametrize("batch", [2, 4, 5, 8])
def test_phases_carry_real_data(batch):
    """x of an op is y of the phase before, which holds no numbers until that has written it; two ops a phase, so that one of them
    is not the last that a CTA finishes.  The values are those of separate calls, launch after launch."""
    dims = [1024, 8192, 2048, 14336, 1152, 4096, 4736]           # k_in of the first phase, then n_out of every phase
    bits = [8, 4, 3, 5, 2, 6]
    fq = P.FlexQ(2 * len(bits))
    for i, b in enumerate(bits):
        for j in range(2):
            g = torch.Generator(device="cuda").manual_seed(2 * i + j)
            w = torch.randn((dims[i + 1] if j == 0 else 96, dims[i]), device="cuda", generator=g) / dims[i] ** 0.5
            fq.fq_pack_layer(2 * i + j, *P.fq_quantize_layer(w, b), b, P.FQ_FMT_PACKED)
    x0 = x_fp16(173, 0, batch, dims[0]).cuda()

    def outputs(i):
        return [torch.empty((batch, n), dtype=torch.float16, device="cuda") for n in (dims[i + 1], 96)]

    seq = [[x0]]
    for i in range(len(bits)):
        seq.append(outputs(i))
        for j in range(2):
            fq.fq_gemv_batched(2 * i + j, seq[i][0], seq[i + 1][j])
    torch.cuda.synchronize()
    assert all(torch.isfinite(t).all() and t.abs().max() > 0 for s in seq for t in s)
    bufs = [[x0]] + [outputs(i) for i in range(len(bits))]
    ops = [(i, j) for i in range(len(bits)) for j in (1, 0)]
    for rep in range(25):
        for pair in bufs[1:]:
            for t in pair:
                t.fill_(float("nan"))
        fq.fq_gemv_stack([2 * i + j for i, j in ops], [bufs[i][0] for i, j in ops], [bufs[i + 1][j] for i, j in ops], [i for i, j in ops], batch)
        torch.cuda.synchronize()
        for i in range(1, len(bufs)):
            assert all(torch.equal(a, b) for a, b in zip(bufs[i], seq[i])), (rep, i)
    assert fq.fq_status() == 0
    fq.fq_destroy()
