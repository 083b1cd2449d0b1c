"""Decode calls whose ops travel as kernel parameters (single calls, short lists without dependencies), and the batch kernel's
activation slots and zero points at their edges."""
import numpy as np
import pytest
import torch

from oracle import fq_oracle as O
from fq_testlib import GEMV_TOL, bits_of, f64_of, make_layer, to_dev, x_fp16

pytestmark = pytest.mark.gpu

# strips that stay whole; one strip that 28 CTAs share; two strips and a ragged one over an odd number of blobs; cut for evenness
SHAPES = [(512, 1024), (20, 14336), (70, 1664), (5120, 8192), (300, 128), (1000, 4224), (96, 2048), (33, 640), (64, 512)]


def _context(P, tag, shapes, nested=()):
    fq, data = P.FlexQ(len(shapes)), []
    bits = [2 + (i + tag) % 7 for i in range(len(shapes))]
    for i, (n, k) in enumerate(shapes):
        stored = 8 if i in nested else bits[i]
        c, s, z = make_layer(tag, i, n, k, stored)
        fq.fq_pack_layer(i, *to_dev(c, s, z), stored, P.FQ_FMT_PLANES if i in nested else P.FQ_FMT_PACKED)
        data.append((c, s, z, bits[i], i in nested))
    fq.fq_set_config(bits)
    return fq, data


def _ref(d, x):
    c, s, z, b, nested = d
    return O.gemv(c >> (8 - b), s, z, b, bits_of(x), parent_bits=8) if nested else O.gemv(c, s, z, b, bits_of(x))


@pytest.mark.parametrize("count", [1, 3, 8, 9])
def test_lists_without_dependencies(count):
    """Eight ops fit the kernel parameters, nine are uploaded as a table: both give what the allocation-free call gives, bit for
    bit, and the oracle's values, also when the list repeats and when a call follows before the previous one is done."""
    import paper_2501_07139_b200 as P
    shapes = SHAPES[:count]
    fq, data = _context(P, 130, shapes, nested=(2, 5))
    xs = [x_fp16(130, i, 1, k).cuda() for i, (n, k) in enumerate(shapes)]
    ys = [torch.full((1, n), float("nan"), dtype=torch.float16, device="cuda") for n, k in shapes]
    order = list(range(count))
    for _ in range(3):
        fq.fq_gemv_stack(order, xs, ys)
    singles = [torch.empty_like(y) for y in ys]
    for i in order:
        fq.fq_gemv(i, xs[i], singles[i])
    assert fq.fq_status() == 0
    for i in order:
        fixed = torch.empty_like(ys[i])
        fq.fq_gemv_static(i, xs[i], fixed)
        assert torch.equal(ys[i], fixed) and torch.equal(singles[i], fixed), i
        assert O.rel_l2(f64_of(ys[i])[0], _ref(data[i], xs[i])[0]) <= GEMV_TOL
    assert fq.fq_status() == 0
    fq.fq_destroy()


def test_captured_single_calls_replay():
    import paper_2501_07139_b200 as P
    shapes = SHAPES[1:3]
    fq, data = _context(P, 131, shapes)
    xs = [x_fp16(131, i, 1, k).cuda() for i, (n, k) in enumerate(shapes)]
    ys = [torch.zeros((1, n), dtype=torch.float16, device="cuda") for n, k in shapes]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for i in range(2):
            fq.fq_gemv(i, xs[i], ys[i])
    for seed in (5, 6):
        for i, (n, k) in enumerate(shapes):
            xs[i].copy_(x_fp16(131, 10 * seed + i, 1, k))
        graph.replay()
        torch.cuda.synchronize()
        for i in range(2):
            assert O.rel_l2(f64_of(ys[i])[0], _ref(data[i], xs[i])[0]) <= GEMV_TOL
    assert fq.fq_status() == 0
    del graph
    fq.fq_destroy()


@pytest.mark.parametrize("batch", [2, 4, 5, 7])
def test_batch_slots_with_infinities_and_short_ops(batch):
    """Activation slots are reused by ops of other lengths: what an op leaves beyond the columns of the next one (here
    infinities) must not reach its sums.  Widths 2..8, columns that do not fill a blob, rows that do not fill a strip."""
    import paper_2501_07139_b200 as P
    shapes = [(2048, 1024), (40, 128), (33, 640), (2048, 1024), (16, 1408), (70, 256), (200, 1152)]
    fq, data = _context(P, 132, shapes, nested=(2, 6))
    xs = [x_fp16(132, i, batch, k).cuda() for i, (n, k) in enumerate(shapes)]
    for i in (0, 3):
        xs[i][:, 100:] = float("inf")
    ys = [torch.full((batch, n), float("nan"), dtype=torch.float16, device="cuda") for n, k in shapes]
    for phases in (None, list(range(len(shapes)))):
        fq.fq_gemv_stack(list(range(len(shapes))), xs, ys, phases, batch)
        assert fq.fq_status() == 0
        for i in (1, 2, 4, 5, 6):
            want = _ref(data[i], xs[i])
            for b in range(batch):
                assert O.rel_l2(f64_of(ys[i])[b], want[b]) <= GEMV_TOL, (i, b)
    fq.fq_destroy()


@pytest.mark.parametrize("batch", [3, 8])
@pytest.mark.parametrize("bits", [2, 4, 5, 8])
def test_batch_zero_points_beyond_the_codes(bits, batch):
    """Zero points up to 1023 (the quantiser stays below 256): q - z is formed exactly all the same.  The weights of a group are
    then nearly equal and the sums cancel, so the reference takes the products (q - z) * s as they are: the oracle's rounding of
    each weight to fp16 is the same error 128 times over, 2^-11 of sums that are up to ten times the result.  What is left is
    the rounding of y (2^-11 of the value, 2.1e-4 in the norm) and fp32 sums (2^-23 of the terms' magnitudes)."""
    import paper_2501_07139_b200 as P
    n, k = 48, 384
    c, s, z = make_layer(133, bits, n, k, bits)
    rng = np.random.default_rng(bits)
    z = rng.integers(0, 1024, z.shape).astype(np.float16).view(np.uint16)
    fq = P.FlexQ(1)
    fq.fq_pack_layer(0, *to_dev(c, s, z), bits, P.FQ_FMT_PACKED)
    x = x_fp16(133, bits, batch, k).cuda()
    y = torch.empty((batch, n), dtype=torch.float16, device="cuda")
    fq.fq_gemv_batched(0, x, y)
    assert fq.fq_status() == 0
    scale, zero = (np.repeat(v.view(np.float16).astype(np.float64), 128, axis=1) for v in (s, z))
    want = f64_of(x) @ ((c.astype(np.float64) - zero) * scale).T
    for b in range(batch):
        assert O.rel_l2(f64_of(y)[b], want[b]) <= 5e-4
    fq.fq_destroy()
