"""Values of the batch decode kernel at the edges of what the calls accept: zero points of any size, activations
that are no numbers."""
import numpy as np
import pytest
import torch

from oracle import fq_oracle as O
from fq_testlib import GEMV_TOL, bits_of, f64_of, make_layer, to_dev, x_fp16

pytestmark = pytest.mark.gpu

ZEROS = [0, 127, 1023, 1024, 1025, 1501, 2047, 2049, 4095, 20000, 65504]      # (fp16 holds 2047 and 2048, not 2049 or 4095)


@pytest.mark.parametrize("batch", [2, 3, 4, 5, 8])
@pytest.mark.parametrize("fmt_bits", [(0, 2), (0, 3), (0, 5), (0, 8), (1, 2), (1, 5), (1, 8)])
def test_zero_points_of_any_size(fmt_bits, batch):
    """w^ = (q - z) * s for every integer z that fp16 holds, a different one per row and group.  The reference takes the products
    as they are; what is left is the rounding of y (2^-11 of the value, 2.1e-4 in the norm) and fp32 sums, 2^-23 of terms
    whose magnitudes add up to some 20 times the result."""
    import paper_2501_07139_b200 as P
    fmt, bits = fmt_bits
    n, k = 75, 1152
    stored = 8 if fmt == P.FQ_FMT_PLANES else bits
    c, s, z = make_layer(134, bits, n, k, stored)
    rng = np.random.default_rng(bits)
    s = (s.view(np.float16) / np.float16(16)).view(np.uint16)               # (65504 codes times the activations stay below fp16's largest)
    z = np.array(ZEROS, dtype=np.float16)[rng.integers(0, len(ZEROS), z.shape)].view(np.uint16)
    z[:, 3] = np.float16(5).view(np.uint16)                                 # groups beside them that need nothing special
    fq = P.FlexQ(1)
    fq.fq_pack_layer(0, *to_dev(c, s, z), stored, fmt)
    fq.fq_set_config([bits])
    x = x_fp16(134, bits, batch, k).cuda()
    y = torch.full((batch, n), float("nan"), dtype=torch.float16, device="cuda")
    fq.fq_gemv_batched(0, x, y)
    assert fq.fq_status() == 0
    q = c.astype(np.float64)
    if bits < stored:
        step = 2.0 ** (stored - bits)
        q = np.floor(q / step) * step + step / 2
    scale, zero = (np.repeat(v.view(np.float16).astype(np.float64), 128, axis=1) for v in (s, z))
    want = f64_of(x) @ ((q - zero) * scale).T
    assert np.max(np.abs(want)) < 60000
    for b in range(batch):
        assert O.rel_l2(f64_of(y)[b], want[b]) <= 5e-4
        # row by row too: a row of small zero points must not hide behind the large ones
        assert np.all(np.abs(f64_of(y)[b] - want[b]) <= 2.0 ** -10 * np.abs(want[b]) + 2e-6 * np.abs(f64_of(x)[b]) @ np.abs((q - zero) * scale).T)
    fq.fq_destroy()


def _high(tag, n, k, bits):
    """A layer with zero points of 1301 here and there, and its exact weights."""
    c, s, z = make_layer(tag, bits, n, k, bits)
    z = np.where(np.random.default_rng(tag).random(z.shape) < 0.3, np.float16(1301), z.view(np.float16)).astype(np.float16).view(np.uint16)
    scale, zero = (np.repeat(v.view(np.float16).astype(np.float64), 128, axis=1) for v in (s, z))
    return (c, s, z), (c - zero) * scale


def test_zero_points_that_come_later(tmp_path):
    """High zero points that are stored after calls have run without any, that come from a file, and that a swap brings in.  A layer
    of ordinary ones beside them keeps its values bit for bit."""
    import paper_2501_07139_b200 as P
    n, k, batch, bits = 200, 1280, 3, 8
    plain, (high, w) = make_layer(136, 0, n, k, bits), _high(137, n, k, bits)
    x = x_fp16(136, 0, batch, k).cuda()

    def check(fq, layer, want):
        y = torch.full((batch, n), float("nan"), dtype=torch.float16, device="cuda")
        fq.fq_gemv_batched(layer, x, y)
        assert fq.fq_status() == 0
        if isinstance(want, torch.Tensor):
            assert torch.equal(y, want)
        else:
            assert all(O.rel_l2(f64_of(y)[b], want[b]) <= 5e-4 for b in range(batch))
        return y

    fq = P.FlexQ(2)
    fq.fq_pack_layer(0, *to_dev(*plain), bits, P.FQ_FMT_PACKED)
    want = f64_of(x) @ w.T
    ys = [check(fq, 0, O.gemv(*plain, bits, bits_of(x))) for _ in range(3)]
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2])
    store = fq.fq_pack_layer(1, *to_dev(*high), bits, P.FQ_FMT_PACKED)
    for _ in range(2):
        check(fq, 1, want)
        check(fq, 0, ys[0])
    path = str(tmp_path / "high.flexq")
    fq.fq_save(path)
    loaded = P.FlexQ(2)
    loaded.fq_load(path)
    swapped = P.FlexQ(1)
    host = store.cpu().pin_memory()
    swapped.fq_host_variant(0, n, k, bits, host)
    swapped.fq_transition_swap([bits])
    for _ in range(2):
        check(loaded, 1, want)
        check(loaded, 0, ys[0])
        check(swapped, 0, want)
    for f in (fq, loaded, swapped):
        f.fq_destroy()


def test_zero_points_that_a_graph_stores():
    """A captured fq_pack_layer stores high zero points after calls have run without any; a captured decode call runs after they were
    stored eagerly."""
    import paper_2501_07139_b200 as P
    n, k, batch, bits = 75, 1152, 4, 8
    low, (high, w) = make_layer(138, 0, n, k, bits), _high(138, n, k, bits)
    x = x_fp16(138, 0, batch, k).cuda()
    want = f64_of(x) @ w.T

    def setup():
        fq = P.FlexQ(1)
        store = fq.fq_pack_layer(0, *to_dev(*low), bits, P.FQ_FMT_PACKED)
        dev = to_dev(*high)

        def pack():
            assert P.lib().fq_pack_layer(fq._h, 0, n, k, bits, 128, P.FQ_FMT_PACKED, *(t.data_ptr() for t in dev), store.data_ptr(),
                                         torch.cuda.current_stream().cuda_stream) == 0

        return fq, pack, dev

    def decode(fq, y):
        fq.fq_gemv_batched(0, x, y)

    y = torch.zeros((batch, n), dtype=torch.float16, device="cuda")
    fq, pack, keep = setup()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pack()
    for _ in range(3):
        decode(fq, y)
        assert fq.fq_status() == 0
    graph.replay()
    for _ in range(2):
        decode(fq, y)
        assert fq.fq_status() == 0
        assert all(O.rel_l2(f64_of(y)[b], want[b]) <= 5e-4 for b in range(batch))
    del graph
    fq.fq_destroy()

    fq, pack, keep = setup()
    for _ in range(3):
        decode(fq, y)
        assert fq.fq_status() == 0
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        decode(fq, y)
    pack()
    graph.replay()
    assert fq.fq_status() == 0
    assert all(O.rel_l2(f64_of(y)[b], want[b]) <= 5e-4 for b in range(batch))
    del graph
    fq.fq_destroy()


@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("batch", [1, 2, 4, 5, 8])
def test_an_activation_that_is_no_number(batch, bad):
    """One infinite or NaN activation makes every output of its batch entry NaN and leaves the other entries alone, wherever it
    stands: in the last columns of a layer that ends inside a blob, and in a layer that is too wide for the batch-1 kernel, where one
    entry takes the same way.  A second op follows in the same launch: nothing of it is touched."""
    import paper_2501_07139_b200 as P
    k = 16384 if batch == 1 else 1408
    fq = P.FlexQ(2)
    layers = [make_layer(135, 0, 70, k, 4), make_layer(135, 1, 33, k, 8)]
    for i, (l, bits) in enumerate(zip(layers, (4, 8))):
        fq.fq_pack_layer(i, *to_dev(*l), bits, P.FQ_FMT_PACKED)
    xs = [x_fp16(135, i, batch, k).cuda() for i in range(2)]
    entry = batch - 1
    for at in (3, k - 1):
        x = xs[0].clone()
        x[entry, at] = bad
        ys = [torch.zeros((batch, n), dtype=torch.float16, device="cuda") for n in (70, 33)]
        fq.fq_gemv_stack([0, 1], [x, xs[1]], ys, [0, 1], batch)
        assert fq.fq_status() == 0
        assert torch.isnan(ys[0][entry].float()).all()
        want = [O.gemv(*l, bits, bits_of(v)) for l, bits, v in zip(layers, (4, 8), xs)]
        for b in range(batch):
            assert b == entry or O.rel_l2(f64_of(ys[0])[b], want[0][b]) <= GEMV_TOL
            assert O.rel_l2(f64_of(ys[1])[b], want[1][b]) <= GEMV_TOL
    fq.fq_destroy()
