"""Graphs that were captured before a context needed larger workspaces: a replay must find what it was captured with."""
import pytest
import torch

from oracle import fq_oracle as O
from fq_testlib import GEMM_TOL, GEMV_TOL, bits_of, f64_of, make_layer, to_dev, x_bf16, x_fp16

pytestmark = pytest.mark.gpu


def _random_layer(P, fq, i, n, k, bits, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    c, s, z = P.fq_quantize_layer(torch.randn((n, k), device="cuda", generator=gen).mul_(0.02), bits)
    fq.fq_pack_layer(i, c, s, z, bits, P.FQ_FMT_PACKED)


def _take_free_memory():
    """Device memory that was given back is taken and overwritten: who still used it would notice."""
    torch.cuda.synchronize()
    return [torch.full((mb << 20,), 0x7b, dtype=torch.uint8, device="cuda") for mb in (1, 2, 4, 8, 16, 32, 34, 48, 64, 72)]


def test_prefill_graph_and_a_larger_layer():
    """fq_gemm by way of a bf16 copy of the layer, captured once the room for it is there; then a larger layer asks for more."""
    import paper_2501_07139_b200 as P
    n, k, m = 9000, 4096, 2304
    fq = P.FlexQ(2)
    _random_layer(P, fq, 0, n, k, 4, 1)
    x = x_bf16(150, 0, m, k).cuda()
    y = torch.zeros((m, n), dtype=torch.bfloat16, device="cuda")
    free = torch.cuda.mem_get_info()[0]
    for _ in range(3):
        fq.fq_gemm(0, x, y)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] >= 2 * n * k, "this shape no longer takes the way that the test is about"
    eager = y.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fq.fq_gemm(0, x, y)
    _random_layer(P, fq, 1, 2 * n, k, 4, 2)
    y1 = torch.zeros((m, 2 * n), dtype=torch.bfloat16, device="cuda")
    for _ in range(3):
        fq.fq_gemm(1, x, y1)
    larger = y1.clone()
    junk = _take_free_memory()
    for _ in range(2):
        y.zero_()
        graph.replay()
        fq.fq_gemm(1, x, y1)
        torch.cuda.synchronize()
        assert torch.equal(y, eager) and torch.equal(y1, larger)
    assert all(int(j.min()) == 0x7b and int(j.max()) == 0x7b for j in junk)
    assert fq.fq_status() == 0
    del graph
    fq.fq_destroy()


def test_decode_graph_and_a_growing_workspace():
    """Captured single calls and a short list, with strips that several CTAs share (their sums and counters are in the workspace);
    then a layer is packed that needs a larger workspace.  Graph and eager calls take turns afterwards, on new activations."""
    import paper_2501_07139_b200 as P
    shapes = [(512, 1024), (20, 14336), (5120, 8192)]
    bits = [4, 3, 5]
    fq = P.FlexQ(4)
    layers = [make_layer(151, i, n, k, b) for i, ((n, k), b) in enumerate(zip(shapes[:2], bits))]
    for i, l in enumerate(layers):
        fq.fq_pack_layer(i, *to_dev(*l), bits[i], P.FQ_FMT_PACKED)
    xs = [x_fp16(151, i, 1, k).cuda() for i, (n, k) in enumerate(shapes)]
    ys = [torch.zeros((1, n), dtype=torch.float16, device="cuda") for n, k in shapes]
    listed = [torch.zeros_like(y) for y in ys]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for i in range(2):
            fq.fq_gemv(i, xs[i], ys[i])
        fq.fq_gemv_stack([0, 1], xs[:2], listed[:2])
    _random_layer(P, fq, 2, *shapes[2], bits[2], 3)
    _random_layer(P, fq, 3, 8192, 14336, 4, 4)
    junk = _take_free_memory()
    eager = torch.empty_like(ys[1])
    for seed in (1, 2, 3):
        for i in range(2):
            xs[i].copy_(x_fp16(151, 10 * seed + i, 1, shapes[i][1]))
        graph.replay()
        fq.fq_gemv(1, xs[1], eager)
        fq.fq_gemv(2, xs[2], ys[2])
        torch.cuda.synchronize()
        for i in range(2):
            want = O.gemv(*layers[i], bits[i], bits_of(xs[i]))[0]
            assert O.rel_l2(f64_of(ys[i])[0], want) <= GEMV_TOL and torch.equal(ys[i], listed[i])
        assert torch.equal(eager, ys[1])
    assert all(int(j.min()) == 0x7b and int(j.max()) == 0x7b for j in junk)
    assert fq.fq_status() == 0
    del graph
    fq.fq_destroy()
