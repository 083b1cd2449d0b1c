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
