"""The first long prompts of a context: the bf16 copy of a layer goes through memory that the context has, in parts."""
import numpy as np
import pytest
import torch

import fq_synth as S
from oracle import fq_oracle as O
from fq_testlib import GEMM_TOL, bits_of, f64_of, x_bf16

pytestmark = pytest.mark.gpu


def _layer(P, fq, i, n, k, bits):
    w = S.weight_rows(S.tensor_key(154, i, S.TENSOR_W), 0, n, k, device="cuda")
    c, s, z = P.fq_quantize_layer(w, bits)
    fq.fq_pack_layer(i, c, s, z, bits, P.FQ_FMT_PACKED)
    return c, s, z


@pytest.mark.parametrize("shape", [(9000, 4096, 2304), (1800, 14336, 1800), (2000, 2048, 1600)])
def test_first_calls(shape):
    """A ragged layer that needs four parts, one that needs three of another height, one that fits: the first call allocates nothing, and the
    first, the second (which asks for room of its own) and the later ones give the same bits, the oracle's within tolerance."""
    import paper_2501_07139_b200 as P
    n, k, m = shape
    x = x_bf16(154, m, m, k).cuda()
    calls = 4
    y = torch.full((calls, m, (n + 7) // 8 * 8 + 8), float("nan"), dtype=torch.bfloat16, device="cuda")
    for rep in range(2):                                    # (the first time kernels are loaded, which takes memory too)
        y.fill_(float("nan"))
        fq = P.FlexQ(1)
        layer = _layer(P, fq, 0, n, k, 4)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        fq.fq_gemm(0, x, y[0][:, :n])
        torch.cuda.synchronize()
        assert rep == 0 or torch.cuda.mem_get_info()[0] == free
        for i in range(1, calls):
            fq.fq_gemm(0, x, y[i][:, :n])
        assert fq.fq_status() == 0
        fq.fq_destroy()
    assert torch.isnan(y[:, :, n:].float()).all()
    assert all(torch.equal(y[0][:, :n], y[i][:, :n]) for i in range(1, calls))
    rows = [0, 127, 128, 1023, m - 1]
    cols = sorted({0, 31, 32, n // 2, n - 1} | set(np.random.default_rng(1).integers(0, n, 40).tolist()))
    c, s, z = (t.cpu().numpy() for t in (layer[0][cols], layer[1][cols], layer[2][cols]))
    want = O.gemm(c, s.view(np.uint16), z.view(np.uint16), 4, bits_of(x[rows]))
    assert O.rel_l2(f64_of(y[0][rows][:, cols]), want) <= GEMM_TOL


def test_first_call_captured():
    """A graph that was captured on a fresh context, replayed after the context has got room of its own."""
    import paper_2501_07139_b200 as P
    n, k, m = 4200, 4096, 2304
    fq = P.FlexQ(1)
    _layer(P, fq, 0, n, k, 4)
    x = x_bf16(154, 1, m, k).cuda()
    y, z = (torch.zeros((m, n), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fq.fq_gemm(0, x, y)
    for seed in (2, 3, 4):
        x.copy_(x_bf16(154, seed, m, k))
        graph.replay()
        fq.fq_gemm(0, x, z)
        torch.cuda.synchronize()
        assert torch.equal(y, z)
    assert fq.fq_status() == 0
    del graph
    fq.fq_destroy()
