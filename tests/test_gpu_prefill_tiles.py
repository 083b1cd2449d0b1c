"""Prefill at the edges of its tiles: token counts around one and two tiles, outputs that do not fill a tile or a stored row
pair, the shortest K, tiles that many CTAs share, tiles that stay whole under capture, and both ways to the same product."""
import numpy as np
import pytest
import torch

from oracle import fq_oracle as O
from fq_testlib import GEMM_TOL, bits_of, f64_of, make_layer, to_dev, x_bf16

pytestmark = pytest.mark.gpu


def _layer(P, tag, n, k, bits, fmt):
    stored = 8 if fmt == P.FQ_FMT_PLANES else bits
    codes, s, z = make_layer(tag, bits, n, k, stored)
    fq = P.FlexQ(1)
    fq.fq_pack_layer(0, *to_dev(codes, s, z), stored, fmt)
    fq.fq_set_config([bits])
    if fmt == P.FQ_FMT_PLANES:
        return fq, lambda x: O.gemm(codes >> (8 - bits), s, z, bits, bits_of(x), parent_bits=8)
    return fq, lambda x: O.gemm(codes, s, z, bits, bits_of(x))


def _check(fq, ref, x, n, call=None):
    m = x.shape[0]
    y = torch.full((m + 2, (n + 7) // 8 * 8 + 8), float("nan"), dtype=torch.bfloat16, device="cuda")
    view = y[1:m + 1, :n]
    (call or fq.fq_gemm)(0, x, view)
    assert fq.fq_status() == 0
    got, want = f64_of(view), ref(x)
    assert np.all(np.isfinite(got))
    assert O.rel_l2(got, want) <= GEMM_TOL
    assert np.max(np.abs(got - want)) <= 4 * GEMM_TOL * np.max(np.abs(want))
    # nothing beside the outputs is written
    assert torch.isnan(y[0].float()).all() and torch.isnan(y[m + 1].float()).all() and torch.isnan(y[:, n:].float()).all()
    return view


@pytest.mark.parametrize("m", [1, 16, 17, 159, 160, 161, 193, 321])
@pytest.mark.parametrize("shape", [(129, 128), (24, 2176), (264, 640)])
def test_token_counts_and_ragged_outputs(m, shape):
    import paper_2501_07139_b200 as P
    n, k = shape
    fq, ref = _layer(P, 120, n, k, 4, P.FQ_FMT_PACKED)
    for _ in range(2):                                      # the second call finds the first one's counters
        _check(fq, ref, x_bf16(120, m, m, k).cuda(), n)
    fq.fq_destroy()


@pytest.mark.parametrize("fmt_bits", [(0, 2), (0, 3), (0, 5), (0, 7), (0, 8), (1, 2), (1, 3), (1, 5), (1, 8)])
def test_every_field_list_with_shared_tiles(fmt_bits):
    """Two row tiles and 34 K stages: 17 CTAs share a tile, runs begin and end inside blobs (none in two tiles: those are
    test_gpu_prefill_plan.py's)."""
    import paper_2501_07139_b200 as P
    fmt, bits = fmt_bits
    n, k, m = 200, 34 * 128, 37
    fq, ref = _layer(P, 121, n, k, bits, fmt)
    _check(fq, ref, x_bf16(121, bits, m, k).cuda(), n)
    fq.fq_destroy()


def test_shared_tiles_do_not_depend_on_timing():
    import paper_2501_07139_b200 as P
    n, k, m = 640, 9984, 77
    fq, ref = _layer(P, 122, n, k, 4, P.FQ_FMT_PACKED)
    assert fq.fq_gemm_plan(0, m)["shared"] and not fq.fq_gemm_plan(0, m)["two_pass"]
    x = x_bf16(122, 0, m, k).cuda()
    first = _check(fq, ref, x, n).clone()
    y = torch.empty((m, n), dtype=torch.bfloat16, device="cuda")
    for _ in range(50):
        fq.fq_gemm(0, x, y)
    assert torch.equal(y, first) and fq.fq_status() == 0
    fq.fq_destroy()


@pytest.mark.parametrize("m", [40, 1030])
def test_captured_calls_replay(m):
    """A graph of two calls, replayed on new activations: whatever the first call would allocate is not there yet."""
    import paper_2501_07139_b200 as P
    n, k = 520, 1280
    fq, ref = _layer(P, 123, n, k, 3, P.FQ_FMT_PACKED)
    x = torch.zeros((m, k), dtype=torch.bfloat16, device="cuda")
    y = [torch.zeros((m, n), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for o in y:
            fq.fq_gemm(0, x, o)
    for seed in (1, 2):
        new = x_bf16(123, seed, m, k).cuda()
        x.copy_(new)
        graph.replay()
        torch.cuda.synchronize()
        want = ref(new)
        for o in y:
            assert O.rel_l2(f64_of(o), want) <= GEMM_TOL
    assert fq.fq_status() == 0
    del graph
    fq.fq_destroy()


@pytest.mark.parametrize("shape", [(300, 256, 257), (1040, 384, 600), (5120, 128, 2048)])
def test_pair_tiles(shape):
    """The GEMM of the two-pass way: ragged against 256 tokens and every width of its output tiles."""
    import paper_2501_07139_b200 as P
    n, k, m = shape
    fq, ref = _layer(P, 124, n, k, 5, P.FQ_FMT_PACKED)
    _check(fq, ref, x_bf16(124, m, m, k).cuda(), n, fq.fq_gemm_two_pass)
    fq.fq_destroy()
