"""The one-kernel way of fq_gemm where it shares tiles, and where it has more whole tiles than the GPU has SMs.  Every test asks
how the shape is run first, so that another choice of the library cannot leave it without a subject."""
import numpy as np
import pytest
import torch

import fq_synth as S
from oracle import fq_oracle as O
from fq_testlib import GEMM_TOL, bits_of, f64_of, x_bf16

pytestmark = pytest.mark.gpu

# (outputs, columns, tokens, bits): one token tile and many; ragged outputs; a last token tile that is not full
SHARED = [(4096, 4096, 77, 4), (4096, 11008, 77, 3), (4096, 11008, 300, 5), (1000, 9984, 45, 8), (700, 14336, 161, 6)]


def _layer(P, n, k, bits, seed):
    w = S.weight_rows(S.tensor_key(156, seed, S.TENSOR_W), 0, n, k, device="cuda")
    c, s, z = P.fq_quantize_layer(w, bits)
    fq = P.FlexQ(1)
    fq.fq_pack_layer(0, c, s, z, bits, P.FQ_FMT_PACKED)

    def rows(cols, x):
        return O.gemm(c[cols].cpu().numpy(), bits_of(s[cols]), bits_of(z[cols]), bits, bits_of(x))
    return fq, rows


def _runs(plan, k):
    """Per block: the pieces (tile, first pair, end) of its run of (tile, K stage) pairs."""
    steps = k // 128
    pairs = plan["tiles"] * steps
    base, extra = divmod(pairs, plan["blocks"])
    out = []
    for b in range(plan["blocks"]):
        lo, hi = b * base + min(b, extra), (b + 1) * base + min(b + 1, extra)
        out.append([(t, max(lo, t * steps) - t * steps, min(hi, (t + 1) * steps) - t * steps) for t in range(lo // steps, (hi - 1) // steps + 1)])
    return out, steps


def _same_product(fq, x, y, n):
    """Element by element beside the two-pass way, whose sums are formed in another order: the last bit of a few may differ."""
    other = torch.empty((x.shape[0], n), dtype=torch.bfloat16, device="cuda") if n % 8 == 0 else None
    if other is None:
        other = torch.empty((x.shape[0], n + 8 - n % 8), dtype=torch.bfloat16, device="cuda")[:, :n]
    fq.fq_gemm_two_pass(0, x, other)
    assert fq.fq_status() == 0
    a, b = y.float(), other.float()
    assert bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 1e-3 * b.pow(2).mean().sqrt()).all())
    assert float((a != b).float().mean()) < 0.02
    return other


@pytest.mark.parametrize("shape", SHARED)
def test_shared_tiles(shape):
    """Blocks whose runs begin in one tile and end in another contribute to both; whoever is last adds the sums up.  Every element,
    sampled outputs against the oracle, the same bits in every repetition, and nothing beside the outputs."""
    import paper_2501_07139_b200 as P
    n, k, m, bits = shape
    fq, rows = _layer(P, n, k, bits, m)
    plan = fq.fq_gemm_plan(0, m)
    assert not plan["two_pass"] and plan["shared"], plan
    runs, steps = _runs(plan, k)
    two = sum(len(r) > 1 and r[0][2] - r[0][1] < steps and r[-1][2] - r[-1][1] < steps for r in runs)
    assert two >= 5, "no block has parts of two tiles"
    x = x_bf16(156, m, m, k).cuda()
    y = torch.full((m + 2, (n + 7) // 8 * 8 + 8), float("nan"), dtype=torch.bfloat16, device="cuda")
    view = y[1:m + 1, :n]
    fq.fq_gemm(0, x, view)
    first = view.clone()
    assert torch.isnan(y[0].float()).all() and torch.isnan(y[m + 1].float()).all() and torch.isnan(y[:, n:].float()).all()
    _same_product(fq, x, first, n)
    cols = sorted({0, 31, 127, 128, n - 1} | set(np.random.default_rng(m).integers(0, n, 40).tolist()))
    assert O.rel_l2(f64_of(first[:, cols]), rows(cols, x)) <= GEMM_TOL
    for _ in range(40):
        fq.fq_gemm(0, x, view)
        fq.fq_gemv(0, *_vectors(n, k))                       # (another kernel in between, which overlaps)
    assert torch.equal(view, first) and fq.fq_status() == 0
    fq.fq_destroy()


_kept = {}


def _vectors(n, k):
    if (n, k) not in _kept:
        _kept[n, k] = (torch.zeros((1, k), dtype=torch.float16, device="cuda"), torch.zeros((1, n), dtype=torch.float16, device="cuda"))
    return _kept[n, k]


def test_more_whole_tiles_than_sms():
    """Three waves of whole tiles, ragged in both directions: the two ways add up in the same order, so they agree bit for bit."""
    import paper_2501_07139_b200 as P
    n, k, m = 11000, 1024, 601
    fq, rows = _layer(P, n, k, 3, 1)
    plan = fq.fq_gemm_plan(0, m)
    assert not plan["two_pass"] and not plan["shared"], plan
    assert plan["tiles"] > 2 * torch.cuda.get_device_properties(0).multi_processor_count == 2 * plan["blocks"], plan
    x = x_bf16(156, 1, m, k).cuda()
    y = torch.full((m, n), float("nan"), dtype=torch.bfloat16, device="cuda")
    for _ in range(2):
        fq.fq_gemm(0, x, y)
    assert torch.equal(y, _same_product(fq, x, y, n))
    cols = [0, 127, 128, 5503, n - 1]
    assert O.rel_l2(f64_of(y[:, cols]), rows(cols, x)) <= GEMM_TOL
    fq.fq_destroy()


def test_long_prompts_take_two_passes():
    import paper_2501_07139_b200 as P
    fq, _ = _layer(P, 4096, 4096, 4, 2)
    assert fq.fq_gemm_plan(0, 8192)["two_pass"] and not fq.fq_gemm_plan(0, 16)["two_pass"]
    for layer, tokens, code in ((0, 0, -3), (1, 16, -1)):
        with pytest.raises(P.FlexQError) as e:
            fq.fq_gemm_plan(layer, tokens)
        assert e.value.code == code
    fq.fq_destroy()
