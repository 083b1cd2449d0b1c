"""Prefill with zero points of any size."""
import numpy as np
import pytest
import torch

from oracle import fq_oracle as O
from fq_testlib import f64_of, make_layer, to_dev, x_bf16

pytestmark = pytest.mark.gpu

ZEROS = [0, 127, 1023, 1024, 1025, 1501, 2047, 2049, 4095, 20000, 65504]


@pytest.mark.parametrize("two_pass", [False, True])
@pytest.mark.parametrize("fmt_bits", [(0, 2), (0, 5), (0, 7), (0, 8), (1, 2), (1, 5), (1, 7), (1, 8)])
def test_zero_points_of_any_size(fmt_bits, two_pass):
    """The reference rounds the exact products (q - z) * s to bf16 once, as the kernels do; what is left is fp32 sums (2^-23 of the
    terms' magnitudes, 30 times the result) and the rounding of Y (2^-9 of the value, 1.7e-3 in the norm)."""
    import paper_2501_07139_b200 as P
    fmt, bits = fmt_bits
    n, k, m = 75, 640, 40
    stored = 8 if fmt == P.FQ_FMT_PLANES else bits
    c, s, z = make_layer(155, bits, n, k, stored)
    z = np.array(ZEROS, dtype=np.float16)[np.random.default_rng(bits).integers(0, len(ZEROS), z.shape)].view(np.uint16)
    fq = P.FlexQ(1)
    fq.fq_pack_layer(0, *to_dev(c, s, z), stored, fmt)
    fq.fq_set_config([bits])
    x = x_bf16(155, bits, m, k).cuda()
    y = torch.full((m, n + 5), float("nan"), dtype=torch.bfloat16, device="cuda")
    (fq.fq_gemm_two_pass if two_pass else fq.fq_gemm)(0, x, y[:, :n])
    assert fq.fq_status() == 0
    q = c.astype(np.float64)
    if bits < stored:
        step = 2.0 ** (stored - bits)
        q = np.floor(q / step) * step + step / 2
    scale, zero = (np.repeat(v.view(np.float16).astype(np.float64), 128, axis=1) for v in (s, z))
    w = torch.from_numpy((q - zero) * scale).float().bfloat16().double().numpy()      # (exact in fp32 up to 13-bit integers, then within 2^-24)
    want, size = f64_of(x) @ w.T, np.abs(f64_of(x)) @ np.abs(w).T
    got = f64_of(y)[:, :n]
    assert O.rel_l2(got, want) <= 2.5e-3
    assert np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 2e-6 * size + 2.0 ** -9 * 1e-3 * size)
    fq.fq_destroy()
