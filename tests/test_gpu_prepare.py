"""The quantiser's single-precision quotients and the blob packer at the places where they could go wrong."""
import numpy as np
import pytest
import torch

import fq_synth as S
from oracle import fq_oracle as O
from fq_testlib import bits_of, make_layer, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [2, 5, 8])
@pytest.mark.parametrize("shape", [(1, 128), (3, 384), (65, 1152)])
def test_quantizer_on_rounding_boundaries(bits, shape):
    """Every quotient on or one ulp beside a tie, codes that clamp, and groups with infinite or huge values: the same
    integers as the oracle, which divides in double.  Group counts that leave a warp's last groups empty."""
    import paper_2501_07139_b200 as P
    n, k = shape
    qmax = 2 ** bits - 1
    rng = np.random.default_rng(bits)
    scale = np.float32(2.0 ** -9 * 1.25)
    half = (rng.integers(-qmax, qmax, (n, k)) + 0.5).astype(np.float32) * scale
    w = np.nextafter(half, np.where(rng.random((n, k)) < 0.5, -np.inf, np.inf).astype(np.float32))
    w = np.where(rng.random((n, k)) < 0.4, half, w).astype(np.float32)
    w[:, 0], w[:, 1] = 0.0, qmax * scale                     # the first group of every row gets exactly this scale
    w[:, 2:128] = np.clip(w[:, 2:128], 0.0, qmax * scale)
    if n > 1:
        w[1, 5] = np.inf
        w[2, 7], w[2, 8] = 3e38, -3e38
        w[2, 200] = 1e-42
    rc, rs, rz = O.quantize(w, bits)
    c, s, z = P.fq_quantize_layer(torch.from_numpy(w).cuda(), bits)
    assert np.array_equal(c.cpu().numpy(), rc)
    assert np.array_equal(bits_of(s), rs) and np.array_equal(bits_of(z), rz)


def test_quantizer_not_a_number():
    """A NaN takes no part in the group's range and gets code 0."""
    import paper_2501_07139_b200 as P
    w = S.weight_rows(S.tensor_key(95, 0, S.TENSOR_W), 0, 4, 256).numpy().copy()
    w[2, 130] = w[2, 131]
    rc, rs, rz = O.quantize(w, 4)
    rc[2, 130] = 0
    w[2, 130] = np.nan
    c, s, z = P.fq_quantize_layer(torch.from_numpy(w).cuda(), 4)
    assert np.array_equal(c.cpu().numpy(), rc)
    assert np.array_equal(bits_of(s), rs) and np.array_equal(bits_of(z), rz)


@pytest.mark.parametrize("shape", [(1, 128), (33, 640), (64, 512), (95, 1408)])
@pytest.mark.parametrize("bits", [2, 3, 7, 8])
def test_pack_from_any_address(bits, shape):
    """Codes at an address that no wide load may start at, rows and columns that do not fill a blob."""
    import paper_2501_07139_b200 as P
    n, k = shape
    codes, s, z = make_layer(96, bits, n, k, bits)
    d = to_dev(codes, s, z)
    off = torch.zeros(n * k + 16, dtype=torch.uint8, device="cuda")
    shifted = off[3:3 + n * k].view(n, k)
    shifted.copy_(d[0])
    fq = P.FlexQ(2)
    a = fq.fq_pack_layer(0, d[0], d[1], d[2], bits, P.FQ_FMT_PACKED)
    b = fq.fq_pack_layer(1, shifted, d[1], d[2], bits, P.FQ_FMT_PACKED)
    assert torch.equal(a, b)
    out = fq.fq_export_layer(1, bits, n, k).cpu().numpy().view(np.uint32).reshape(n, -1)
    assert np.array_equal(out, O.pack_bitstream(codes, bits))
    fq.fq_destroy()
