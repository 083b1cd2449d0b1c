"""Nested children at batch 1: every position that a code can have in the stored words, one at a time."""
import numpy as np
import pytest
import torch

import paper_2501_07139_b200 as P

pytestmark = pytest.mark.gpu

N, K = 48, 640                       # a whole strip and a half; a whole blob and a quarter of the next


@pytest.mark.parametrize("bits", range(2, 9))
def test_one_hot_columns(bits):
    """x is 1 in one column: y is that column's dequantised weight, rounded once to fp16 (the sums have one term)."""
    rng = np.random.default_rng(bits)
    codes = rng.integers(0, 256, size=(N, K), dtype=np.uint8)
    scales = (rng.integers(1024, 2048, size=(N, K // 128)) * 2.0 ** -20).astype(np.float16)
    zeros = rng.integers(0, 256, size=(N, K // 128)).astype(np.float16)
    fq = P.FlexQ(1)
    fq.fq_pack_layer(0, torch.from_numpy(codes).cuda(), torch.from_numpy(scales).cuda(), torch.from_numpy(zeros).cuda(), 8, P.FQ_FMT_PLANES)
    fq.fq_set_config([bits])
    step = 1 << (8 - bits)
    child = (codes.astype(np.int64) // step) * step + step // 2
    group = np.arange(K) // 128
    want = ((child - zeros.astype(np.int64)[:, group]) * scales.astype(np.float64)[:, group]).astype(np.float16)
    # all four columns of a lane, both halves of a step, all eight steps of a superstep, both supersteps, the second blob
    columns = sorted({32 * j + p for j in range(16) for p in (0, 5, 17, 30)} | {512, 547, 639})
    x = torch.zeros((len(columns), K), dtype=torch.float16, device="cuda")
    for i, k in enumerate(columns):
        x[i, k] = 1.0
    y = torch.zeros((len(columns), N), dtype=torch.float16, device="cuda")
    for i in range(len(columns)):
        fq.fq_gemv(0, x[i], y[i])
    assert fq.fq_status() == 0
    assert np.array_equal(y.cpu().numpy(), want[:, columns].T)
