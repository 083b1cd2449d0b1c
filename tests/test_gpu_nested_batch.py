"""Nested children at batch 2..8: every position that a code can have in the stored words, one column per batch entry."""
import numpy as np
import pytest
import torch

import paper_2501_07139_b200 as P

pytestmark = pytest.mark.gpu

N, K = 48, 640                       # a whole strip and a half; a whole blob and a quarter of the next


def _nested(bits):
    """A nested layer with a child of that many bits active, and the child's weights as fp16 rounds them."""
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
    return fq, ((child - zeros.astype(np.int64)[:, group]) * scales.astype(np.float64)[:, group]).astype(np.float16)


# all four columns of a lane, both halves of a step, all eight steps of a superstep, both supersteps, the second blob
COLUMNS = sorted({32 * j + p for j in range(16) for p in (0, 5, 17, 30)} | {512, 547, 639})


@pytest.mark.parametrize("batch", [2, 4, 5, 8])
@pytest.mark.parametrize("bits", range(2, 9))
def test_one_hot_columns_of_a_batch(bits, batch):
    """x is 1 in one column of an entry: q - z, the product and the sum of one term are exact up to the rounding of y."""
    fq, want = _nested(bits)
    for i in range(0, len(COLUMNS), batch):
        columns = (COLUMNS + COLUMNS[:batch])[i:i + batch]
        x = torch.zeros((batch, K), dtype=torch.float16, device="cuda")
        for b, k in enumerate(columns):
            x[b, k] = 1.0
        y = torch.full((batch, N), 7.0, dtype=torch.float16, device="cuda")
        fq.fq_gemv_batched(0, x, y)
        assert np.array_equal(y.cpu().numpy(), want[:, columns].T)
    assert fq.fq_status() == 0
