"""fq_gemm behind a kernel that lets its successors begin long before it ends."""
import pytest
import torch

import paper_2501_07139_b200 as P
from oracle import fq_oracle as O
from fq_testlib import GEMM_TOL, bits_of, f64_of, make_layer, to_dev, x_bf16

pytestmark = pytest.mark.gpu

# lets the next kernel begin, then takes its time and writes what that one reads
SLOW = r"""
extern "C" __global__ void slow_copy(const unsigned* from, unsigned* to, int words, int ms)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    do {
        __nanosleep(100000);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    } while (t - t0 < 1000000ull * ms);
    for (int i = threadIdx.x; i < words; i += blockDim.x) to[i] = from[i];
}
"""


@pytest.mark.parametrize("n,k,m", [(128, 128, 40), (1000, 2048, 77)])
def test_the_time_limit_begins_when_the_previous_kernel_has_ended(n, k, m):
    """Waits of fq_gemm have a limit of two seconds, none of which the previous kernel uses up; X is read only when that has ended."""
    bits = 5
    fq = P.FlexQ(1)
    layer = make_layer(183, 0, n, k, bits)
    fq.fq_pack_layer(0, *to_dev(*layer), bits, P.FQ_FMT_PACKED)
    x = x_bf16(183, 0, m, k).cuda()
    late, y = torch.zeros_like(x), torch.empty((m, n), dtype=torch.bfloat16, device="cuda")
    slow = torch.cuda._compile_kernel(SLOW, "slow_copy")
    fq.fq_gemm(0, late, y)                               # (from the second call on launches overlap)
    torch.cuda.synchronize()
    slow((1, 1, 1), (256, 1, 1), (x, late, m * k // 2, 2300))
    fq.fq_gemm(0, late, y)
    assert fq.fq_status() == 0
    want = O.gemm(*layer, bits, bits_of(x[:3]))
    assert O.rel_l2(f64_of(y)[:3], want) <= GEMM_TOL
    again = torch.empty_like(y)
    fq.fq_gemm(0, x, again)
    torch.cuda.synchronize()
    assert torch.equal(y, again)
    fq.fq_destroy()
