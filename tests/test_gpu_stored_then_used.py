"""Weights that are stored and used at once: fq_gemm straight after fq_pack_layer into the same buffer, nothing between the two."""
import pytest
import torch

import paper_2501_07139_b200 as P
from fq_testlib import make_layer, to_dev, x_bf16

pytestmark = pytest.mark.gpu


class Repacked:
    """A layer whose store is packed over and over, from two sets of codes in turn."""

    def __init__(self, n, k, m, bits, fmt):
        self.n, self.k, self.bits, self.fmt = n, k, bits, fmt
        self.fq = P.FlexQ(1)
        self.sets = [to_dev(*make_layer(181 + i, bits, n, k, bits)) for i in range(2)]
        self.store = self.fq.fq_pack_layer(0, *self.sets[0], bits, fmt)
        self.x = x_bf16(181, 0, m, k).cuda()
        self.want = []
        for i in range(2):
            torch.cuda.synchronize()
            self.pack(i)
            torch.cuda.synchronize()
            self.want.append(self.gemm(torch.zeros((m, n), dtype=torch.bfloat16, device="cuda")))
        torch.cuda.synchronize()
        assert not torch.equal(*self.want)

    def pack(self, i):
        c, s, z = self.sets[i]
        rc = P.lib().fq_pack_layer(self.fq._h, 0, self.n, self.k, self.bits, 128, self.fmt, c.data_ptr(), s.data_ptr(), z.data_ptr(),
                                   self.store.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == 0

    def gemm(self, y):
        return self.fq.fq_gemm(0, self.x, y)

    def outputs(self, count):
        return [torch.zeros_like(self.want[0]) for _ in range(count)]


# one stage of weights, a few, enough for every SM; the way that shares tiles and the one that does not; both formats
CASES = [(128, 128, 9, 4, P.FQ_FMT_PACKED), (96, 640, 77, 8, P.FQ_FMT_PLANES), (4096, 4096, 77, 3, P.FQ_FMT_PACKED), (2048, 1024, 300, 8, P.FQ_FMT_PACKED)]


@pytest.mark.parametrize("n,k,m,bits,fmt", CASES)
def test_packed_and_multiplied_at_once(n, k, m, bits, fmt):
    r = Repacked(n, k, m, bits, fmt)
    ys = r.outputs(48)
    for i, y in enumerate(ys):
        r.pack(i % 2)
        r.gemm(y)
        if i % 3 == 0:
            r.gemm(y)                                    # (the second call after a change is one that overlaps)
    torch.cuda.synchronize()
    assert all(torch.equal(y, r.want[i % 2]) for i, y in enumerate(ys))
    # on another stream: what was in order on one of them is not on the other
    other = torch.cuda.Stream()
    with torch.cuda.stream(other):
        for i, y in enumerate(ys):
            r.pack((i + 1) % 2)
            r.gemm(y)
    torch.cuda.synchronize()
    assert all(torch.equal(y, r.want[(i + 1) % 2]) for i, y in enumerate(ys))
    assert r.fq.fq_status() == 0
    r.fq.fq_destroy()


@pytest.mark.parametrize("n,k,m,bits,fmt", CASES[1:3])
def test_packed_and_multiplied_in_a_graph(n, k, m, bits, fmt):
    r = Repacked(n, k, m, bits, fmt)
    ys = r.outputs(8)
    # a multiplication that is captured right after weights were stored puts nothing in order for the calls that run at once
    only = torch.cuda.CUDAGraph()
    r.gemm(ys[0])
    torch.cuda.synchronize()
    with torch.cuda.graph(only):
        r.gemm(ys[7])
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        for i in range(7):
            r.pack(i % 2)
            if i % 2:
                only.replay()
            else:
                r.gemm(ys[7])
            r.gemm(ys[i])
    torch.cuda.synchronize()
    assert all(torch.equal(ys[i], r.want[i % 2]) for i in range(7))
    # storing and using in one graph
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for i, y in enumerate(ys):
            r.pack(i % 2)
            r.gemm(y)
    for _ in range(3):
        for y in ys:
            y.zero_()
        graph.replay()
        r.gemm(ys[0])                                    # (the graph's last weights)
        torch.cuda.synchronize()
        assert all(torch.equal(y, r.want[i % 2]) for i, y in enumerate(ys) if i)
        assert torch.equal(ys[0], r.want[1])
    assert r.fq.fq_status() == 0
    del only, graph
    r.fq.fq_destroy()
