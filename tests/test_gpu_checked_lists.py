"""The bounds-checked build on short lists of decode calls (their ops are kernel parameters) and on short prompts whose tiles are
shared: no check fires, and the results are those of the normal build."""
import os
import subprocess
import sys

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

pytestmark = pytest.mark.gpu


def _run(P):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    shapes = [(512, 1024), (20, 14336), (70, 1664), (4096, 4096), (300, 128), (1000, 4224), (96, 2048), (33, 640)]
    fq, out = P.FlexQ(len(shapes)), {}
    for i, (n, k) in enumerate(shapes):
        c, s, z = P.fq_quantize_layer(torch.randn((n, k), device="cuda", generator=gen).mul_(0.02), 2 + i % 7)
        fq.fq_pack_layer(i, c, s, z, 2 + i % 7, P.FQ_FMT_PACKED)
    xs = [torch.randn((1, k), device="cuda", generator=gen).half() for n, k in shapes]
    for count in (1, 3, 8):
        ys = [torch.zeros((1, n), dtype=torch.float16, device="cuda") for n, k in shapes[:count]]
        fq.fq_gemv_stack(list(range(count)), xs[:count], ys)
        assert fq.fq_status() == 0, count
        out.update({f"list{count}_{i}": y.cpu() for i, y in enumerate(ys)})
    for i, m in ((3, 77), (3, 300), (5, 19)):
        x = torch.randn((m, shapes[i][1]), device="cuda", generator=gen).bfloat16()
        y = torch.zeros((m, shapes[i][0]), dtype=torch.bfloat16, device="cuda")
        fq.fq_gemm(i, x, y)
        assert fq.fq_status() == 0, (i, m)
        out[f"gemm{i}_{m}"] = y.cpu()
    fq.fq_destroy()
    return out


def test_checked_build_on_lists_and_short_prompts(tmp_path):
    import paper_2501_07139_b200 as P
    normal = _run(P)
    out = tmp_path / "checked.pt"
    r = subprocess.run([sys.executable, os.path.abspath(__file__), str(out)], env=dict(os.environ, FLEXQ_LIBRARY="checked"),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    checked = torch.load(out)
    assert set(checked) == set(normal)
    for key in normal:
        assert torch.equal(normal[key], checked[key]), key


if __name__ == "__main__":
    import paper_2501_07139_b200 as P
    assert os.path.basename(P.lib_path()) == "libflexq_checked.so", P.lib_path()
    torch.save(_run(P), sys.argv[1])
