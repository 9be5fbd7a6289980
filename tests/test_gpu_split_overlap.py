"""pw_split_field's three launches overlap: back to back on one stream, on
other outputs and replayed from a CUDA graph they give the bits of a single
synchronised call."""
import pytest
import torch

from paper_2107_13500_gb300 import pw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (33, 5, 3), (127, 17, 64), (130, 250, 9)])
def test_split_field_overlapped(shape):
    nx, ny, nz = shape
    gen = torch.Generator(device="cuda").manual_seed(5)
    fields = []
    for _ in range(4):
        f = pw.empty_field(nx, ny, nz, torch.float64)
        f.copy_(torch.rand(f.shape, generator=gen, device="cuda", dtype=torch.float64).mul_(20.0).sub_(7.0))
        fields.append(f)
    want = []
    for f in fields:
        p, m = pw.split_field(f, nx, ny)
        torch.cuda.synchronize()
        want.append((p.clone(), m.clone()))

    # back to back, each field's output written again by the next call on it
    out = [pw.split_field(f, nx, ny)[0] for f in fields]
    means = [torch.empty(nz, dtype=torch.float64, device="cuda") for _ in fields]
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    for f, p, m in zip(fields * 3, out * 3, means * 3):
        pw.split_field(f, nx, ny, out=p, mean=m)
    torch.cuda.synchronize()
    for p, m, (wp, wm) in zip(out, means, want):
        assert torch.equal(p, wp) and torch.equal(m, wm)

    with torch.cuda.graph(graph):
        for f, p, m in zip(fields, out, means):
            pw.split_field(f, nx, ny, out=p, mean=m)
    for t in out + means:
        t.zero_()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for p, m, (wp, wm) in zip(out, means, want):
        assert torch.equal(m, wm)
        assert torch.equal(p[:, :, :nx + 2], wp[:, :, :nx + 2])
