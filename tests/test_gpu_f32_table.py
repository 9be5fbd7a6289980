"""Mode "f32" reads only the coefficients of its table. A table of the caller's
own, which may hold level means, takes the mean + perturbation arithmetic."""
import numpy as np
import pytest

from paper_2107_13500_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2107_13500_gb300 import build, pw
    build.build()
    pw.load_library()
    return torch


@pytest.mark.parametrize("aligned", [True, False])
def test_f32_with_a_mean_table_is_the_split_form(gpu, aligned):
    from paper_2107_13500_gb300 import pw
    torch = gpu
    nx, ny, nz = 133, 9, 11
    dz = synth.dz_stretched(nz)
    c = pw.make_coeffs(nz, 50.0, 40.0, dz).to_device()
    f = [pw.field_from_numpy(a, nx, aligned=aligned) for a in synth.fields_modes(nx, ny, nz, 50.0, 40.0, dz, seed=4)]
    fp, means = zip(*(pw.split_field(t, nx, ny, out=pw.empty_field(nx, ny, nz, torch.float32, aligned=aligned)) for t in f))
    table = torch.from_numpy(pw.make_split_table(c, *(m.cpu().numpy() for m in means))).cuda()
    want = pw.advect(*fp, c, nx, ny, mode="split", split_table=table)
    got = pw.advect(*fp, c, nx, ny, mode="f32", split_table=table)
    plain = pw.advect(*fp, c, nx, ny, mode="f32")
    doms = [dict(u=fp[0], v=fp[1], w=fp[2], nx=nx, ny=ny, coeffs=c, split_table=t) for t in (table, None)]
    b = pw.Batch(doms, "f32", 0)
    b.run()
    one = pw.Batch(doms[1:], "f32", 0)
    one.run()
    torch.cuda.synchronize()
    assert pw.device_status() == 0
    assert b.dt == pw.PW_F32_SPLIT and one.dt == pw.PW_F32
    scale = max(float(t.abs().max()) for t in plain)
    for w_, g, bb, p, oo, bp in zip(want, got, b.outputs()[0], plain, one.outputs()[0], b.outputs()[1]):
        assert torch.equal(g, w_) and torch.equal(bb, w_) and torch.equal(oo, p)
        assert not torch.equal(g, p)
        # the second domain of the mixed batch: zero means through the general
        # form; each product rounded once more or less, of sums of six terms
        assert float((bp - p).abs().max()) <= 64 * 2.0 ** -24 * scale
