"""A float batch plan launched as the other float dtype is reported, as
pw_advect_batched documents: PW_F32 leaves the mean terms out."""
import pytest

from paper_2107_13500_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("built,launched", [("split", "f32"), ("f32", "split"), ("f32", "f32"), ("split", "split")])
@pytest.mark.parametrize("variant", [0, 7])
def test_float_plans_belong_to_their_dtype(built, launched, variant):
    import torch
    from paper_2107_13500_gb300 import build, pw
    build.build()
    nx, ny, nz = 40, 11, 9
    c = pw.make_coeffs(nz, 50.0, 50.0, synth.dz_stretched(nz)).to_device()
    f = [pw.field_from_numpy(a, nx, torch.float32) for a in synth.fields_iid(nx, ny, nz, seed=2)]
    table = torch.from_numpy(pw.make_split_table(c, *([1.0] * nz,) * 3)).cuda() if built == "split" else None
    dom = dict(u=f[0], v=f[1], w=f[2], nx=nx, ny=ny, coeffs=c)
    if table is not None:
        dom["split_table"] = table
    b = pw.Batch([dom], built, variant)
    pw.device_status()
    b.dt = pw.MODES[launched]
    b.run()
    assert pw.device_status() == (0 if built == launched else pw.PW_EINVAL)
