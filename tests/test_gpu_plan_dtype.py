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


@pytest.mark.parametrize("means", [False, True])
@pytest.mark.parametrize("form", ["advect", "batch"])
def test_a_table_with_means_given_as_pw_f32_is_reported(monkeypatch, form, means):
    """The C entry points' PW_F32 leaves the mean terms out (the Python ones take
    such a table through PW_F32_SPLIT, which is turned off here)."""
    import torch
    from paper_2107_13500_gb300 import build, pw
    build.build()
    nx, ny, nz = 140, 9, 7
    c = pw.make_coeffs(nz, 50.0, 50.0, synth.dz_stretched(nz)).to_device()
    f = [pw.field_from_numpy(a, nx, torch.float32) for a in synth.fields_iid(nx, ny, nz, seed=2)]
    table = torch.from_numpy(pw.make_split_table(c, *([0.5 if means else 0.0] * nz,) * 3)).cuda()
    monkeypatch.setattr(pw, "_arithmetic", lambda mode, split_table: pw.MODES[mode])
    pw.device_status()
    if form == "advect":
        pw.advect(*f, c, nx, ny, mode="f32", split_table=table)
    else:
        b = pw.Batch([dict(u=f[0], v=f[1], w=f[2], nx=nx, ny=ny, coeffs=c, split_table=table)], "f32", 0)
        b.run()
    assert pw.device_status() == (pw.PW_EINVAL if means else 0)
