"""The two forms of the FP32 forward path: mode "f32" leaves out the products
with level means, which are 0 there. Every other operation rounds alike, so on
finite values both forms give the same bits; an infinity or NaN reaches the
same outputs in both (0 times an infinity is NaN in the general form)."""
import numpy as np
import pytest

from paper_2107_13500_gb300 import synth
from tests.helpers import interior

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(133, 9, 11), (128, 8, 12), (37, 21, 2)])
@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("special", [None, np.inf, -np.inf, np.nan])
def test_f32_is_the_general_form_with_means_of_zero(shape, aligned, special):
    import torch
    from paper_2107_13500_gb300 import build, pw
    build.build()
    nx, ny, nz = shape
    dz = synth.dz_stretched(nz)
    c = pw.make_coeffs(nz, 50.0, 40.0, dz).to_device()
    a = [x.copy() for x in synth.fields_iid(nx, ny, nz, seed=4)]
    if special is not None:
        a[0][1, 3, 5] = special
        a[2][nz - 1, ny - 1, nx - 2] = special
    f = [pw.field_from_numpy(x, nx, torch.float32, aligned=aligned) for x in a]
    table = torch.from_numpy(pw.make_split_table(c, *([0.0] * nz,) * 3)).cuda()
    got = pw.advect(*f, c, nx, ny, mode="f32")
    want = pw.advect(*f, c, nx, ny, mode="split", split_table=table)
    doms = [dict(u=f[0], v=f[1], w=f[2], nx=nx, ny=ny, coeffs=c, split_table=t) for t in (table, None)]
    mixed, plain = pw.Batch(doms, "f32", 0), pw.Batch(doms[1:], "f32", 0)
    mixed.run()
    plain.run()
    torch.cuda.synchronize()
    assert pw.device_status() == 0
    assert special is None or not bool(torch.isfinite(want[0]).all())
    for g, w, m, p in zip(got, want, mixed.outputs()[1], plain.outputs()[0]):
        assert torch.equal(g.view(torch.int32), p.view(torch.int32))
        if special is None:
            assert torch.equal(g, w) and torch.equal(g, m)
        else:
            g, w, m = (interior(t.cpu().numpy(), nx, ny) for t in (g, w, m))
            fine = np.isfinite(w)
            assert np.array_equal(np.isfinite(g), fine) and np.array_equal(np.isfinite(m), fine)
            assert np.array_equal(g[fine], w[fine]) and np.array_equal(m[fine], w[fine])
