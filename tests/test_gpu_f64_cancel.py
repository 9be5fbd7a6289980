"""The FP64 forward path on near-uniform winds, whose products cancel to a
small part of their magnitudes: per point within 1e-13 of the sum of the
products' magnitudes of the oracle, as pw_advect documents."""
import numpy as np
import pytest

from paper_2107_13500_gb300 import synth
from tests.helpers import interior, to_device, to_numpy_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [1e-8, 1e-10, 1e-12])
@pytest.mark.parametrize("wind", [0.5, 0.1, 0.035])
def test_near_uniform_winds(oracle_lib, wind, eps):
    import torch
    from paper_2107_13500_gb300 import build, pw
    build.build()
    nx, ny, nz = 70, 37, 12
    dz = synth.dz_stretched(nz)
    f = [s * wind * (1.0 + 0.1 * eps * a) for s, a in zip((1.0, -0.7, 0.0), synth.fields_iid(nx, ny, nz, seed=3))]
    c = pw.make_coeffs(nz, 50.0, 50.0, dz).to_device()
    got = pw.advect(*(to_device(a, nx, torch.float64) for a in f), c, nx, ny, mode="f64")
    torch.cuda.synchronize()
    assert pw.device_status() == 0
    ref, ab = oracle_lib.advect(*f, oracle_lib.coeffs(nz, 50.0, 50.0, dz), nx, ny, want_abs=True, nthreads=8)
    for g, o, a in zip(got, ref, ab):
        g, o, a = (interior(t, nx, ny) for t in (to_numpy_f64(g, f[0].shape[2], nx), o, a))
        assert np.all(np.abs(g - o) <= 1e-13 * a), float(np.max(np.abs(g - o) / np.maximum(a, 1e-300)))


@pytest.mark.parametrize("ratio", [0.0, 1e-6, 1e-4])
@pytest.mark.parametrize("which", ["x", "y"])
@pytest.mark.parametrize("scale", [1e-5, 1e-6])
def test_unequal_horizontal_coefficients_with_fields_of_unequal_size(oracle_lib, ratio, which, scale):
    """Large products of the direction whose coefficient is small or 0 do not
    stand for the magnitude of the sum."""
    import torch
    from paper_2107_13500_gb300 import build, pw
    build.build()
    nx, ny, nz = 70, 37, 9
    dz = synth.dz_uniform(nz, 1e4)
    f = [a.copy() for a in synth.fields_iid(nx, ny, nz, seed=4)]
    f[0 if which == "y" else 1] *= scale
    f[2] *= 0.0
    c = pw.make_coeffs(nz, 50.0, 50.0, dz)
    if which == "y":
        c.tcy = c.tcx * ratio
    else:
        c.tcx = c.tcy * ratio
    co = {k: (np.array(v, copy=True) if isinstance(v, np.ndarray) else v) for k, v in c.as_dict().items()}
    got = pw.advect(*(to_device(a, nx, torch.float64) for a in f), c.to_device(), nx, ny, mode="f64")
    torch.cuda.synchronize()
    assert pw.device_status() == 0
    ref, ab = oracle_lib.advect(*f, co, nx, ny, want_abs=True, nthreads=8)
    for g, o, a in zip(got, ref, ab):
        g, o, a = (interior(t, nx, ny) for t in (to_numpy_f64(g, f[0].shape[2], nx), o, a))
        assert np.all(np.abs(g - o) <= 1e-13 * a), float(np.max(np.abs(g - o) / np.maximum(a, 1e-300)))
