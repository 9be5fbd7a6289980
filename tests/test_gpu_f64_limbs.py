"""The FP64 forward path where its fixed-point form changes scale or gives way
to FP64 evaluation: winds far from one metre per second, levels of different
magnitude in one column, values too small for the window beside large ones,
infinities and NaN, zero fields, coefficients of any size and sign."""
import numpy as np
import pytest

from paper_2107_13500_gb300 import synth
from tests.helpers import compare_f64, interior, to_device, to_numpy_f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2107_13500_gb300 import build, pw
    build.build()
    pw.load_library()
    return torch


def _advect(gpu, fields, c, nx, ny):
    from paper_2107_13500_gb300 import pw
    dev = [to_device(f, nx, gpu.float64) for f in fields]
    out = pw.advect(*dev, c, nx, ny, mode="f64")
    gpu.cuda.synchronize()
    assert pw.device_status() == 0
    return [to_numpy_f64(t, fields[0].shape[2], nx) for t in out]


def _check(gpu, oracle_lib, fields, nx, ny, nz, dx=50.0, dy=50.0, dz=None, rho=None, rhon=None, edit=None):
    """Against the oracle at the path's own tolerance (1e-13 of the strict scale and normwise); where the oracle
    overflows, so does the path."""
    from paper_2107_13500_gb300 import pw
    dz = synth.dz_stretched(nz) if dz is None else dz
    c = pw.make_coeffs(nz, dx, dy, dz, rho, rhon)
    if edit:
        edit(c)
    co = {k: (np.array(v, copy=True) if isinstance(v, np.ndarray) else v) for k, v in c.as_dict().items()}
    ref, ab = oracle_lib.advect(*fields, co, nx, ny, want_abs=True, nthreads=8)
    got = _advect(gpu, fields, c.to_device(), nx, ny)
    for g, o, a in zip(got, ref, ab):
        over = ~np.isfinite(o)
        assert np.array_equal(over, ~np.isfinite(g))
        g[over] = o[over] = a[over] = 0.0
    compare_f64(got, ref, ab, nx, ny)
    return got, ref


@pytest.mark.parametrize("scale", [2.0 ** -300, 2.0 ** -40, 1e-6, 1e-3, 0.05, 128.0, 1e3, 2.0 ** 40, 2.0 ** 290])
def test_scales_of_the_winds(gpu, oracle_lib, scale):
    nx, ny, nz = 53, 37, 14
    _check(gpu, oracle_lib, [f * scale for f in synth.fields_iid(nx, ny, nz, seed=5)], nx, ny, nz)


@pytest.mark.parametrize("case", ["levels", "fields", "spike", "tiny", "wide", "zero_w", "zero_u", "zero_levels"])
def test_magnitudes_mixed_in_a_column(gpu, oracle_lib, case):
    """Steps between levels of different scale, levels refused for one value,
    fields of very different magnitude, and fields or levels of zeros."""
    nx, ny, nz = 70, 40, 20
    u, v, w = (f.copy() for f in synth.fields_iid(nx, ny, nz, seed=6))
    if case == "levels":
        for k in range(nz):
            for f in (u, v, w):
                f[k] *= 2.0 ** (3 * (k % 11) - 12)
    elif case == "fields":
        u *= 100.0
        w *= 1e-9
    elif case == "spike":
        u[7, 20, 30] = 1e15
        v[11, 5, 66] = -3e200
    elif case == "tiny":
        u[5, 10, 10], v[9, 33, 64], w[14, 17, 33] = 1e-25, 1e-300, 5e-324
    elif case == "wide":
        r = synth.uniform(7, 0, u.size, -14.0, 0.0).reshape(u.shape)
        u, v, w = (synth.fill_periodic_halo(f * 10.0 ** r, nx, ny) for f in (u, v, w))
    elif case == "zero_w":
        w[:] = 0.0
    elif case == "zero_u":
        u[:] = 0.0
        v[:, 12:20] = 0.0
    else:
        for f in (u, v, w):
            f[3:6] = 0.0
            f[12] = -0.0
    _check(gpu, oracle_lib, (u, v, w), nx, ny, nz)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_infinities_and_nan_reach_the_points_that_read_them(gpu, oracle_lib, value):
    """The finite outputs are those of the oracle, the others lie where the
    oracle's lie."""
    from paper_2107_13500_gb300 import pw
    nx, ny, nz = 40, 20, 9
    u, v, w = (f.copy() for f in synth.fields_iid(nx, ny, nz, seed=8))
    u[4, 10, 12] = value
    w[6, 3, 34] = value
    dz = synth.dz_stretched(nz)
    c = pw.make_coeffs(nz, 50.0, 50.0, dz)
    ref = oracle_lib.advect(u, v, w, oracle_lib.coeffs(nz, 50.0, 50.0, dz), nx, ny)
    got = _advect(gpu, (u, v, w), c.to_device(), nx, ny)
    for g, o in zip(got, ref):
        g, o = interior(g, nx, ny), interior(o, nx, ny)
        fine = np.isfinite(o)
        assert np.array_equal(np.isfinite(g), fine) and not fine.all()
        assert np.max(np.abs(g[fine] - o[fine])) <= 1e-13 * np.max(np.abs(o[fine]))


@pytest.mark.parametrize("case", ["coarse", "fine", "anisotropic", "negative", "huge", "zero_x", "one_huge_level"])
def test_coefficients_of_any_size(gpu, oracle_lib, case):
    """Horizontal over vertical spacings from 1e-4 to 1e4 (the window of w
    moves with the largest ratio), and coefficients that no limb number
    holds."""
    nx, ny, nz = 37, 21, 12
    kw, edit = {}, None
    if case == "coarse":
        kw = dict(dx=3000.0, dy=3000.0, dz=synth.dz_uniform(nz, 0.3))
    elif case == "fine":
        kw = dict(dx=1.0, dy=1.0, dz=synth.dz_uniform(nz, 1e4))
    elif case == "anisotropic":
        kw = dict(dx=1e4, dy=1.0)
    elif case == "negative":
        def edit(c):
            c.tcy = -c.tcy
            c.tz4[1] *= -1.0
            c.tz4[2, ::2] *= -0.5
    elif case == "huge":
        kw = dict(dx=1e-200, dy=1e-200)
    elif case == "zero_x":
        def edit(c):
            c.tcx = 0.0
    else:
        def edit(c):
            c.tz4[0, 5] = 1e30
    _check(gpu, oracle_lib, synth.fields_iid(nx, ny, nz, seed=9), nx, ny, nz, edit=edit, **kw)


def test_launch_forms_agree_on_mixed_scales(gpu):
    """Which steps are limb steps depends on the data only: one launch, level
    slabs and a batch give the same bits on levels of every scale."""
    import torch
    from paper_2107_13500_gb300 import pw
    nx, ny, nz = 90, 50, 33
    fields = [f.copy() for f in synth.fields_iid(nx, ny, nz, seed=11)]
    for k in range(nz):
        for f in fields:
            f[k] *= 2.0 ** (5 * (k % 7) - 15)
    fields[2][9, 30, 40] = 1e-30
    c = pw.make_coeffs(nz, 50.0, 50.0, synth.dz_stretched(nz)).to_device()
    dev = [to_device(f, nx, torch.float64) for f in fields]
    want = pw.advect(*dev, c, nx, ny, mode="f64")
    outs = []
    for v in range(pw.variant_count("f64")):
        b = pw.Batch([dict(u=dev[0], v=dev[1], w=dev[2], nx=nx, ny=ny, coeffs=c)], "f64", v)
        b.run()
        outs.append(b.outputs()[0])
    host = [pw.pinned_field(nx, ny, nz) for _ in range(3)]
    for h, a in zip(host, fields):
        h[:, :, : nx + 2] = torch.from_numpy(a[:, :, : nx + 2])
    for n in (4, 33):
        outs.append([t.cuda() for t in pw.advect_host(*host, c, nx, ny, mode="f64", nchunks=n)])
    torch.cuda.synchronize()
    assert pw.device_status() == 0
    inside = (slice(None), slice(1, ny + 1), slice(1, nx + 1))
    for o in outs:
        for a, b in zip(o, want):
            assert torch.equal(a[inside], b[inside])
