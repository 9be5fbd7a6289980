"""The windows of the FP64 forward path: w and the vertical coefficients against
u and v from fine to coarse grids, fields far below one another, windows that
change from level to level, values below their window, subnormals, zeros. Per
point within 1e-13 of the sum of the products' magnitudes of the oracle, as
pw_advect documents (plus the oracle's own underflow); one launch, level slabs
and a batch give the same bits. And the calls that such winds make take no
longer than native FP64 evaluation would."""
import numpy as np
import pytest

from paper_2107_13500_gb300 import synth
from tests.helpers import interior, to_device, to_numpy_f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    from paper_2107_13500_gb300 import build, pw
    build.build()
    pw.load_library()
    return torch


def _fields(kind, nx, ny, nz):
    u, v, w = (f.copy() for f in synth.fields_iid(nx, ny, nz, seed=21))
    k = np.arange(nz)[:, None, None]
    j = np.arange(ny + 2)[None, :, None] / ny
    i = np.arange(u.shape[2])[None, None, :] / nx
    if kind == "w_tiny":
        w *= 1e-9
    elif kind == "v_tiny":
        v *= 1e-8
    elif kind == "u_tiny":
        u *= 2.0 ** -30
    elif kind == "v_zero":
        v *= 0.0
    elif kind == "u_zero":  # and the others small away from the middle, where a sum's last bits show its window
        g = np.exp(-0.5 * ((i - 0.5) ** 2 * nx * nx + (j - 0.5) ** 2 * ny * ny) / 64.0) + 0 * k
        u, v, w = u * 0.0, v * g, w * g
    elif kind == "only_w":
        u *= 0.0
        v *= 0.0
    elif kind == "growing":
        u, v, w = (f * 2.0 ** (1.5 * k) for f in (u, v, w))
    elif kind == "jumps":
        s = 2.0 ** (37.0 * ((k % 3) - 1) * (k % 2))
        u, v, w = u * s, v * s, w / s
    elif kind == "vortices":  # zero to rounding on lines of the grid
        u, v = 10 * np.sin(4 * np.pi * i) * np.cos(2 * np.pi * j) + 0 * k, -10 * np.cos(4 * np.pi * i) * np.sin(2 * np.pi * j) + 0 * k
        w = np.sin(4 * np.pi * i) * np.sin(2 * np.pi * j) * np.sin(np.pi * k / (nz - 1))
    elif kind == "bump":
        g = np.exp(-0.5 * ((i - 0.5) ** 2 * nx * nx + (j - 0.5) ** 2 * ny * ny) / 16.0) + 0 * k
        u, v, w = 10 * g, -7 * g, g
    elif kind == "subnormal":
        w *= 1e-310
        u[:, 5, 7:19] = 3e-310
    elif kind == "mixed":
        w[::2] = 0.0
        u[3:6] *= 1e-20
        v[9] *= 1e15
    return [np.ascontiguousarray(synth.fill_periodic_halo(np.ascontiguousarray(f), nx, ny)) for f in (u, v, w)]


KINDS = ["iid", "w_tiny", "v_tiny", "u_tiny", "u_zero", "v_zero", "only_w", "growing", "jumps", "vortices", "bump", "subnormal", "mixed"]


@pytest.mark.parametrize("dx,dy", [(50.0, 50.0), (1000.0, 1000.0), (2.0e4, 2.0e4), (1.0e5, 1.0e5), (1.0, 1.0), (1000.0, 10.0)])
@pytest.mark.parametrize("kind", KINDS)
def test_windows_against_the_oracle(gpu, oracle_lib, kind, dx, dy):
    from paper_2107_13500_gb300 import pw
    nx, ny, nz = 70, 39, 17
    dz = synth.dz_stretched(nz)
    rho, rhon = (None, None) if kind != "iid" else synth.density_exponential(dz)
    c = pw.make_coeffs(nz, dx, dy, dz, rho, rhon).to_device()
    f = _fields(kind, nx, ny, nz)
    dev = [to_device(a, nx, gpu.float64) for a in f]
    want = pw.advect(*dev, c, nx, ny, mode="f64")
    batch = pw.Batch([dict(u=dev[0], v=dev[1], w=dev[2], nx=nx, ny=ny, coeffs=c)], "f64", 0)
    batch.run()
    host = [pw.pinned_field(nx, ny, nz) for _ in range(3)]
    for h, a in zip(host, f):
        h[:, :, : nx + 2] = gpu.from_numpy(a[:, :, : nx + 2])
    slabs = [t.cuda() for t in pw.advect_host(*host, c, nx, ny, mode="f64", nchunks=nz)]
    gpu.cuda.synchronize()
    assert pw.device_status() == 0
    ref, ab = oracle_lib.advect(*f, oracle_lib.coeffs(nz, dx, dy, dz, rho, rhon), nx, ny, want_abs=True, nthreads=8)
    inside = (slice(None), slice(1, ny + 1), slice(1, nx + 1))
    for g, b, s, o, a in zip(want, batch.outputs()[0], slabs, ref, ab):
        assert gpu.equal(g[inside], b[inside]) and gpu.equal(g[inside], s[inside])
        g, o, a = (interior(t, nx, ny) for t in (to_numpy_f64(g, f[0].shape[2], nx), o, a))
        err = np.abs(g - o)
        assert np.all(err <= 1e-13 * a + 16 * 5e-324), (float(np.max(err / np.maximum(a, 1e-300))), np.argwhere(err > 1e-13 * a)[:4])


def test_no_wind_takes_longer_than_native_fp64(gpu):
    """Native FP64 evaluation takes 1.75 times the fixed-point form on i.i.d.
    winds over 50 m (1066 and 607 us at 512x512x64). Coarse grids, updrafts and
    winds that vanish somewhere stay below that."""
    from paper_2107_13500_gb300 import pw
    torch = gpu
    nx, ny, nz = 512, 256, 64
    dz = synth.dz_stretched(nz)
    gen = torch.Generator(device="cuda").manual_seed(1)
    x, y, z = (torch.arange(n, device="cuda", dtype=torch.float64) / n for n in (nx, ny, nz))

    def field(val):
        f = pw.empty_field(nx, ny, nz, torch.float64)
        f[:, 1:ny + 1, 1:nx + 1] = val
        return pw.fill_periodic_halo(f, nx, ny)

    def noise(a):
        return (torch.rand((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64) * 2 - 1) * a

    def micros(winds, dx):
        f = [field(t) for t in winds]
        c = pw.make_coeffs(nz, dx, dx, dz).to_device()
        out = tuple(pw.field_like(f[0]) for _ in range(3))
        best = []
        for _ in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            pw.advect(*f, c, nx, ny, mode="f64", out=out)
            b.record()
            b.synchronize()
            best.append(a.elapsed_time(b) * 1e3)
        return min(best)

    plain = micros([noise(10.0) for _ in range(3)], 50.0)
    sx, cx, sy, cy = (g(2 * np.pi * t) for t, g in ((x, torch.sin), (x, torch.cos), (y[:, None], torch.sin), (y[:, None], torch.cos)))
    zz = torch.cos(np.pi * z)[:, None, None]
    cases = {
        "iid, 400 m": ([noise(10.0) for _ in range(3)], 400.0),
        "iid, 4000 m": ([noise(10.0) for _ in range(3)], 4000.0),
        "updrafts": ([noise(5.0), noise(5.0), noise(60.0)], 200.0),
        "vortex": ([10 * sx * cy * zz, -10 * cx * sy * zz, torch.zeros((nz, ny, nx), device="cuda", dtype=torch.float64)], 50.0),
        "weak v and w": ([5.0 + noise(1e-8), noise(1e-8), noise(1e-8)], 50.0),
    }
    slow = {k: round(micros(*v) / plain, 2) for k, v in cases.items()}
    assert max(slow.values()) <= 1.75, slow
