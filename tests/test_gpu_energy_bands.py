"""The energy budget at the edges of its work split (row bands of a cluster,
columns of a CTA, groups of levels in the totals) and on float values that the
integer widening leaves to the hardware, against the oracle's compensated sums."""
import numpy as np
import pytest

from paper_2107_13500_gb300 import synth
from tests.helpers import to_numpy_f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2107_13500_gb300 import build, pw
    build.build()
    pw.load_library()
    return torch


@pytest.mark.parametrize("wind,tend", [("float64", "float64"), ("float64", "float32"), ("float32", "float32")])
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 2), (257, 7, 33), (256, 9, 32), (40, 33, 65), (600, 64, 3)])
def test_budget_bands_against_oracle(gpu, oracle_lib, wind, tend, shape):
    """Tolerance: a thread adds at most ceil(rows of a band) * ceil(nx / 256)
    products, and the trees, CTAs and levels at most 5 + 8 + 8 + nz more sums:
    under 200 roundings of 2^-53 of the sum of magnitudes here; 1e-13 is 900."""
    from paper_2107_13500_gb300 import pw
    torch = gpu
    nx, ny, nz = shape
    gen = torch.Generator(device="cuda").manual_seed(nx + ny)

    def fields(name):
        dt = getattr(torch, name)
        out = []
        for _ in range(3):
            f = pw.empty_field(nx, ny, nz, dt)
            f.copy_(torch.rand(f.shape, generator=gen, device="cuda", dtype=torch.float64) * 20 - 10)
            if name == "float32":
                f[:, 1::3, 1::5] = 1e-41  # a subnormal float
            out.append(f)
        return out

    w, s = fields(wind), fields(tend)
    dz = synth.dz_stretched(nz)
    wu_h, ww_h = pw.make_energy_weights(nz, dz)
    tot, level = pw.energy_budget(*w, *s, nx, ny, torch.from_numpy(wu_h).cuda(), torch.from_numpy(ww_h).cuda())
    sy = synth.row_stride(nx, 8)
    wn = [to_numpy_f64(t.double(), sy, nx) for t in w]
    sn = [to_numpy_f64(t.double(), sy, nx) for t in s]
    ref = oracle_lib.energy_budget(*wn, *sn, wu_h, ww_h, nx, ny)
    tot, level = tot.cpu().numpy(), level.cpu().numpy()
    for n in range(3):
        assert abs(tot[n] - ref[n]) <= 1e-13 * ref[3 + n]
        assert abs(tot[3 + n] - ref[3 + n]) <= 1e-13 * ref[3 + n]
        p = wn[n][:, 1:ny + 1, 1:nx + 1] * sn[n][:, 1:ny + 1, 1:nx + 1]
        scale = np.abs(p).sum(axis=(1, 2))
        assert np.all(np.abs(level[:, n] - p.sum(axis=(1, 2))) <= 1e-13 * scale)
        assert np.all(np.abs(level[:, 3 + n] - scale) <= 1e-13 * scale)
    again, _ = pw.energy_budget(*w, *s, nx, ny, torch.from_numpy(wu_h).cuda(), torch.from_numpy(ww_h).cuda())
    assert np.array_equal(again.cpu().numpy(), tot)
    w[0][0, 1, 1] = float("inf")
    s[0][0, 1, 1] = 1.0
    tot, _ = pw.energy_budget(*w, *s, nx, ny, torch.ones(nz, dtype=torch.float64, device="cuda"),
                              torch.ones(nz, dtype=torch.float64, device="cuda"))
    assert np.isinf(tot.cpu().numpy()[[0, 3]]).all() and np.isfinite(tot.cpu().numpy()[[1, 2, 4, 5]]).all()
