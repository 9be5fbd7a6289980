"""The fused forward-Euler step (one update launch with its halo, one transposed
launch, the adjoint accumulated in place) against the separate torch and halo
operations it stands for: equal bit for bit, forward and backward."""
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


def _separate_step(autograd, x, c, nx, ny, dt, mode):
    s = autograd.advect(*x, c, nx, ny, mode)
    return tuple(autograd.FillPeriodicHalo.apply(f + dt * t, nx, ny) for f, t in zip(x, s))


@pytest.mark.parametrize("mode", ["f64", "paired", "f32"])
@pytest.mark.parametrize("shape", [(1, 1, 3), (1, 9, 2), (9, 1, 4), (2, 2, 5), (37, 13, 6), (129, 17, 3), (254, 6, 2)])
@pytest.mark.parametrize("aligned", [True, False])
def test_euler_step_equals_separate_operations(gpu, mode, shape, aligned):
    """Single columns and rows (the halo cells of both sides fold into one
    cell), widths around the block of columns, heights around the block of
    rows; values in the row padding pass through."""
    from paper_2107_13500_gb300 import autograd, pw
    torch = gpu
    nx, ny, nz = shape
    tdt = torch.float32 if mode == "f32" else torch.float64
    c = pw.make_coeffs(nz, 50.0, 50.0, synth.dz_stretched(nz)).to_device()
    gen = torch.Generator(device="cuda").manual_seed(7)

    def field():
        f = pw.empty_field(nx, ny, nz, tdt, aligned=aligned)
        return f.copy_(torch.rand(f.shape, generator=gen, device="cuda", dtype=tdt) * 20 - 10)

    x = [field() for _ in range(3)]
    for f in x:
        pw.fill_periodic_halo(f, nx, ny)
    cot = [field() for _ in range(3)]
    got, want = [], []
    for step, res in ((lambda a: autograd.euler_step(*a, c, nx, ny, 0.3, mode), got),
                      (lambda a: _separate_step(autograd, a, c, nx, ny, 0.3, mode), want)):
        a = [t.detach().requires_grad_() for t in x]
        y = step(a)
        res += [t.detach() for t in y]
        res += list(torch.autograd.grad(y, a, [t.expand_as(t) for t in cot]))
    torch.cuda.synchronize()
    assert pw.device_status() == 0
    for g, w in zip(got, want):
        assert torch.equal(g, w)


def test_euler_step_unused_outputs_and_broadcast_gradients(gpu):
    """Gradients that autograd materialises (an output nobody used) or expands
    (a sum) arrive in other strides than the fields'."""
    from paper_2107_13500_gb300 import autograd, pw
    torch = gpu
    nx, ny, nz = 21, 10, 4
    c = pw.make_coeffs(nz, 50.0, 40.0, synth.dz_stretched(nz)).to_device()
    x = [pw.field_from_numpy(f, nx) for f in synth.fields_iid(nx, ny, nz, seed=3)]
    grads = []
    for step in (autograd.euler_step, lambda u, v, w, *a: _separate_step(autograd, (u, v, w), *a)):
        a = [t.detach().requires_grad_() for t in x]
        y = step(*a, c, nx, ny, 0.25, "f64")
        grads.append(torch.autograd.grad(y[0].sum(), a))
    for g, w in zip(*grads):
        assert torch.equal(g, w)


def test_euler_periodic_rejects_aliases(gpu):
    from paper_2107_13500_gb300 import pw
    import ctypes
    nx, ny, nz = 12, 6, 3
    f = [pw.empty_field(nx, ny, nz) for _ in range(8)]
    d = pw.dims_of(f[0], nx, ny)
    p = [ctypes.c_void_p(t.data_ptr()) for t in f]
    lib = pw.load_library()

    def call(ins, outs, width=f[0].shape[2]):
        return lib.pw_euler_periodic(pw.PW_F64, *ins, 0.1, ctypes.byref(d), width, *outs, pw._stream_handle())

    assert call(p[:6], (p[0], p[6], p[7])) == pw.PW_EALIAS
    assert call(p[:6], (p[6], p[6], p[7])) == pw.PW_EALIAS
    assert call(p[:6], (p[6], None, p[7])) == pw.PW_ENULL
    assert call(p[:6], (p[6], p[7], p[7]), nx + 1) == pw.PW_EINVAL
