"""Values below their window and changes of window in csrc/pw_limb.cuh, cut
towards zero to the unit exactly; and sums whose large products cancel (near-uniform winds),
against exact integers: the result keeps its bits below one unit of the upper
sum. Bound: one rounding of the result (half a unit in its last place) plus
what the products' dropped limbs come to, 2^-24 of the 2^28 units that the
products' magnitudes reach: 2^-52 of the sum of |q||a + b|."""
import ctypes
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2107_13500_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    so = str(tmp_path_factory.mktemp("limb") / "limb_host.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", build.CSRC,
                    os.path.join(HERE, "limb_host.cpp"), "-o", so], check=True, capture_output=True)
    return ctypes.CDLL(so)


def _ints(p, bits=140):
    """Every double times 2^bits, as Python integers (exact)."""
    return [int(math.ldexp(float(x), bits)) for x in p]


def _ulp(exact, bits):
    """A unit in the last place of the double nearest to exact * 2^-bits, in units of 2^-bits."""
    return 0 if exact == 0 else 2.0 ** (abs(exact).bit_length() - 53)


@pytest.mark.parametrize("eps", [1e-6, 1e-8, 1e-9, 1e-10, 1e-11, 1e-12, 0.0])
@pytest.mark.parametrize("wind", [100.0, 30.0, 5.0, 0.5, 0.1, 0.035])
def test_near_uniform_winds_keep_their_tendency(lib, wind, eps):
    n, E = 400, 7
    r = np.random.default_rng(int(wind * 1000))
    p = wind * (1.0 + eps * r.uniform(-1, 1, (n, 9)))
    p[:, 5:] *= -0.7
    out, ok, enough = np.zeros(n), np.zeros(n, np.uint8), np.zeros(n, np.uint8)
    c = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    lib.limb_su_sums(n, E, c(np.ascontiguousarray(p)), c(out), c(ok), c(enough))
    assert ok.all() and enough.all()
    for row, got in zip(p, out):
        uw, uc, ue, us, un, vs, vse, vc, ve = _ints(row)
        exact = uw * (uw + uc) - ue * (uc + ue) + us * (vs + vse) - un * (vc + ve)
        a = abs(uw * (uw + uc)) + abs(ue * (uc + ue)) + abs(us * (vs + vse)) + abs(un * (vc + ve))
        err = abs(int(math.ldexp(float(got), 280)) - exact)
        assert err <= 0.5 * _ulp(exact, 280) + 2.0 ** -52 * a, (wind, eps, err / a)


@pytest.mark.parametrize("ratio", [0.0, 1e-6, 1e-4, 0.25, 1.0 - 2.0 ** -53])
@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("u_scale", [1.0, 1e-4, 2.0 ** -16, 2.0 ** -19])
def test_products_with_small_coefficients_do_not_settle_a_sum(lib, ratio, swap, u_scale):
    """tcx != tcy: large products of the direction whose coefficient is small or
    0 say nothing about the sum. What the rule settles is within the bound
    above, with the coefficients in the magnitudes."""
    n, E = 1000, 7
    r = np.random.default_rng(5)
    p = r.uniform(5.0, 15.0, (n, 9)) * r.choice([-1.0, 1.0], (n, 9))
    p[:, :5] *= u_scale / 10.0
    rx, ry = (ratio, 1.0) if swap else (1.0, ratio)
    out, ok, enough = np.zeros(n), np.zeros(n, np.uint8), np.zeros(n, np.uint8)
    c = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    lib.limb_su_joined(n, E, ctypes.c_double(rx), ctypes.c_double(ry), c(np.ascontiguousarray(p)), c(out), c(ok), c(enough))
    assert ok.all()
    cx, cy = _ints((rx, ry), 80)
    for row, got, settled in zip(p, out, enough):
        uw, uc, ue, us, un, vs, vse, vc, ve = _ints(row)
        exact = cx * (uw * (uw + uc) - ue * (uc + ue)) + cy * (us * (vs + vse) - un * (vc + ve))
        a = cx * (abs(uw * (uw + uc)) + abs(ue * (uc + ue))) + cy * (abs(us * (vs + vse)) + abs(un * (vc + ve)))
        err = abs(int(math.ldexp(float(got), 360)) - exact)
        if settled:
            assert err <= 0.5 * _ulp(exact, 360) + 2.0 ** -52 * a, err / a
    if u_scale == 1.0 and ratio > 0.1:
        assert enough.mean() > 0.99


def _value(limbs):
    return (int(limbs[0]) << 58) + (int(limbs[1]) << 29) + int(limbs[2])


def _cut(x, bits):
    """Integer x * 2^-bits towards zero (bits may be negative) and whether it lost anything."""
    if bits <= 0:
        return x << -bits, False
    q = abs(x) >> bits
    return (q if x >= 0 else -q), (q << bits) != abs(x)


@pytest.mark.parametrize("up", [0, 1, 3, 6, 26, 31, 32, 33, 58, 64, 77, 87, 95, -1, -4, -29, -32, -60, -64, -80])
def test_cut_values_and_changes_of_window(lib, up):
    r = np.random.default_rng(up + 200)
    E = 7
    top = min(E, E + up)  # every value fits both windows
    x = np.ldexp(r.uniform(0.5, 1.0, 4000), top - r.integers(0, 130, 4000)) * r.choice([-1.0, 1.0], 4000)
    x[::7] = np.ldexp(np.round(np.ldexp(x[::7], 20)), -20)  # short significands, many of them 0
    x[::11] = np.sign(x[::11]) * np.ldexp(1.0, top - 1 - r.integers(0, 100, x[::11].size))
    x[:6] = 0.0, -0.0, 5e-324, -5e-324, 1e-310, -2.0 ** -1022
    a, b = np.zeros((x.size, 4), np.int32), np.zeros((x.size, 4), np.int32)
    c = lambda t: t.ctypes.data_as(ctypes.c_void_p)
    lib.limb_cut_and_shift(x.size, E, up, c(x), c(a), c(b))
    for v, p, q in zip(x, a, b):
        m, e = math.frexp(float(v))
        want, lost = _cut(int(m * 2.0 ** 53), 53 - e + (E - 86))
        assert _value(p) == want and bool(p[3]) == lost, v
        want, lost = _cut(want, up)
        assert _value(q) == want and bool(q[3]) == lost, (v, up)
        for t in (p, q):
            assert 0 <= t[1] < 2 ** 29 and 0 <= t[2] < 2 ** 29 and abs(int(t[0])) <= 2 ** 28


def test_coefficients_below_their_window(lib):
    r = np.random.default_rng(1)
    x = np.ldexp(r.uniform(0.5, 1.0, 4000), 2 - r.integers(0, 130, 4000)) * r.choice([-1.0, 1.0], 4000)
    out = np.zeros((x.size, 4), np.int32)
    lib.limb_cut_coef(x.size, x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p))
    for v, p in zip(x, out):
        m, e = math.frexp(float(v))
        want, lost = _cut(int(m * 2.0 ** 53), 53 - e - 87)
        assert _value(p) == want and bool(p[3]) == lost, v


@pytest.mark.parametrize("E", [7, -200, 300])
def test_values_far_below_their_window(lib, E):
    r = np.random.default_rng(2)
    x = np.ldexp(r.uniform(0.5, 1.0, 6000), E - 32 - r.integers(0, 90, 6000)) * r.choice([-1.0, 1.0], 6000)
    x[::5] = np.sign(x[::5]) * np.ldexp(1.0, E - 33 - r.integers(0, 60, x[::5].size))
    x[:6] = 0.0, -0.0, 5e-324, -5e-324, 1e-310, -2.0 ** -1022
    out = np.zeros((x.size, 4), np.int32)
    lib.limb_cut_low(x.size, E, x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p))
    for v, p in zip(x, out):
        m, e = math.frexp(float(v))
        want, lost = _cut(int(m * 2.0 ** 53), 53 - e + (E - 86))
        assert _value(p) == want and bool(p[3]) == lost, v
        assert 0 <= p[1] < 2 ** 29 and 0 <= p[2] < 2 ** 29
