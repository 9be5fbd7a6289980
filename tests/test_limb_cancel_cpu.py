"""Sums of csrc/pw_limb.cuh whose large products cancel (near-uniform winds),
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
