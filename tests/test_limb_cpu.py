"""The fixed-point arithmetic of the FP64 forward path (csrc/pw_limb.cuh)
against exact integer arithmetic: splits over and around the whole window, and
700,000 sums as a stencil point forms them, each within half a unit in the
last place plus two units of 2^-53 of the sum of its products' magnitudes
(tests/limb_check.cpp, compiled with the host compiler)."""
import os
import shutil
import subprocess

import pytest

from paper_2107_13500_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_limb_arithmetic_against_exact_integers(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "limb_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", build.CSRC,
                    os.path.join(HERE, "limb_check.cpp"), "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    words = out.stdout.split()
    cases, bad, small = (int(words[k]) for k in (1, 3, 5))
    assert cases > 1_000_000 and bad == 0 and small < cases // 10
