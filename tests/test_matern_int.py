"""The integer Matern evaluation (csrc/matern_int.cuh) on the CPU, against long double.

Its intermediates keep 57 bits or more and it rounds to double once: half an ulp (1.11e-16)
and a few units of 2^-57 (7e-18) each from the root, the exponential and the factor, so the
closed forms must stay within 1.5e-16 relative, plus x 2^-60 from e^-x (x is formed with three
truncations at 2^-62; an FP64 x = r / theta2 alone carries x 2^-53).  A general nu adds its polynomials' rounding to
double (12 coefficients, each half an ulp of the largest: below 2.5e-16 together).  Squared
distances of 0, subnormal or not finite and far too large ones are left to the FP64 evaluation."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1708_02835_gb300", "csrc")


def test_integer_matern_on_the_host(tmp_path):
    if np.finfo(np.longdouble).eps >= 2.0 ** -60 or not shutil.which("g++") or not shutil.which("gcc"):
        pytest.skip("needs gcc and a long double of more than 60 bits")
    obj, exe = str(tmp_path / "host.o"), str(tmp_path / "check")
    subprocess.run(["gcc", "-O2", "-std=gnu11", "-c", os.path.join(CSRC, "matern_host.c"), "-o", obj], check=True)
    shutil.copy(os.path.join(CSRC, "matern_int.cuh"), str(tmp_path / "matern_int.cuh"))
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", str(tmp_path), "-I", CSRC,
                    os.path.join(ROOT, "tests", "df_host", "check_int.cpp"), obj, "-lm", "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300, check=True).stdout
    print(out)
    v = dict(kv.split("=") for kv in out.split())
    assert int(v["taken"]) > 2_000_000 and int(v["edge"]) == 0
    for k in ("half", "threehalf", "fivehalf"):
        assert float(v[k]) <= 1.5e-16, v
    assert float(v["general"]) <= 4e-16, v
