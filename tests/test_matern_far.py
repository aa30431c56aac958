"""General smoothness at large distances, on the CPU: the integer evaluation covers x = r / theta2 up
to the polynomials' end at 1,280 (beyond 640 too, where the alternative is the direct recurrence of
about 1,100 FP64 operations an entry), within the bar of test_matern_int.py, and 0 below the
smallest normal double."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1708_02835_gb300", "csrc")


def test_general_nu_far_distances_on_the_host(tmp_path):
    if np.finfo(np.longdouble).eps >= 2.0 ** -60 or not shutil.which("g++") or not shutil.which("gcc"):
        pytest.skip("needs gcc and a long double of more than 60 bits")
    obj, exe = str(tmp_path / "host.o"), str(tmp_path / "check")
    subprocess.run(["gcc", "-O2", "-std=gnu11", "-c", os.path.join(CSRC, "matern_host.c"), "-o", obj], check=True)
    shutil.copy(os.path.join(CSRC, "matern_int.cuh"), str(tmp_path / "matern_int.cuh"))
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", str(tmp_path), "-I", CSRC,
                    os.path.join(ROOT, "tests", "df_host", "check_int_far.cpp"), obj, "-lm", "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60, check=True).stdout
    v = dict(kv.split("=") for kv in out.split())
    assert int(v["taken"]) > 2000 and int(v["left"]) == 0 and int(v["wrong_far"]) == 0, out
    assert float(v["worst"]) <= 4e-16, out
