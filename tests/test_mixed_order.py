"""The two streams of the mixed factorisation, on the CPU: every pair of launches that touch the
same tile is ordered by the events between them, and every update is applied once, before its
tile is factored or solved.  The rule of which launch writes which tile is the library's own
(csrc/mixed_order.cuh); the program lays the launches and waits of factor_mixed on vector clocks,
for every number of tiles up to 14, bands up to 6 and both kinds of modes.  Without the corner
tiles ahead of the column's event it counts 7,856 unordered pairs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1708_02835_gb300", "csrc")


def test_every_tile_access_is_ordered(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "df_host", "check_mixed_order.cpp"),
                    "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120, check=True).stdout
    v = dict(kv.split("=") for kv in out.split())
    assert int(v["seen"]) > 100_000 and int(v["races"]) == 0 and int(v["wrong"]) == 0, out


def test_factor_mixed_follows_the_rule():
    """The order of the calls in factor_mixed that the model restates."""
    src = open(os.path.join(CSRC, "mixed.cu")).read()
    body = src[src.index("cudaError_t factor_mixed("):src.index("// out = L^-1 rhs with the inverted diagonal tiles")]
    marks = ["order::potrf_waits_for_column(tl.band)", "launch_panel64(", "cudaEventRecord(ev_diag, side)",
             "cudaStreamWaitEvent(side, ev_col, 0)", "launch_band_solve(", "cudaEventRecord(ev_panel, side)",
             "order::kBandBand", "launch_trsm_tc(", "order::kColumn", "cudaEventRecord(ev_col, s)",
             "order::kRest"]
    at = -1
    for m in marks:
        at = body.find(m, at + 1)
        assert at >= 0, m
