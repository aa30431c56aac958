"""The second streams of a factorisation on the way out, against a fake CUDA runtime on the CPU: work
that an early return leaves on one is waited for by the call's stream (record, wait) before the
stream is released, by the host if that fails, and not a second time after an orderly end."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.join(ROOT, "tests", "df_host")
CSRC = os.path.join(ROOT, "paper_1708_02835_gb300", "csrc")


def test_side_stream_is_joined_on_every_way_out(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    shutil.copy(os.path.join(HERE, "fake_cuda_runtime.h"), str(tmp_path / "cuda_runtime.h"))
    shutil.copy(os.path.join(CSRC, "side_stream.cuh"), str(tmp_path / "side_stream.cuh"))
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", str(tmp_path), os.path.join(HERE, "check_side_stream.cpp"), "-o", exe],
                   check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60, check=True).stdout
    v = dict(line.split("=") for line in out.split("\n") if line)
    assert v == {"early": "rwse", "joined": "rw|se", "fail_r": "ry!", "fail_w": "rwy!", "none": ""}


@pytest.mark.parametrize("name,owner", [("chol64.cu", "fork.create(s, false)"), ("mixed.cu", "chain.create(s, true)")])
def test_every_second_stream_is_one(name, owner):
    """No driver makes a stream without it."""
    src = open(os.path.join(CSRC, name)).read()
    assert owner in src and "cudaStreamCreate" not in src
