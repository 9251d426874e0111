"""The fixed-point operator reads the geometric factors of its own element only,
at every order and in both thread layouts: the device header, compiled for the
host with loads that check their address (no GPU)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("CUDA headers not found")
    return inc


def test_factor_loads_stay_in_the_element(tmp_path):
    exe = str(tmp_path / "operator_reads")
    subprocess.run(["g++", "-std=c++20", "-O1", "-ffp-contract=off", "-pthread", "-I", cuda_include(),
                    os.path.join(HERE, "host", "operator_reads.cpp"), "-o", exe], check=True)
    rows = [list(map(int, r.split())) for r in
            subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) == 15 * 3
    assert [r for r in rows if r[3]] == []
