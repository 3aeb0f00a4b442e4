"""The rotation layout's tabu ends, on the CPU (tests/host_tabu_ends.cu): marks,
ring and slots against a plain table of ends, past iteration 2^15 too."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_tabu_ends(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "host_tabu_ends")
    # the host code only: no device code is generated or run
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-o",
                    exe, os.path.join(HERE, "host_tabu_ends.cu")], check=True)
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0 and res.stdout.strip() == "ok", res.stdout
