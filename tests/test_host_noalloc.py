"""qap_batch_search_noalloc allocates nothing on the host either, on the CPU: the
source of the call names no container or allocation, and its planning
(tests/host_noalloc_plans.cu) makes none."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
API = os.path.join(HERE, "..", "paper_2307_11248_gb300", "csrc", "qap_api.cu")


def test_the_call_names_no_allocation():
    with open(API) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    start = text.index('extern "C" qap_status qap_batch_search_noalloc(')
    body = text[start:text.index("\n}\n", start)]
    found = re.findall(r"std::(?:vector|string|unique_ptr|make_\w+)|\bnew\b|\bmalloc\b|cudaMalloc\w*|\bgrow\(",
                       body)
    assert not found, found


def test_planning_allocates_nothing(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "host_noalloc_plans")
    # the host code only: no device code is generated or run
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-o",
                    exe, os.path.join(HERE, "host_noalloc_plans.cu")], check=True)
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0 and res.stdout.strip() == "ok", res.stdout
