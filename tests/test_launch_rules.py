"""Launch rules of the library (launch.h) compiled as host code by nvcc and
checked without a GPU: which grids count as filling the device's SMs, and which
launches start while the kernel before them ends.  With a GPU: a launch that the
runtime refuses, whose error the launcher returns and clears."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _build(tmp_path, name):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / name)
    src = os.path.join(ROOT, "tests", "native", name + ".cu")
    inc = os.path.join(ROOT, "paper_1101_0086_gb300", "csrc")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-I", inc, src, "-o", exe],
                   check=True, capture_output=True, timeout=600)
    return exe


def test_launch_rules(tmp_path):
    r = subprocess.run([_build(tmp_path, "launch_rules_check")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.gpu
def test_refused_launch_is_returned_and_cleared(tmp_path):
    r = subprocess.run([_build(tmp_path, "refused_launch_check")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
