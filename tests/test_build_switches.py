"""The switches that device.cuh documents compile (no GPU needed)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("switch", ["MPA_F32X2=0", "MPA_F32X2_SCALE=0", "MPA_F32X2_POLY=1", "MPA_FMA_BFLY=0"])
def test_switch_compiles(tmp_path, switch):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-D" + switch,
                        "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1101_0086_gb300", "csrc"),
                        "-c", os.path.join(ROOT, "tests", "native", "switches_check.cu"), "-o", str(tmp_path / "s.o")],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
