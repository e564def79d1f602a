"""Host check of the fixed-point collision of the FP64 storage
(csrc/lbm_collide_fixed.cuh): built with nvcc for the CPU and run here; see
tests/host/fixed_check.cu."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_collision_is_no_further_off_than_fp64(tmp_path):
    """Largest and RMS error against long double at most the plain FP64
    form's, over flows, laws, drags and parameters; values out of range
    refused with nothing changed."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "fixed_check")
    src = os.path.join(ROOT, "tests", "host", "fixed_check.cu")
    inc = os.path.join(ROOT, "paper_2011_15073_gb300", "csrc")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", inc, src, "-o", exe], check=True, timeout=300)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("OK"), r.stdout[-2000:]
