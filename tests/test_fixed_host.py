"""Host check of the fixed-point arithmetic behind the FP64 kernels
(csrc/lbm_fixed.cuh): built with nvcc for the CPU and run here; see
tests/host/pow_check.cu."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build(tmp_path, name):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / name)
    src = os.path.join(ROOT, "tests", "host", name + ".cu")
    inc = os.path.join(ROOT, "paper_2011_15073_gb300", "csrc")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", inc, src, "-o", exe], check=True, timeout=300)
    return exe


def test_power_is_within_three_quarters_of_an_ulp(tmp_path):
    # half an ulp of rounding; ln 2 (|e| 2^-56.4 + 2^-56) / 2^-52 < 0.2 from
    # the logarithm and the product for |e| < 2; 0.03 from the exponential
    r = subprocess.run([build(tmp_path, "pow_check")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("OK"), r.stdout[-2000:]
    law, every = (float(r.stdout.split()[i]) for i in (2, 4))
    assert law < 0.75 and every < 0.75
