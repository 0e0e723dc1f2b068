"""The 96-bit fixed-point arithmetic of the float64 sweeps, checked on the host.

The functions compile as host code too, so nvcc builds a small host program
that compares them with 128-bit integer arithmetic: sums, shifts, products,
conversions from and to float64 (exact in the range the scale covers), and the
element factors' encoding.
"""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_matches_wide_integers(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "fixed_point"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2301_07457_gb300", "csrc"),
                    "-o", str(exe), os.path.join(ROOT, "tests", "native", "fixed_point.cu")],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("ok ")
