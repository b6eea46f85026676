"""Host check of the fixed-point transforms: every radix, both directions, against long double.
An output's error: half a unit per rounded multiplication on its path and a quarter for each halving,
at most 6 units for the longest (radix 9 and 12)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_small_transforms_and_quotients(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "fx_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_1804_05087_gb300", "csrc"), os.path.join(ROOT, "tests", "host", "fx_check.cu"),
                    "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    rows = [line.split() for line in out if line]
    assert len(rows) == 14
    for r, s, err in rows:
        assert float(err) < 6.0, (r, s, err)
