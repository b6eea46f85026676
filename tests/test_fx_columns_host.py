"""Host check of the fixed-point column arithmetic of the forward Chebyshev transform at the limits of its
scale. Error of a coefficient relative to the column's sum of moduli S: the scale leaves S 2^sh at least
2^57 (16 bits of S or 17 of a pair, rounded up, are scaled to 62 or 59), so each of the up to 258 values'
roundings (half a unit), the halving of the end points, the dropped low products (129 quarters) and the
constants' 2^-57 stay below 258 units in all: 258 * 2^-57 = 1.8e-15; the long double sum adds 258 * 2^-64."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_forward_columns(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "cheb_fx_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_1804_05087_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "cheb_fx_check.cu"), "-o", exe], check=True)
    rows = [line.split() for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
            if line]
    assert [int(r[0]) for r in rows][0] == 5 and int(rows[-1][0]) == 257
    for ny, err in rows:
        assert float(err) < 2e-15, (ny, err)


def test_transforms_at_the_kernels_bound(tmp_path):
    """Error of an output, in units: the 6 of the transforms below 2^55 (test_fx_host.py); the long double
    reference's 64 bits at 2^60.5, a sixteenth per term and 12 terms; per input a twiddle's rounding (half a
    unit in each of 4 products' shifts and the constants' 2^-63 of 2^60, an eighth), at most 3 units, of
    which the output sums up to 12."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "fx_limits_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_1804_05087_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "fx_limits_check.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    rows = [line.split() for line in out if line]
    assert len(rows) == 14
    for r, s, err in rows:
        assert float(err) < 6.0 + 1.0 + 3.0 * int(r), (r, s, err)
