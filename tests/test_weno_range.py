"""The FP64 nonlinear reconstructions and their transposes stay right for data
of any size whose smoothness indicators (squares of the data) FP64 can hold
(csrc/recon.cuh, csrc/adjoint.cuh), on the host against the formulas of
Sec. 2.1 in long double."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fp64_weno_keeps_its_range(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "range_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2",
                    "-I", os.path.join(ROOT, "paper_2005_08736_gb300", "csrc"),
                    "-I", os.path.join(ROOT, "include"), "-x", "cu",
                    os.path.join(ROOT, "tests", "support", "range_check.cu"), "-o", exe],
                   check=True, capture_output=True)
    values, transposes = (float(x) for x in subprocess.run([exe], check=True, capture_output=True,
                                                           text=True).stdout.split())
    # FP64 rounding (1e-16) through indicators that may be 1e-4 of the largest
    # and weights with their squares: 1e-12 and, one derivative more, 1e-10.
    assert values < 1e-12, values
    assert transposes < 1e-10, transposes
