"""The pair arithmetic that k_march runs (csrc/march.cuh, csrc/packed.cuh,
csrc/compat.cuh) against the scalar functions, half by half on the host: the
scaled tangential reconstructions, the compatibility state's midpoint rule and
the conditions under which it is taken, and the face fields on smooth, rough
and mixed pairs.  The tiles that evaluated these in scalar form are gone, so
the two forms meet here."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_march_pairs_match_the_scalar_functions(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "march_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2",
                    "-I", os.path.join(ROOT, "paper_2005_08736_gb300", "csrc"),
                    "-I", os.path.join(ROOT, "include"), "-x", "cu",
                    os.path.join(ROOT, "tests", "support", "march_check.cu"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    tangential, rule, fields = (float(x) for x in out[:3])
    taken, refused, mixed = (int(x) for x in out[3:])
    # A dozen FP32 roundings (6e-8) of numbers of the stated sizes, the
    # derivatives' coefficients summing to 4; for the compatibility state the
    # direct form's cancelling moments too.  A wrong term would show at the
    # size of the jumps, 1e-4 and more.
    assert tangential < 3e-6, tangential
    assert rule < 3e-7, rule
    assert fields < 2e-6, fields
    assert min(taken, refused, mixed) > 500, (taken, refused, mixed)
