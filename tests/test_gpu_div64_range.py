"""The FP64 quotient of the physics (m_div) against the correctly rounded division over all
exponents, and around the edges of the range it takes (tests/host/tc_div64_range_check.cu).

Bound: its error is below 0.51 units of the last place (tests/test_gpu_div64.py), below one unit
where it is subnormal, so it is the rounded quotient or a neighbour of it; and it is infinite or NaN
only where the division is."""
import json
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_08024_gb300", "csrc")


def test_quotient_over_all_exponents(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "tc_div64_range_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "tc_div64_range_check.cu"), "-o", exe], check=True,
                   capture_output=True)
    r = json.loads(subprocess.run([exe], check=True, capture_output=True, text=True).stdout)
    assert r["not_finite"] == 0 and r["units"] <= 1, r
