"""The FP64 quotient of the physics (m_div) on the GPU, and exp64 and log64 against their
host build (tests/host/tc_div64_check.cu).

Bound of the quotient: the reciprocal y is good to ~2^-53 after its step, so the corrected
quotient rounds once, plus the correction's error, |q - a/b| 2^-53 / ulp: 0.51 units.  The
exponential and the logarithm are the same operations on both sides: equal bits."""
import json
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_08024_gb300", "csrc")


def test_quotient_and_tables_on_the_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "tc_div64_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "tc_div64_check.cu"), "-o", exe], check=True,
                   capture_output=True)
    r = json.loads(subprocess.run([exe], check=True, capture_output=True, text=True).stdout)
    assert r["div_ulp"] < 0.51, r
    assert r["exp_differs"] == 0 and r["log_differs"] == 0 and r["special_differs"] == 0, r
