"""The FP32 dual-number derivatives (source_tangents, csrc/tc_dual.cuh) over the whole range of
states, T = 1 to 1e9 K, n = 1e-4 to 1e6, abundances from 0 up, on the host build of the library's
own physics (tests/host/tc_tangent_range_check.cu): every value and derivative is finite, and the
derivatives along ln T hold the bound of tests/test_tangent.py, 1e-4 of their magnitude plus that of
the terms they are differences of.  (Gas without metals is left out: where it has no ions either,
x_e n < 1e-30, it leaves FP32's range, and the plain iteration takes it.)"""
import json
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_08024_gb300", "csrc")


def test_tangents_stay_finite_and_right(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "tc_tangent_range_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-x", "cu", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "tc_tangent_range_check.cu"), "-o", exe],
                   check=True, capture_output=True)
    r = json.loads(subprocess.run([exe], check=True, capture_output=True, text=True).stdout)
    assert r["bad"] == 0, r
    for k in ("H", "CH2", "CHp"):
        assert r[k] <= 1e-4, r
