"""The table-driven FP64 exponential and logarithm (csrc/tc_exp64.cuh) on the host, against
long double: the same operations as on the device (every rounding is FP64's or an FMA's).

Bounds, from the method: half a unit in the last place for the final rounding; the parts
added there are below 2^-8 of the result (exp64: |p| <= ln2/1024; log64: 2^-8 once the table
part is nonzero), so their own roundings add at most 2^-8 units or so each.  Around 1 the
logarithm is r + r^2 q: one unit.
"""
import json
import os
import platform
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_08024_gb300", "csrc")


def test_exp64_and_log64_round_to_half_a_unit(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    if platform.machine() not in ("x86_64", "aarch64"):
        pytest.skip("needs a long double wider than double")
    exe = str(tmp_path / "tc_exp64_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-x", "cu", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "tc_exp64_check.cu"), "-o", exe], check=True,
                   capture_output=True)
    r = json.loads(subprocess.run([exe], check=True, capture_output=True, text=True).stdout)
    assert r["ends"] == 1
    assert r["exp"] < 0.52 and r["exp_small"] < 0.52, r
    assert r["log"] < 0.53 and r["log_bins"] < 1.0 and r["log_one"] < 1.0, r
