"""The FP64 Newton's Jacobian from FP32 dual numbers (source_tangents, csrc/tc_dual.cuh)
against central differences of the FP64 source terms, on the host build of the library's
own physics (tests/host/tc_tangent_check.cu).

Bound: an FP32 operation rounds to 6e-8 and a term passes through at most ~30 of them in
a row (and through exponentials with arguments up to ~30, whose rounding the exponential
scales by as much), so a derivative is good to ~1e-4 of its magnitude plus that of the
terms it is a difference of.  A wrong derivative of any one term leaves a part of order
one.  The differences' own errors are below 1e-8 (step 1e-5, relative).

The solve that uses it must also hold abundances that leave FP32's range: dense cells
without ionisation, whose x_H+ decays by many orders of magnitude a substep.
"""
import json
import os
import shutil
import subprocess

import numpy as np
import pytest

import synthgen
from tests.test_host_step import exe as host_exe, host_step, tc  # noqa: F401  (fixtures)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_08024_gb300", "csrc")
IN_KEYS = ("n", "chi_pe", "chi_lw", "f_h2", "f_c", "F_lyc", "xi", "Zg", "Zd", "T", "xH2", "xHp")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("tangent") / "tc_tangent_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-x", "cu", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "tc_tangent_check.cu"), "-o", out],
                   check=True, capture_output=True)
    return out


@pytest.mark.parametrize("workload", ["slab", "states", "photoionised", "no_dust"])
def test_dual_jacobian_matches_differences(check, tmp_path, workload):
    cells = synthgen.slab(ncell=400, key=21) if workload == "slab" else synthgen.cells_4096(n=400, key=22)
    if workload == "photoionised":
        cells["F_lyc"] = np.full(400, 1e9)
    if workload == "no_dust":
        cells["Zd"] = np.zeros(400)
    path = tmp_path / "cells.bin"
    with open(path, "wb") as fh:
        fh.write(np.int64(400).tobytes())
        for k in IN_KEYS:
            fh.write(np.ascontiguousarray(np.broadcast_to(np.asarray(cells[k], np.float64), (400,))).tobytes())
        fh.write(np.float64(0.0).tobytes())
    r = json.loads(subprocess.run([check, str(path)], check=True, capture_output=True, text=True).stdout)
    bad = {k: v for k, v in r.items() if not v < 1e-4}
    assert not bad, bad


def test_traces_below_fp32_range_stay_positive(host_exe, tc, tmp_path):  # noqa: F811
    import oracle
    one = np.ones(4)
    cells = dict(n=5.8e3 * one, chi_pe=0.02 * one, chi_lw=2.6e-4 * one, f_h2=one, f_c=one, F_lyc=0 * one,
                 xi=np.array([0.0, 0.0, 1e-25, 2e-16]), Zg=one, Zd=one, T=100 * one,
                 xH2=np.array([0.0, 0.3, 0.0, 0.0]), xHp=np.array([1e-4, 1e-40, 1e-4, 0.0]))
    import tests.test_host_step as hs
    dt, hs.DT = hs.DT, 3.15576e13
    try:
        g = host_step(host_exe, tc, cells, tc.TC_MODE_NEWTON_FP64, tmp_path)
    finally:
        hs.DT = dt
    ref = oracle.step(cells, 3.15576e13, oracle.default_params(mode=1))
    assert np.array_equal(g["status"], ref["status"]) and np.array_equal(g["nsub"], ref["nsub"])
    assert np.all(g["xHp"] >= 0.0)
    for k in ("T", "xH2", "xHp"):
        np.testing.assert_allclose(g[k], ref[k], rtol=1e-9, atol=0.0 if k == "T" else 1e-14, err_msg=k)
