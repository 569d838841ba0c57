"""Roots of the FP64 Newton's fast path (newton_tangent) against long double roots of the same
substep, on the host build of the library's own functions (tests/host/tc_root_check.cu): no
absolute floor, so that x_H2 of 1e-20 to 1e-15 in hot gas counts as much as any.

Bound: a solve ends when every step is below newton_rtol = 1e-12 of its unknown, or when the last
two show that the next would be below a hundredth of it; what is left is at most such a step, and
the residual's rounding (1e-16, through coefficients up to 1e3) is a tenth of it: 2e-12.
"""
import json
import os
import shutil
import subprocess

import numpy as np
import pytest

import synthgen

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_08024_gb300", "csrc")
IN_KEYS = ("n", "chi_pe", "chi_lw", "f_h2", "f_c", "F_lyc", "xi", "Zg", "Zd", "T", "xH2", "xHp")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("root") / "tc_root_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-x", "cu", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "tc_root_check.cu"), "-o", out],
                   check=True, capture_output=True)
    return out


def _snr(k):
    """Supernova interiors: the slab's cells at a hundredth of their density, hot and ionised."""
    c = synthgen.slab(ncell=k, key=51)
    r = np.random.default_rng(52)
    return dict(c, n=0.01 * c["n"], T=10.0 ** r.uniform(6.0, 8.0, k), xH2=np.zeros(k), xHp=np.ones(k))


def _hii(k):
    c = synthgen.slab(ncell=k, key=53)
    r = np.random.default_rng(54)
    return dict(c, F_lyc=10.0 ** r.uniform(5.0, 11.0, k), T=np.full(k, 1e4), xHp=np.full(k, 0.5), xH2=np.zeros(k))


CELLS = {"snr": lambda: _snr(800), "hii": lambda: _hii(400), "states": lambda: synthgen.cells_4096(n=600, key=55),
         "slab": lambda: synthgen.slab(ncell=1500, key=56)}


@pytest.mark.parametrize("dt_yr", [1e4, 1e5])
@pytest.mark.parametrize("workload", sorted(CELLS))
def test_roots_match_long_double(check, tmp_path, workload, dt_yr):
    cells = CELLS[workload]()
    n = cells["T"].size
    path = tmp_path / "cells.bin"
    with open(path, "wb") as fh:
        fh.write(np.int64(n).tobytes())
        for k in IN_KEYS:
            v = cells.get(k, {"f_c": 1.0, "F_lyc": 0.0}.get(k, 1.0))
            fh.write(np.ascontiguousarray(np.broadcast_to(np.asarray(v, np.float64), (n,))).tobytes())
        fh.write(np.float64(dt_yr * 3.15576e7).tobytes())
    r = json.loads(subprocess.run([check, str(path)], check=True, capture_output=True, text=True).stdout)
    assert r["miscounted"] == 0, r  # an abandoned solve's iterations are in newton_iters
    assert r["noroot"] == 0 and r["left"] < 0.02 * r["substeps"], r
    assert max(r[k] for k in ("T", "xH2", "xHp")) <= 2e-12, r
