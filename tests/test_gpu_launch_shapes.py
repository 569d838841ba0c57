"""Launch shapes of the step kernels: results do not depend on them.

* mixed and seeded mixed kernels: blocks of 32 to 512 threads that meet at each substep, on
  ragged launches (lanes without a cell, blocks partly empty), give the same bits;
* cooperative kernels: one to eight cells a warp (chosen by the launch's cells) against one
  lane per cell, at the FP64 bound of the other parity tests.
"""
import os

import numpy as np
import pytest

import synthgen
from tests._parity import assert_fp64_parity

pytestmark = pytest.mark.gpu
DT = synthgen.DT_1E4YR
KEYS = ("T", "xH2", "xHp", "xe", "xCp", "xCO", "nsub", "status", "iters")


@pytest.fixture(scope="module")
def tc():
    import torch
    assert torch.cuda.is_available()
    import paper_2210_08024_gb300 as P
    P.build()
    from paper_2210_08024_gb300 import tc as T
    return T


def _step(tc, cells, mode, **kw):
    import torch
    d = tc.to_device(cells)
    st = tc.Stepper(mode, **kw)
    if mode == tc.TC_MODE_MIXED_SEEDED:
        import paper_2210_08024_gb300 as P
        with open(os.path.join(os.path.dirname(P.__file__), "weights", "seed_slab.bin"), "rb") as fh:
            st.load_mlp(fh.read())
    st.step(d, DT)
    torch.cuda.synchronize()
    st.close()
    return tc.from_device(d)


@pytest.mark.parametrize("mode", [2, 3])
@pytest.mark.parametrize("n", [1, 33, 513, 2999])
def test_mixed_blocks_agree_bit_for_bit(tc, mode, n):
    cells = synthgen.slab(ncell=n, key=31)
    ref = _step(tc, cells, mode, block=32, lanes_per_cell=1)
    for block, per_sm in ((128, 0), (256, 0), (512, 0), (512, 1)):
        g = _step(tc, cells, mode, block=block, blocks_per_sm=per_sm, lanes_per_cell=1)
        for k in KEYS:
            assert np.array_equal(g[k], ref[k]), (block, k)


@pytest.mark.parametrize("n", [1, 7, 608, 609, 1217, 4865])
def test_cooperative_groups_match_one_lane(tc, n):
    cells = synthgen.slab(ncell=n, key=32) if n > 700 else synthgen.cells_4096(n=n, key=33)
    ref = _step(tc, cells, 1, lanes_per_cell=1)
    g = _step(tc, cells, 1, lanes_per_cell=4)
    assert_fp64_parity(g, ref, "cooperative, %d cells" % n)
    assert np.array_equal(g["nsub"], ref["nsub"])
