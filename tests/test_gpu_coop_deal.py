"""Cells dealt to the warps of a cooperative launch (no cost hint, every cell with its own
lanes) and cells claimed from the queue (with a hint, or one cell more than there are lanes)
give the same bits, each cell advanced once."""
import numpy as np
import pytest

import synthgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("n", [257, 609, 4863, 4864, 4865])
def test_dealt_and_queued_cells_agree(mode, n):
    import paper_2210_08024_gb300 as P
    P.build()
    from paper_2210_08024_gb300 import tc
    c = synthgen.slab(ncell=n, key=35)
    hinted = dict(c, cost_hint=np.arange(n, dtype=np.int32))
    a = tc.step_numpy(c, synthgen.DT_1E4YR, mode, lanes_per_cell=4)
    b = tc.step_numpy(hinted, synthgen.DT_1E4YR, mode, lanes_per_cell=4)
    assert np.all(a["nsub"] > 0)
    for k in ("T", "xH2", "xHp", "xe", "xCp", "xCO", "nsub", "status", "iters"):
        assert np.array_equal(a[k], b[k]), k
