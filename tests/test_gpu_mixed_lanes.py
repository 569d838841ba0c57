"""The default lanes per cell of the mixed mode: four while every cell's lanes are resident at once
(128 cells per SM), else one.  Four lanes and one differ by the polish's remainder, so the line is
part of the results: they equal, bit for bit, those of the stated number of lanes."""
import numpy as np
import pytest

import synthgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,lanes", [(1, 4), (4864, 4), (4865, 4), (19456, 4), (19457, 1)])
def test_default_lanes(n, lanes):
    import paper_2210_08024_gb300 as P
    P.build()
    import torch
    from paper_2210_08024_gb300 import tc
    n = n * torch.cuda.get_device_properties(0).multi_processor_count // 152 if n > 1 else n
    c = synthgen.cells_4096(n=n, key=41)
    a = tc.step_numpy(c, 1e2 * 3.15576e7, tc.TC_MODE_MIXED)
    b, other = (tc.step_numpy(c, 1e2 * 3.15576e7, tc.TC_MODE_MIXED, lanes_per_cell=k) for k in (lanes, 5 - lanes))
    assert n == 1 or any(not np.array_equal(other[k], b[k]) for k in ("T", "xH2", "xHp", "xe"))
    for k in ("T", "xH2", "xHp", "xe", "xCp", "xCO", "nsub", "status", "iters"):
        assert np.array_equal(a[k], b[k]), k
