"""The four lanes of a cell share the exponentials of its temperature blocks.

Each lane evaluates every fourth exponential and hands it to the others.  Which ones exist
depends on the switches (no ro-vibrational cooling, no CIE, constant k_gr), so the kernel is
compared with the one-lane kernel, which evaluates them in place, under each of them, on
temperatures from 12 K to 1e7 K and on ragged launches, at the FP64 bound of the other parity
tests.
"""
import numpy as np
import pytest

import synthgen
from tests._parity import assert_fp64_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, 1, 2, 4, 7])
@pytest.mark.parametrize("n", [1, 35, 1201])
def test_shared_exponentials_match_one_lane(flags, n):
    import paper_2210_08024_gb300 as P
    P.build()
    from paper_2210_08024_gb300 import tc
    c = synthgen.cells_4096(n=n, key=34)
    c["T"] = np.geomspace(12.0, 1e7, n)
    a = tc.step_numpy(c, 1e-2 * synthgen.DT_1E4YR, 1, lanes_per_cell=1, flags=flags)
    b = tc.step_numpy(c, 1e-2 * synthgen.DT_1E4YR, 1, lanes_per_cell=4, flags=flags)
    assert_fp64_parity(b, a, "flags %d, %d cells" % (flags, n))
    assert np.array_equal(a["nsub"], b["nsub"]) and not np.any(b["status"] & tc.TC_ST_ERROR_MASK)
