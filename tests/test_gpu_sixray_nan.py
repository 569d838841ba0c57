"""NaN densities in the six-ray fields, with the low word of a canonical NaN and with others: the
fields are NaN exactly where the statement in numpy has them so, whatever the payload."""
import numpy as np
import pytest

from oracle import sixray as sr
from tests.test_gpu_sixray import PC, _gpu, _grid, tc  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("payload", [0x7FF8000000000000, 0x7FF80000FFFFFFFF, 0xFFF8000000000001, 0x7FFFFFFFFFF80000,
                                     0x7FF8000040000200])
def test_nan_payloads_propagate(tc, payload):  # noqa: F811
    n, x = _grid((9, 11, 13), key=71)
    n.view(np.uint64)[4, 5, 6] = payload
    x.view(np.uint64)[2, 3, 4] = payload
    g = _gpu(tc, n, x, 2.0 * PC)
    with np.errstate(invalid="ignore"):
        r = sr.sixray(n, x, 2.0 * PC)
    for k in ("chi_pe", "chi_lw", "f_h2", "N_eff", "xi"):
        assert np.array_equal(np.isnan(g[k]), np.isnan(r[k])), k
