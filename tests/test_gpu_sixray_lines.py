"""The six-ray line kernel at the edges of its rules: lines that fill a warp exactly, by one
more or one less, on flattened odd planes; 8, 16 and 32 segments a line with remainders;
lines shorter than the segments; empty and nearly empty columns; strong shielding.
Tolerance: that of the other six-ray tests, 1e-10 against the numpy statement."""
import numpy as np
import pytest

from oracle import sixray as sr
from tests.test_gpu_sixray import PC, RTOL, _compare, _gpu, _grid, tc  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 4, 8), (31, 1, 33), (17, 33, 3), (33, 63, 65), (64, 64, 64), (129, 31, 7),
                                   (2, 150, 130), (7, 2, 1)])
@pytest.mark.parametrize("mu", [-6.0, 3.0])
def test_line_edges(tc, shape, mu):  # noqa: F811
    n, x = _grid(shape, key=sum(shape) + 1, mu=mu, sig=2.0)
    x[n > np.median(n)] = 0.0
    n.ravel()[:: 7] = 1e-12
    g = _gpu(tc, n, x, 3.0 * PC, chi0=1.5, xi0=1e-16, Zd=1.3)
    r = sr.sixray(n, x, 3.0 * PC, chi0=1.5, xi0=1e-16, Zd=1.3)
    _compare(g, r, rtol=RTOL)
