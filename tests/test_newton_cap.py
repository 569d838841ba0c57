"""tc_params.newton_max caps a substep's solve in the FP64 Newton mode, whichever of its iterations
take it, on the host build of the step functions: a substep that neither restarts nor halves spends
at most that many iterations, and cells without either keep the oracle's results."""
import numpy as np
import pytest

import oracle
import synthgen
from tests._parity import assert_fp64_parity
from tests.test_host_step import DT, exe as host_exe, host_step, tc  # noqa: F401  (fixtures)


class Capped:
    def __init__(self, tc, cap):
        self.tc, self.cap = tc, cap

    def tc_params_default(self, mode):
        p = self.tc.tc_params_default(mode)
        p.newton_max = self.cap
        return p


@pytest.mark.parametrize("cap", [3, 4, 6, 27, 28])
def test_cap_holds(host_exe, tc, tmp_path, cap):  # noqa: F811
    c = synthgen.cells_4096(n=256, key=61)
    g = host_step(host_exe, Capped(tc, cap), c, tc.TC_MODE_NEWTON_FP64, tmp_path)
    plain = g["status"] == 0
    assert np.all(g["iters"][plain] <= cap * g["nsub"][plain])
    ref = oracle.step(c, DT, oracle.default_params(mode=1))
    both = plain & (ref["status"] == 0)
    assert_fp64_parity({k: g[k][both] for k in ("T", "xH2", "xHp")}, {k: ref[k][both] for k in ("T", "xH2", "xHp")},
                       "cap %d" % cap)
