"""The benchmark's DRAM traffic figure belongs to one kernel in one launch shape on one grid (it is
the resident threads' stacks): any other launch has none."""
import pytest

import bench

PEAKS = {"fp64_fma_per_s": 5e11, "weights": {"div": 5.7, "sqrt": 8.6, "exp": 10.8, "log": 20.9}}
SHAPE = {"block": 128, "blocks_per_sm": 0, "lanes_per_cell": 1, "ms": 52.0}


@pytest.mark.parametrize("mode,ncell,shape,has", [
    ("newton", 2097152, SHAPE, True), ("newton", 2097152, dict(SHAPE, blocks_per_sm=8), True),
    ("newton", 2097152, dict(SHAPE, block=64), False), ("newton", 2097152, dict(SHAPE, blocks_per_sm=4), False),
    ("newton", 2097152, dict(SHAPE, lanes_per_cell=4), False), ("newton", 64 ** 3, SHAPE, False),
    ("paper", 2097152, SHAPE, False)])
def test_traffic_only_for_the_profiled_launch(mode, ncell, shape, has):
    r = {"kernel_ms": 50.0, "launch_shape": shape}
    t = bench.roofline_of(bench.work_per_cell(), r, mode, ncell, PEAKS)["traffic"]
    assert (t == bench.TRAFFIC_BYTES_PER_CELL * ncell) if has else t is None
