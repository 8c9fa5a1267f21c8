"""A moving body's link geometry does not depend on how large its region is.

The region covers the whole trajectory. With at most 4096 chunks of 32 nodes in it the
record kernel sums the chunk counts before its block itself; above that they come from
scans. The same first poses with a far pose added later give the larger region: the
populations agree bit for bit, and the force, summed over records in region order, to
rounding (1e-12 of its largest component).
"""
import numpy as np
import pytest

from paper_2009_04604_gb300 import lbm

pytestmark = pytest.mark.gpu
DIMS = (152, 46, 44)
STEPS = 6


def run(shape, far, dtype):
    t = np.zeros((STEPS + 2, 9))
    t[:, 0] = 24.3 + 0.4 * np.arange(STEPS + 2)
    t[:, 1:3] = 22.6, 21.4
    t[:, 3] = 0.4
    t[:, 8] = 0.003
    if far:
        t = np.vstack([t, t[-1]])
        t[-1, 0] = 129.0
    s = lbm.Simulation(lbm.D3Q19, DIMS, 0.8, dtype)
    s.build_geometry()
    s.set_moving_body(shape, t)
    s.init(1.0, (0.01, 0.0, 0.0))
    s.step(STEPS)
    out = s.get_populations(), s.wall_force(1)
    s.close()
    return out


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", [dict(type="sphere", tag=1, r=(16.2, 0, 0)),
                                   dict(type="ellipsoid", tag=1, r=(9.3, 16.0, 15.4), ang=0.6)])
def test_large_and_small_regions_agree(shape, dtype):
    f0, F0 = run(shape, False, dtype)
    f1, F1 = run(shape, True, dtype)
    assert np.isfinite(f0).all() and np.abs(F0).max() > 0
    assert np.array_equal(f0, f1)
    assert np.abs(F0 - F1).max() <= 1e-12 * np.abs(F0).max()
