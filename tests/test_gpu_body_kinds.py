"""The node kinds of a moving body's region are those of the same shape in a static geometry.

The region's nodes are decided in FP32 away from the surface and in FP64 near it, the
static build's all in FP64. Compared at the first pose and after some steps of a path that
moves and, for the sphere, spins; with slender ellipsoids turned to an angle.
"""
import numpy as np
import pytest

from paper_2009_04604_gb300 import lbm

pytestmark = pytest.mark.gpu
STEPS = 5
CASES = [(lbm.D2Q9, (96, 80, 1), dict(type="sphere", r=(11.3, 0, 0))),
         (lbm.D2Q9, (96, 80, 1), dict(type="ellipsoid", r=(16.0, 4.1, 1.0), ang=0.7)),
         (lbm.D2Q9, (1200, 1100, 1), dict(type="ellipsoid", r=(500.0, 0.4, 1.0), ang=0.41)),
         (lbm.D2Q9, (1200, 1100, 1), dict(type="ellipsoid", r=(0.02, 510.0, 1.0), ang=1.1)),
         (lbm.D3Q19, (64, 48, 40), dict(type="sphere", r=(9.7, 0, 0))),
         (lbm.D3Q19, (64, 56, 40), dict(type="ellipsoid", r=(18.0, 0.3, 8.0), ang=0.9)),
         (lbm.D3Q27, (48, 48, 40), dict(type="ellipsoid", r=(5.2, 11.0, 0.6), ang=2.2))]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("lat,dims,shape", CASES)
def test_region_kinds(lat, dims, shape, dtype):
    v = np.array([0.31, -0.17, 0.13 if dims[2] > 1 else 0.0])
    c0 = np.array([d / 2.0 - 0.37 for d in dims[:2]] + [dims[2] / 2.0 - 0.21 if dims[2] > 1 else 0.0])
    traj = np.zeros((STEPS + 2, 9))
    traj[:, :3] = c0 + v * np.arange(STEPS + 2)[:, None]
    traj[:, 3:6] = v
    s = lbm.Simulation(lat, dims, 0.8, dtype)
    s.build_geometry()
    s.set_moving_body(dict(shape, tag=1), traj)
    s.init(1.0)
    for k in range(0, STEPS + 1, STEPS):
        t = lbm.Simulation(lat, dims, 0.8, dtype)
        t.build_geometry(None, None, [dict(shape, tag=1, c=tuple(traj[k, :3]))])
        assert np.array_equal(s.get_geometry()[0], t.get_geometry()[0])
        t.close()
        if k == 0:
            assert (s.get_geometry()[0] == lbm.SOLID).any() or shape["r"][0] < 0.1
            s.step(STEPS)
    s.close()
