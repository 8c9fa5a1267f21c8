"""Lattices with more rows than a grid has: the bulk step hands over to the tile table.

The bulk step's grid is the lattice, so from 65536 rows on its variants run the tile
table's kernel. Both sides of that line give the states of the split step (variant 9, which
always runs from a table), byte for byte.
"""
import numpy as np
import pytest

from paper_2009_04604_gb300 import lbm
from paper_2009_04604_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [65535, 65536, 65601])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_rows_beyond_the_grid(ny, dtype):
    dims, Q = (31, ny, 1), 9
    N = dims[0] * ny
    rng = np.random.default_rng(2)
    flags = np.where(rng.random(N) < 0.05, lbm.SOLID, lbm.FLUID).astype(np.uint8)
    q = rng.uniform(0.05, 1.0, (N, Q))
    c, w = lbm.lattice_info(lbm.D2Q9)
    rho, u, xi = W.random_fields(N, 5, Q=Q, two_d=True)
    f = w * rho[:, None] * (1 + 3 * u @ c.T) * (1 + xi)
    out = []
    for launch in (None, (32, 4, 11, 2), (32, 4, 9, 1)):
        s = lbm.Simulation(lbm.D2Q9, dims, 0.8, dtype)
        s.set_options("elibb_fq", 1.0, (1e-5, 0, 0))
        s.set_geometry(flags, q)
        if launch:
            s.set_launch(*launch)
        s.set_populations(f)
        s.step(5)
        out.append(s.save()[128:])
        s.close()
    assert out[0] == out[1] == out[2]
