"""The boundary rule in the lattice tiles (one link per lane) against the boundary tiles.

Launch variants 0-3, 11 and 12 evaluate the links of a 32-node chunk with at most 24
boundary nodes in its lattice warp; variant 9 evaluates every record in boundary
tiles. Both run the same rounded operations, so the stored states agree byte for byte.
The geometries cover chunks with few and with many boundary nodes, chunks on both sides
of the 24-node line, links that leave the lattice through the periodic (and sheared)
wrap, open and moving links, ragged rows, and several rounds of links per chunk.
"""
import numpy as np
import pytest

from paper_2009_04604_gb300 import lbm
from paper_2009_04604_gb300 import workloads as W

pytestmark = pytest.mark.gpu
HEADER = 128


def chunk_row(nx, ny, nz, seed):
    """One wall row above every fluid row, cut so that chunks hold 1 to 32 boundary nodes."""
    rng = np.random.default_rng(seed)
    flags = np.zeros((nz, ny, nx), np.uint8)
    for z in range(nz):
        for y in range(0, ny, 6):
            a = int(rng.integers(0, 8))
            flags[z, y, a:a + int(rng.choice([1, 5, 22, 23, 24, 25, 26, 31, 40]))] = lbm.SOLID
    return flags.reshape(-1)


def state(lat, dims, dtype, bc, coll, force, xshift, geo, launch):
    s = lbm.Simulation(lat, dims, 0.73, dtype)
    s.set_options(bc, 1.0, force, xshift)
    s.set_collision(coll)
    s.set_geometry(*geo)
    s.set_launch(*launch)
    c, w = lbm.lattice_info(lat)
    N, Q = int(np.prod(dims)), len(w)
    rho, u, xi = W.random_fields(N, 5, Q=Q, two_d=lat == lbm.D2Q9)
    s.set_populations(w * rho[:, None] * (1 + 3 * u @ c.T) * (1 + xi))
    s.step(6)
    out = s.save()[HEADER:]
    f = s.get_populations()
    s.close()
    return out, f


@pytest.mark.parametrize("lat,dims,xshift", [(lbm.D3Q19, (70, 14, 5), 0), (lbm.D2Q9, (96, 25, 1), 7),
                                             (lbm.D3Q27, (33, 13, 4), 0)])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("bc,coll,force", [("elibb_f", "bgk", (0, 0, 0)), ("elibb_fq", "bgk", (1e-4, 2e-5, 0)),
                                           ("elibb_f", "trt", (1e-4, -1e-5, 0)), ("elibb_fq", "trt", (0, 0, 0))])
@pytest.mark.parametrize("solid", [0.01, 0.06, 0.2, None])
def test_links_against_boundary_tiles(lat, dims, xshift, dtype, bc, coll, force, solid):
    Q = {lbm.D2Q9: 9, lbm.D3Q19: 19, lbm.D3Q27: 27}[lat]
    flags, q, uw, uw1, tag = W.random_geometry(dims, 11, solid or 0.1, 0.02, Q, moving=True)
    if solid is None:
        flags = chunk_row(*dims, 3)
        uw[:len(uw) // 2] = 0.0
        uw1[:len(uw1) // 2] = 0.0
    if lat == lbm.D2Q9:
        uw[..., 2] = uw1[..., 2] = 0.0
    geo = (flags, q, uw, uw1, tag)
    want, f = state(lat, dims, dtype, bc, coll, force, xshift, geo, (32, 4, 9, 1))
    assert np.isfinite(f).all()
    for launch in [(32, 4, 0, 2), (32, 8, 3, 4), (32, 4, 11, 1), (32, 8, 12, 1)]:
        got, _ = state(lat, dims, dtype, bc, coll, force, xshift, geo, launch)
        assert got == want, launch
