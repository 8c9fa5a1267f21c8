"""Density, velocity and mass read-out against FP64 sums of the same stored populations.

get_populations returns the stored values exactly in FP64 (up to the addition of
w_i rho0), so the host's FP64 sums are the reference. The kernel sums FP32 values
as pairs of floats. Its bound: every one of the at most Q + 2 additions rounds the
low half once, and the low half is at most (Q + 2) 2^-24 S with S = sum |f_i - w_i rho0|
(+ rho0 for the density's last one), so the error is below (Q + 2)^2 2^-48 S, plus
2^-52 of the value itself for the FP64 additions. The quotient adds 2^-44 of itself.
"""
import numpy as np
import pytest

from paper_2009_04604_gb300 import lbm

pytestmark = pytest.mark.gpu

CASES = [(lbm.D2Q9, (37, 9, 1)), (lbm.D2Q9, (32, 8, 1)), (lbm.D3Q19, (33, 7, 5)), (lbm.D3Q27, (65, 5, 3)),
         (lbm.D3Q19, (1, 3, 2))]


def make(lat, dims, dtype, force):
    s = lbm.Simulation(lat, dims, 0.8, dtype)
    s.set_options(lbm.BC_ELIBB_F, 1.0, force, 0)
    flags = np.zeros(int(np.prod(dims)), np.uint8)
    flags[::5] = lbm.SOLID
    s.set_geometry(flags)
    return s, flags == 0


@pytest.mark.parametrize("dtype", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("lat,dims", CASES)
@pytest.mark.parametrize("force", [(0.0, 0.0, 0.0), (1e-3, -2e-4, 3e-5)])
def test_fields_against_fp64_sums(lat, dims, dtype, force):
    s, fluid = make(lat, dims, dtype, force)
    c, w = lbm.lattice_info(lat)
    Q, N = len(w), fluid.size
    rng = np.random.default_rng(7)
    s.set_populations(w * (1.0 + 0.05 * rng.standard_normal((N, 1))) + 0.02 * w * rng.standard_normal((N, Q)))
    f = s.get_populations() - np.where(fluid[:, None], w, 0.0)
    F = np.array(force if lat != lbm.D2Q9 else (force[0], force[1], 0.0))
    rho = np.where(fluid, 1.0 + f.sum(1), 0.0)
    u = np.where(fluid[:, None], (f @ c + 0.5 * F) / np.where(fluid, rho, 1.0)[:, None], 0.0)
    S = np.abs(f).sum(1)
    e = (Q + 2) ** 2 * 2.0 ** -48 * (S + 1.0) + Q * 2.0 ** -52 * (1.0 + S)
    r, v = (t.cpu().numpy() for t in s.macros())
    assert np.all(np.abs(r - rho) <= e)
    assert np.all(np.abs(v - u) <= 2 * e[:, None] + 2.0 ** -44 * np.abs(u))
    assert abs(s.mass() - rho.sum()) <= e.sum() + N * 2.0 ** -52 * rho.sum()


@pytest.mark.parametrize("value", [1e31, 3e38, np.inf, -np.inf, np.nan])
def test_values_beyond_the_pair_sums(value):
    lat, dims = lbm.D3Q19, (40, 3, 3)
    s, fluid = make(lat, dims, "f32", (0.0, 0.0, 0.0))
    c, w = lbm.lattice_info(lat)
    f = np.tile(w, (fluid.size, 1))
    f[fluid] += 1e-3
    f[7, 3] = f[8, :] = value  # nodes 7 and 8 are fluid
    s.set_populations(f)
    r, v = (t.cpu().numpy() for t in s.macros())
    ok = fluid.copy()
    ok[[7, 8]] = False
    assert np.all(np.isfinite(r[ok])) and np.all(np.isfinite(v[ok]))
    if np.isfinite(value):
        st = s.get_populations()
        want = 1.0 + (st - w).sum(1)
        assert np.allclose(r[[7, 8]], want[[7, 8]], rtol=1e-12)
        big = np.abs(v[7] - ((st[7] - w) @ c) / want[7])
        assert np.all(big <= 1e-12)
    else:
        assert not np.isfinite(r[7]) and not np.isfinite(r[8])
        with pytest.raises(lbm.LBMError):
            s.mass()
