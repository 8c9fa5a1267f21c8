"""Density, velocity and mass of FP32, FP16 and BF16 populations against exact sums.

The populations are made of values that the storage type holds exactly and that are
multiples of 2^-50, so that the reference is exact in integers and fractions: values over
26 binades, and a fluid near rest under a density offset, where the momentum is a small
difference of large terms.

Bound. With D = sum t_i, J = sum c t_i, R = rho0 + D and S = sum |t_i| the kernel's sums
are exact up to their last slice, 2^-54 S, and then rounded: to D, to J and J + F/2, to R,
and the quotient, 2^-53 each. So r is within e_r = 2^-53 (|R| + |D|) + 2^-54 S, and u
within (2^-53 (|J| + |J + F/2|) + 2^-54 S) / |R| + |U| (e_r / |R| + 2^-53), 1 % added for
the products of these.
"""
from fractions import Fraction as Fr

import numpy as np
import pytest

from paper_2009_04604_gb300 import lbm

pytestmark = pytest.mark.gpu
UNIT = 2.0 ** -50


def stored(x, dtype):
    """x rounded to what the storage holds, in multiples of UNIT."""
    if dtype == "f16":
        return (x * 2.0 ** 14).astype(np.float16).astype(np.float64) * 2.0 ** -14
    x = x.astype(np.float32)
    if dtype == "bf16":
        x = (x.view(np.uint32) & np.uint32(0xffff0000)).view(np.float32)
    return np.trunc(x.astype(np.float64) / UNIT) * UNIT


def wide(rng, N, Q, w, c):
    t = np.exp2(rng.uniform(-26.0, -4.0, (N, Q))) * rng.choice([-1.0, 1.0], (N, Q))
    t[rng.random((N, Q)) < 0.05] = 0.0
    return t


def near_rest(rng, N, Q, w, c):
    u = 1e-8 * rng.standard_normal((N, 3))
    return w * (0.05 * rng.uniform(0.5, 1.5, (N, 1)) + 3.0 * (u @ c.T))


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("lat,dims", [(lbm.D2Q9, (37, 9, 1)), (lbm.D3Q19, (33, 5, 3)), (lbm.D3Q27, (32, 4, 3))])
@pytest.mark.parametrize("force", [(0.0, 0.0, 0.0), (1e-3, -2e-4, 3e-5)])
@pytest.mark.parametrize("values", [wide, near_rest])
def test_fields_against_exact_sums(values, force, lat, dims, dtype):
    c, w = lbm.lattice_info(lat)
    Q, N = len(w), int(np.prod(dims))
    s = lbm.Simulation(lat, dims, 0.8, dtype)
    s.set_options(lbm.BC_ELIBB_F, 1.0, force, 0)
    s.set_geometry(np.zeros(N, np.uint8))
    t = stored(values(np.random.default_rng(3), N, Q, w, c), dtype)
    s.set_populations(w + t)
    r, u = (x.cpu().numpy() for x in s.macros())
    ti = np.rint(t / UNIT).astype(np.int64).astype(object)
    ui = Fr(1, 2 ** 50)
    F = [Fr(x) / 2 for x in force[:2]] + [Fr(force[2]) / 2 if lat != lbm.D2Q9 else Fr(0)]
    e53, total, total_bound = Fr(1, 2 ** 53), Fr(0), Fr(0)
    for n in range(N):
        D = sum(ti[n]) * ui
        S = sum(abs(x) for x in ti[n]) * ui
        R = 1 + D
        er = Fr(101, 100) * (e53 * (abs(R) + abs(D)) + e53 / 2 * S)
        assert abs(Fr(float(r[n])) - R) <= er
        total += R
        total_bound += er
        for a in range(3):
            J = sum(int(c[i, a]) * ti[n, i] for i in range(Q)) * ui
            U = (J + F[a]) / R
            eu = (e53 * (abs(J) + abs(J + F[a])) + e53 / 2 * S) / abs(R) + abs(U) * (er / abs(R) + e53)
            assert abs(Fr(float(u[n, a])) - U) <= Fr(101, 100) * eu
    assert abs(Fr(s.mass()) - total) <= total_bound + N * e53 * total
