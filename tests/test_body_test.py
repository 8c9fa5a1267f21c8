"""The FP32 test of a moving body's region agrees with the FP64 definition wherever it
decides, for spheres and for ellipsoids up to the aspect ratios a lattice can hold.

csrc/body_test.hpp is compiled here as plain C++. The points are lattice nodes, and the
centre is placed so that each lies within a chosen distance of the surface, down to 1e-9
of it, on either side; a node's neighbours are tested with the stepped offsets that the
kernel uses.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2009_04604_gb300", "csrc")
SOURCE = """
#include "body_test.hpp"
extern "C" void sides(int D, int n, const double *r, const double *ca, const double *sa, const double *c,
                      const int *x, const int *step, int *out, float *tol) {
  for (int k = 0; k < n; ++k) {
    const lbm::BodySurface b = lbm::body_surface(D, r + 3 * k, ca[k], sa[k]);
    float d[3];
    for (int a = 0; a < 3; ++a) d[a] = a < D ? (float)(x[3 * k + a] - c[3 * k + a]) - step[3 * k + a] : 0.0f;
    out[k] = lbm::body_side(b, d[0], d[1], d[2]);
    tol[k] = b.tol;
  }
}
"""


@pytest.fixture(scope="module")
def sides(tmp_path_factory):
    d = tmp_path_factory.mktemp("body")
    src, lib = str(d / "sides.cpp"), str(d / "sides.so")
    open(src, "w").write(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib],
                   check=True)
    fn = ctypes.CDLL(lib).sides

    def run(D, r, ca, sa, c, x, step):
        n = len(ca)
        out, tol = np.zeros(n, np.int32), np.zeros(n, np.float32)
        ptr = [np.ascontiguousarray(v).ctypes.data_as(ctypes.c_void_p) for v in (r, ca, sa, c)]
        xi, st = np.ascontiguousarray(x, np.int32), np.ascontiguousarray(step, np.int32)
        fn(D, n, *ptr, xi.ctypes.data_as(ctypes.c_void_p), st.ctypes.data_as(ctypes.c_void_p),
           out.ctypes.data_as(ctypes.c_void_p), tol.ctypes.data_as(ctypes.c_void_p))
        return out, tol
    return run


def points(D, n, rmin, rmax, seed):
    rng = np.random.default_rng(seed)
    r = np.ones((n, 3))
    r[:, :D] = np.exp(rng.uniform(np.log(rmin), np.log(rmax), (n, D)))
    r[0::2, 0], r[0::2, 1] = rmax, rmin  # half of them at the full ratio
    swap = rng.random(n) < 0.5
    r[swap, :2] = r[swap, 1::-1]
    ang = rng.uniform(0, 2 * np.pi, n)
    ca, sa = np.cos(ang), np.sin(ang)
    s = rng.standard_normal((n, 3)) * (np.arange(3) < D)  # a point of the unit sphere, often near a tip
    s[rng.random(n) < 0.5] *= [1.0, 1e-4, 1e-4]
    s /= np.linalg.norm(s, axis=1, keepdims=True)
    b = s * r * (1.0 + rng.choice([-1, 1], (n, 1)) * 10.0 ** rng.uniform(-9, -2, (n, 1)))
    p = np.stack([ca * b[:, 0] - sa * b[:, 1], sa * b[:, 0] + ca * b[:, 1], b[:, 2]], 1)
    x = rng.integers(0, 16000, (n, 3)) * (np.arange(3) < D)
    step = rng.integers(-1, 2, (n, 3)) * (np.arange(3) < D)
    return r, ca, sa, (x - step) - p, x, step


def solid(D, r, ca, sa, c, x):
    d = x - c
    t0 = (ca * d[:, 0] + sa * d[:, 1]) / r[:, 0]
    t1 = (ca * d[:, 1] - sa * d[:, 0]) / r[:, 1]
    t2 = d[:, 2] / r[:, 2] if D == 3 else 0.0
    return t0 * t0 + t1 * t1 + t2 * t2 <= 1.0


@pytest.mark.parametrize("D", [2, 3])
@pytest.mark.parametrize("rmin,rmax", [(0.5, 40.0), (4.0, 4.0), (1.0, 7600.0), (0.05, 7600.0), (1e-3, 7600.0), (1e-6, 7600.0)])
def test_decided_nodes_are_those_of_fp64(sides, D, rmin, rmax):
    r, ca, sa, c, x, step = points(D, 200000, rmin, rmax, 5)
    side, _ = sides(D, r, ca, sa, c, x, step)
    want = solid(D, r, ca, sa, c, x - step)
    wrong = (side != 0) & ((side > 0) != want)
    assert not wrong.any(), (int(wrong.sum()), r[wrong][:3])


def test_ordinary_bodies_are_decided_in_fp32(sides):
    """The margin stays thin for the bodies of the workloads: nodes 5 % off the surface are decided."""
    rng = np.random.default_rng(2)
    n = 1000
    r = np.tile([8.0, 4.0, 4.0], (n, 1))
    side, tol = sides(3, r, np.ones(n), np.zeros(n), np.zeros((n, 3)),
                      rng.integers(-12, 13, (n, 3)), np.zeros((n, 3), int))
    assert tol.max() < 2e-3
    assert (side != 0).mean() > 0.99


@pytest.mark.parametrize("r", [(0.0, 0.0, 0.0), (-3.0, -3.0, -3.0), (1e-40, 5.0, 5.0), (3e38, 1.0, 1.0)])
def test_degenerate_axes_are_never_decided_wrongly(sides, r):
    rng = np.random.default_rng(3)
    n = 500
    x = rng.integers(-6, 7, (n, 3))
    R = np.tile(np.array(r), (n, 1))
    side, _ = sides(3, R, np.ones(n), np.zeros(n), np.zeros((n, 3)), x, np.zeros((n, 3), int))
    with np.errstate(all="ignore"):
        want = solid(3, np.abs(R), np.ones(n), np.zeros(n), np.zeros((n, 3)), x)
    if r[0] == 0.0:
        want = (x == 0).all(1)
    assert not ((side != 0) & ((side > 0) != want)).any()
