"""Options set between steps.

Setting the options in force again changes nothing and costs next to nothing: graphs and
tile tables stay. Changed options take effect at the next step, whichever way the steps
are launched: directly at first, from short graphs later, from long ones in between.
"""
import time

import numpy as np
import pytest

from paper_2009_04604_gb300 import lbm
from paper_2009_04604_gb300 import workloads as W

pytestmark = pytest.mark.gpu
FORCES = [(1e-5, 0, 0), (0, 2e-5, 0), (0, 0, 0), (-1e-5, 3e-6, 0)]


def sim(body):
    w = W.shear_channel_ellipse(64, 50, ra=5.0, rb=3.0) if body else W.sphere_duct((48, 20, 18), 3.0, (14.0, 9.6, 8.7))
    s = lbm.Simulation(w["lattice"], w["dims"], w["tau"], "f32")
    s.set_options("elibb_f", 1.0)
    s.build_geometry(w["base"], w["base_u"], w["shapes"])
    if body:
        s.set_free_body(w["body"], w["inertia"], 8)
    s.init(1.0, (0.01, 0.0, 0.0))
    return s


def seconds(s, fn, n=40):
    best = 1e30
    for _ in range(5):
        s.synchronize()
        t = time.perf_counter()
        for _ in range(n):
            fn()
        s.synchronize()
        best = min(best, (time.perf_counter() - t) / n)
    return best


@pytest.mark.parametrize("body", [False, True])
def test_same_options_keep_the_graphs(body):
    s = sim(body)
    s.set_options("elibb_f", 1.0, FORCES[0])
    for _ in range(20):
        s.step(1)
    plain = seconds(s, lambda: s.step(1))

    def again():
        s.set_options("elibb_f", 1.0, FORCES[0])
        s.set_wall_neq(lbm.NEQ_BOUNCE_BACK)
        s.set_collision("bgk")
        s.set_refill("equilibrium", 10)
        s.step(1)
    assert seconds(s, again) <= 2.0 * plain + 10e-6


@pytest.mark.parametrize("body", [False, True])
@pytest.mark.parametrize("piece", [1, 3, 8, 9])
def test_changed_options_between_steps(piece, body):
    """`piece` steps at a time against the same steps taken one by one on a fresh handle per
    force (its state handed over), which launches them directly."""
    a = sim(body)
    state = None
    for force in FORCES:
        a.set_options("elibb_f", 1.0, force)
        for _ in range(72 // piece):
            a.step(piece)
        b = sim(body)
        b.set_options("elibb_f", 1.0, force)
        if state is not None:
            b.load(state)
        for _ in range(72):
            b.set_collision("trt")  # a change, so that no graph is kept
            b.set_collision("bgk")
            b.step(1)
        state = b.save()
        assert np.array_equal(a.get_populations(), b.get_populations())
        b.close()
