"""Steps on streams that cannot be captured, and inside a caller's capture.

lbm_step replays captured graphs. The capture runs on a stream of the handle's own, so
that a handle on the legacy stream steps like any other, any number of steps, and a
caller may capture steps into a graph of its own. The states agree byte for byte with
those of a handle on a stream of its own.
"""
import numpy as np
import pytest

from paper_2009_04604_gb300 import lbm
from paper_2009_04604_gb300 import workloads as W

pytestmark = pytest.mark.gpu
LEGACY = 1  # cudaStreamLegacy


class RawStream:
    def __init__(self, handle):
        self.cuda_stream = handle


def sim(stream, body):
    if body:
        w = W.shear_channel_ellipse(64, 50, ra=5.0, rb=3.0)
    else:
        w = W.sphere_duct((48, 20, 18), 3.0, (14.0, 9.6, 8.7))
    s = lbm.Simulation(w["lattice"], w["dims"], w["tau"], "f32", stream=stream)
    s.set_options("elibb_f", 1.0)
    s.build_geometry(w["base"], w["base_u"], w["shapes"])
    if body:
        s.set_free_body(w["body"], w["inertia"], 8)
    s.init(1.0, (0.01, 0.0, 0.0))
    return s


@pytest.mark.parametrize("body", [False, True])
@pytest.mark.parametrize("steps", [[1], [3, 1, 1], [9], [33, 7]])
def test_legacy_stream(steps, body):
    a, b = sim(None, body), sim(RawStream(LEGACY), body)
    for n in steps * 3:
        a.step(n)
        b.step(n)
    assert a.save() == b.save()


@pytest.mark.parametrize("body", [False, True])
@pytest.mark.parametrize("warm,steps", [(1, 2), (9, 10), (32, 32), (1, 34)])
def test_inside_a_callers_capture(warm, steps, body):
    """Captured after `warm` steps, replayed once: as many steps as were captured."""
    import torch
    a = sim(None, body)
    st = torch.cuda.Stream()
    b = sim(st, body)
    a.step(warm)
    b.step(warm)
    b.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        b.step(steps)
    with torch.cuda.stream(st):
        g.replay()
    a.step(steps)
    b.synchronize()
    assert a.save() == b.save()


@pytest.mark.parametrize("captured", [False, True])
def test_batch(captured):
    """A batch on the legacy stream, and one whose steps the caller captures."""
    import torch
    st = torch.cuda.Stream()
    a, b = sim(None, False), sim(st if captured else RawStream(LEGACY), False)
    batch = [lbm.Batch([s]) for s in (a, b)]
    for x in batch:
        x.step(33)
    b.synchronize()
    batch[0].step(34)
    if captured:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            batch[1].step(34)
        with torch.cuda.stream(st):
            g.replay()
    else:
        batch[1].step(34)
    b.synchronize()
    assert a.save() == b.save()
    for x in batch:
        x.close()
