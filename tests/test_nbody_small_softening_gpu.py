"""Softenings so small that the cube of 1/r of a body's pair with itself is beyond FP32: the pair adds
nothing, in every schedule and form (the change of form lies at eps2 = 2^-66), also for a body at the
origin, where the ring's padding is, and close pairs along an axis.  Bound of test_nbody_gpu.py."""
import numpy as np
import pytest

import workloads as W
from _gpu import requires_gpu
from test_nbody_gpu import as32, check, run

pytestmark = [pytest.mark.gpu, requires_gpu]

SCHEDULES = [{}, dict(ring_p=4, ring_k=1), dict(ring_p=8, ring_k=2), dict(ring_p=16, ring_k=4)]


@pytest.mark.parametrize("eps2", [1e-37, 1e-30, 2.0 ** -84, 2.0 ** -67, float(np.nextafter(np.float32(2.0 ** -66), np.float32(0))), 2.0 ** -66])
@pytest.mark.parametrize("kw", SCHEDULES, ids=lambda kw: "tiled" if not kw else f"ring{kw['ring_p']}")
@pytest.mark.parametrize("n", [1, 129, 1500])
def test_a_body_does_not_act_on_itself(ora, n, kw, eps2):
    x = as32(W.nbody_bodies(n, 300 + n))
    x[:, 3] *= 100.0
    x[0, :3] = 0.0
    got = run(x, x, eps2, **kw)
    assert np.isfinite(got).all() and (got[:, 3] == 0).all()
    check(ora, x, x, eps2, got)


@pytest.mark.parametrize("kw", SCHEDULES, ids=lambda kw: "tiled" if not kw else f"ring{kw['ring_p']}")
def test_close_pairs(ora, kw):
    x = as32(np.array([[0, 0, 0, 1], [1e-15, 0, 0, 2], [0, 3e-15, 0, 0.5], [1, 0, 0, 1]], dtype=np.float64))
    check(ora, x, x, 1e-30, run(x, x, 1e-30, **kw))
