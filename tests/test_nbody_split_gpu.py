"""Edges of the tiled two-array kernel's split of z (eight CTAs x eight warps, steps of eight
bodies, tiles of 256) and of its 128-body x blocks, within the FP32 bound of test_nbody_gpu.py."""
import numpy as np
import pytest

import workloads as W
from _gpu import requires_gpu
from test_nbody_gpu import as32, check, run

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("eps2", [0.0, 1e-3])
@pytest.mark.parametrize("nx,nz", [(1, 1), (127, 63), (128, 64), (129, 65), (31, 511), (33, 513), (257, 2047),
                                   (5, 2048), (130, 2049), (64, 16385), (1, 0)])
def test_split_edges(ora, nx, nz, eps2):
    x = as32(W.nbody_bodies(nx, 100 + nx))
    z = as32(W.nbody_bodies(max(nz, 1), 200 + nz))[:nz]
    got = run(x, z, eps2)
    assert (got[:, 3] == 0).all()
    if nz == 0:
        assert (got == 0).all()
    else:
        check(ora, x, z, eps2, got)


def test_padding_does_not_meet_a_body_at_the_origin(ora):
    x = np.zeros((3, 4))
    z = as32(W.nbody_bodies(5, 9))
    check(ora, x, z, 1e-30, run(x, z, 1e-30))
