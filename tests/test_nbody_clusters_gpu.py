"""Both cluster sizes of the tiled n^2 kernel: the smallest x arrays that four CTAs an x block are taken
for, and the ones before, with z of a tile per CTA and one more; sampled bodies within the FP32 bound
of test_nbody_gpu.py."""
import numpy as np
import pytest
import torch

import workloads as W
from _gpu import requires_gpu
from test_nbody_gpu import as32, check, run

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("eps2", [0.0, 1e-30, 1e-3])
@pytest.mark.parametrize("nz", [1, 1023, 1024, 1025, 2500])
@pytest.mark.parametrize("extra", [0, 1])
def test_cluster_sizes(ora, extra, nz, eps2):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = (6 * sms + 3) // 4                      # x blocks from which four CTAs share one
    nx = 128 * (blocks - 1) + extra                  # the last block empty, or one body
    x, z = as32(W.nbody_bodies(nx, 50 + extra)), as32(W.nbody_bodies(nz, 60 + nz))
    got = run(x, z, eps2)
    assert (got[:, 3] == 0).all()
    check(ora, x, z, eps2, got, rows=np.r_[0:40, nx // 2:nx // 2 + 40, nx - 130:nx])
