"""The z-marching tensor-core weight gradient at the edges of its range.

|gw - oracle| <= 2e-5 sum_v |gy[v, o] x[v + off(t), i]| element by element,
the bound of the other weight-gradient kernels (sums over voxels in FP32),
and bitwise repeatable.  Rows of one K step up to two x blocks, row counts
that take one to four rows per step, a single plane, channel counts that are
one slice, several, and the largest; columns that end inside a CTA's range.
"""
import numpy as np
import pytest
import torch

import oracle.nn as onn
from paper_2603_23343_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = [((1, 1, 16), 16, 16), ((3, 5, 16), 48, 32), ((4, 6, 32), 16, 16), ((5, 9, 128), 32, 16), ((2, 8, 64), 96, 32),
         ((7, 4, 64), 64, 16), ((3, 2, 128), 48, 16), ((2, 4, 128), 128, 32), ((40, 4, 128), 16, 16),
         ((2, 3, 256), 48, 32), ((33, 12, 32), 80, 16)]


@pytest.mark.parametrize("shape,ci,co", CASES)
def test_weight_gradient_edges(gpu_lib, shape, ci, co):
    nz, ny, nx = shape
    x = torch.from_numpy(inputs.uniform_pm1(401, 0, nz * ny * nx * ci, np.float32).reshape(nz, ny, nx, ci)).bfloat16()
    gy = torch.from_numpy(inputs.uniform_pm1(402, 0, nz * ny * nx * co, np.float32).reshape(nz, ny, nx, co)).bfloat16()
    gw = gpu_lib.conv3_backward_weight(x.cuda(), gy.cuda())
    assert torch.equal(gw, gpu_lib.conv3_backward_weight(x.cuda(), gy.cuda()))
    x64, gy64 = x.double().numpy(), gy.double().numpy()
    ref = onn.conv3_weight_grad(x64, gy64)
    bound = onn.conv3_weight_grad(np.abs(x64), np.abs(gy64))
    assert np.all(np.abs(gw.cpu().double().numpy() - ref) <= 2e-5 * bound + 1e-30)
