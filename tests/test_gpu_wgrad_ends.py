"""The weight gradients of the network's ends (16 -> 1 and 2 -> 16 channels) at the edges of the
tensor-core kernel's chunks, rows, x blocks and CTA ranges, and at a width it does not take.
|gw - oracle| <= 2e-5 sum_v |gy[v, o] x[v + off(t), i]| element by element, the bound of the
other weight-gradient kernels (sums over voxels in FP32), and bitwise repeatable."""
import numpy as np
import pytest
import torch

import oracle.nn as onn
from paper_2603_23343_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 16), (3, 5, 16), (2, 8, 32), (4, 9, 64), (1, 17, 96), (5, 7, 128), (2, 3, 160), (3, 16, 256),
          (40, 16, 128), (3, 4, 8)]


@pytest.mark.parametrize("ci,co", [(16, 1), (2, 16)])
@pytest.mark.parametrize("shape", SHAPES)
def test_weight_gradient_ends(gpu_lib, shape, ci, co):
    nz, ny, nx = shape
    n = nz * ny * nx
    x = torch.from_numpy(inputs.uniform_pm1(411, 0, n * ci, np.float32).reshape(nz, ny, nx, ci)).bfloat16()
    gy = torch.from_numpy(inputs.uniform_pm1(412, 0, n * co, np.float32).reshape(nz, ny, nx, co)).bfloat16()
    xd, gd = x.cuda(), gy.cuda()
    gw = gpu_lib.conv3_backward_weight(xd, gd)
    assert torch.equal(gw, gpu_lib.conv3_backward_weight(xd, gd))
    x64, gy64 = x.double().numpy(), gy.double().numpy()
    ref = onn.conv3_weight_grad(x64, gy64)
    bound = onn.conv3_weight_grad(np.abs(x64), np.abs(gy64))
    assert np.all(np.abs(gw.cpu().double().numpy() - ref) <= 2e-5 * bound + 1e-30)
