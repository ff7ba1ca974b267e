"""The convolutions of 1 and 2 to 16 channels at the edges of their rows, x blocks and row groups:
forward 2 -> 16 and the data gradient of 16 -> 1, against the oracle in FP64 on the same BF16 inputs.
|y - ref| <= 2e-6 sum |x w| (54 products at most, exact in FP32, summed in FP32)."""
import numpy as np
import pytest
import torch

import oracle.nn as onn
from paper_2603_23343_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 16), (3, 5, 16), (2, 8, 32), (1, 9, 48), (4, 17, 64), (5, 7, 128), (2, 3, 144), (3, 16, 256),
          (3, 4, 8), (2, 3, 5)]


def bf16(seed, *shape):
    return torch.from_numpy(inputs.uniform_pm1(seed, 0, int(np.prod(shape)), np.float32).reshape(shape)).bfloat16()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("relu", [False, True])
def test_forward_2_to_16(gpu_lib, shape, relu):
    x, w = bf16(421, *shape, 2), bf16(422, 16, 27, 2)
    y = gpu_lib.conv3_forward(x.cuda(), w.cuda(), relu=relu).cpu().double().numpy()
    x64, w64 = x.double().numpy(), w.double().numpy()
    ref = onn.conv3(x64, w64)
    bound = onn.conv3(np.abs(x64), np.abs(w64))
    assert np.all(np.abs(y - (np.maximum(ref, 0) if relu else ref)) <= 2e-6 * bound + 1e-30)


@pytest.mark.parametrize("shape", SHAPES)
def test_data_gradient_16_to_1(gpu_lib, shape):
    gy, w = bf16(423, *shape, 1), bf16(424, 1, 27, 16)
    gx = gpu_lib.conv3_backward_data(gy.cuda(), w.cuda()).cpu().double().numpy()
    # the adjoint: taps mirrored, channels swapped
    wt = np.ascontiguousarray(w.double().numpy()[:, ::-1, :].transpose(2, 1, 0))
    g64 = gy.double().numpy()
    assert np.all(np.abs(gx - onn.conv3(g64, wt)) <= 2e-6 * onn.conv3(np.abs(g64), np.abs(wt)) + 1e-30)
