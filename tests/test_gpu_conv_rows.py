"""The tensor-core convolution for rows of 16, 32 and 64 voxels at the edges of its tiles.

|y - oracle| <= 2e-5 sum |w x| element by element (BF16 inputs taken exactly,
FP32 accumulation), the bound of the other tensor-core convolutions; with
and without ReLU.  Row counts that leave the last tile or the last CTA partly
outside the grid, one row, one plane, and grids large enough for the most
tiles per CTA.
"""
import numpy as np
import pytest
import torch

import oracle.nn as onn
from paper_2603_23343_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [(1, 2, 64), (3, 10, 64), (2, 1, 64), (2, 2, 32), (5, 12, 32), (1, 8, 16), (4, 4, 16), (3, 24, 16)]
CHANNELS = [(16, 16), (48, 16), (96, 32), (16, 48), (64, 64), (32, 96)]


def case(shape, ci, co, seed):
    n = int(np.prod(shape))
    x = torch.from_numpy(inputs.uniform_pm1(seed, 0, n * ci, np.float32).reshape(*shape, ci)).bfloat16()
    w = torch.from_numpy(inputs.uniform_pm1(seed + 1, 0, co * 27 * ci, np.float32).reshape(co, 27, ci)).bfloat16()
    return x, w


def check(gpu_lib, shape, ci, co, relu):
    x, w = case(shape, ci, co, 500 + ci)
    y = gpu_lib.conv3_forward(x.cuda(), w.cuda(), relu=relu).cpu().double().numpy()
    x64, w64 = x.double().numpy(), w.double().numpy()
    ref = onn.conv3(x64, w64)
    bound = onn.conv3(np.abs(x64), np.abs(w64))
    assert np.all(np.abs(y - (np.maximum(ref, 0.0) if relu else ref)) <= 2e-5 * bound + 1e-30)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ci,co", CHANNELS)
def test_short_rows(gpu_lib, shape, ci, co):
    check(gpu_lib, shape, ci, co, relu=(ci == 16))


@pytest.mark.parametrize("shape,ci,co", [((40, 66, 64), 16, 16), ((40, 66, 64), 16, 32), ((70, 68, 32), 16, 16),
                                         ((66, 40, 16), 32, 64)])
def test_short_rows_many_tiles(gpu_lib, shape, ci, co):
    check(gpu_lib, shape, ci, co, relu=False)


def test_short_rows_keep_special_values(gpu_lib):
    """Infinity and NaN reach exactly the outputs whose taps read them."""
    x, w = case((3, 8, 32), 16, 16, 520)
    x[1, 3, 0, 2], x[2, 7, 31, 5] = float("inf"), float("nan")
    y = gpu_lib.conv3_forward(x.cuda(), w.cuda()).cpu()
    touched = torch.zeros(3, 8, 32, dtype=torch.bool)
    touched[0:3, 2:5, 0:2] = True
    touched[1:3, 6:8, 30:32] = True
    assert torch.equal(~torch.isfinite(y).all(dim=3), touched)
