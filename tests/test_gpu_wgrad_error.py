"""Error of the weight gradient against FP64 sums, relative in the Frobenius norm, where the sums are
longest: it comes from the tensor core's accumulator, which truncates, and grows with the number of
voxels a CTA adds up.

Bounds: the errors of the same products taken in tiles of 128 voxels, 304 CTAs (152 for 96 input
channels) with runs of 896 voxels, the mean over six inputs."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ci,co,shape,bound", [(48, 16, (64, 64, 64), 6.26e-7), (16, 16, (64, 64, 64), 6.26e-7),
                                               (16, 32, (32, 64, 128), 6.27e-7), (96, 32, (64, 32, 64), 5.81e-7)])
def test_weight_gradient_error(gpu_lib, ci, co, shape, bound):
    errs = []
    for seed in range(3):
        g = torch.Generator(device="cuda").manual_seed(100 + seed)
        x = torch.relu(torch.randn((*shape, ci), generator=g, device="cuda")).bfloat16()
        gy = (torch.randn((*shape, co), generator=g, device="cuda") * 0.1).bfloat16()
        gw = gpu_lib.conv3_backward_weight(x, gy).double()
        xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1, 1, 1))
        gf = gy.double().reshape(-1, co)
        ref = torch.empty_like(gw)
        nz, ny, nx = shape
        for t in range(27):
            a, b, c = t // 9, t // 3 % 3, t % 3
            ref[:, t] = gf.T @ xp[a:a + nz, b:b + ny, c:c + nx].reshape(-1, ci)
        errs.append(float((gw - ref).norm() / ref.norm()))
    assert sum(errs) / len(errs) <= bound, errs
