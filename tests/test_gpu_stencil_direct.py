"""The plain-load stencil against the TMA engine and the FP64 oracle.

Constant coefficients: bit for bit the engine's result (gbpcg_stencil_apply_variant,
FP32), on sizes either side of the one from which the engine takes over.  Block
coefficients and 16-bit types: within 1e-5 (FP32) or half a unit in the last place
(2^-8, 2^-11) of the oracle relative to the largest entry; blocks cut off at the far
ends, block edges that do not divide a thread's run of planes, one row or plane, and a
base address that TMA cannot take.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_23343_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 4), (5, 3, 32), (17, 40, 36), (64, 64, 64), (125, 250, 256),
                                   (126, 250, 256)])
def test_direct_equals_engine(gpu_lib, shape):
    p = torch.from_numpy(inputs.uniform_rhs(shape, 601)).cuda()
    assert torch.equal(gpu_lib.stencil_apply(p), gpu_lib.stencil_apply_variant(0, p))


@pytest.mark.parametrize("shape,kb", [((1, 1, 1), 8), ((23, 17, 33), 8), ((40, 9, 70), 3), ((19, 21, 64), (4, 5, 6)),
                                      ((50, 1, 257), 16)])
@pytest.mark.parametrize("dtype,bound", [(torch.float32, 1e-5), (torch.bfloat16, 2 ** -8), (torch.float16, 2 ** -11)])
def test_direct_block_coefficients(gpu_lib, shape, kb, dtype, bound):
    kbx, kby, kbz = (kb,) * 3 if isinstance(kb, int) else kb
    nb = (-(-shape[0] // kbz), -(-shape[1] // kby), -(-shape[2] // kbx))
    k = inputs.lognormal_blocks(nb[2], nb[1], nb[0], 602)
    scale = 1.0 if dtype != torch.float16 else 2.0 ** -12  # h^-2 k would overflow FP16
    p = torch.from_numpy(inputs.uniform_rhs(shape, 603) * scale).to(dtype)
    q = gpu_lib.stencil_apply(p.cuda(), k_block=torch.from_numpy(k).cuda(), kb=(kbx, kby, kbz)).cpu().double().numpy()
    full = np.repeat(np.repeat(np.repeat(k, kbz, 0), kby, 1), kbx, 2)[:shape[0], :shape[1], :shape[2]]
    ref = oracle.apply(p.double().numpy(), full.astype(np.float64), 1)
    assert np.max(np.abs(q - ref)) <= bound * np.max(np.abs(ref))


def test_direct_takes_an_unaligned_base(gpu_lib):
    shape = (9, 10, 12)
    store = torch.empty(int(np.prod(shape)) + 1, device="cuda")
    p = store[1:].view(shape)
    p.copy_(torch.from_numpy(inputs.uniform_rhs(shape, 604)))
    assert torch.equal(gpu_lib.stencil_apply(p), gpu_lib.stencil_apply(p.clone()))
