"""The V-cycle's kernels at the edges of their ranges (gbpcg_mg_vcycle).

Level kernels: four points a thread inside one coefficient block, four points
across blocks (block edge not a multiple of 4), two points (rows of 4 m + 2
cells), rows longer and shorter than a warp's segments.  The tail of levels up
to 4096 cells: one, two and three levels in shared memory, a coarsest level
swept by one CTA, by the cluster (more than 4096 cells) and in global memory
(one level whose planes are too large).

Solves: the passes on the march (block edges of 4 m and others, odd nz at one
level) and through the TMA ring (an odd ny, a grid above the march's range).
"""
import numpy as np
import pytest
import torch

import oracle
import oracle.mg as mg
from paper_2603_23343_gb300 import inputs
from test_gpu_mg import vcycle_abs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,kb", [
    ((24, 24, 24), 0),     # level 0 above the tail, 12^3 swept by one CTA
    ((24, 20, 40), 6),     # blocks of 6: a thread's points lie in two blocks
    ((24, 20, 40), 4),
    ((16, 24, 24), 1),     # a block per point
    ((48, 48, 44), 8),     # level 1 has rows of 22 cells
    ((8, 8, 512), 8),      # rows of many segments, a tail of one level
    ((16, 16, 16), 8),     # the whole hierarchy in the tail: three levels
    ((8, 16, 32), 3),
    ((8, 8, 8), 0),        # two levels
    ((34, 34, 40), 8),     # coarsest 17 x 17 x 20 on the cluster
    ((17, 17, 20), 8),     # the same as the only level
    ((4, 64, 64), 0),      # one level of 16384 cells, a plane per CTA of the cluster
    ((1, 128, 200), 0),    # one level, swept in global memory
])
def test_vcycle_levels(gpu_lib, shape, kb):
    k, kd = None, None
    if kb:
        k = inputs.lognormal_blocks(*inputs.block_counts(shape[2], shape[1], shape[0], kb), 31).astype(np.float64)
        kd = torch.from_numpy(k).float().cuda()
    r = inputs.uniform_rhs(shape, 32)
    z, levels = gpu_lib.mg_vcycle(torch.from_numpy(r).cuda(), k_block=kd, kb=kb or 8)
    ops = mg.hierarchy(shape, k, kb or 8)
    assert levels == len(ops)
    r64 = r.astype(np.float64)
    # each level's step rounds its sums to FP32: 2e-5 of the sums' absolute values, as for the other shapes
    err = np.abs(z.cpu().double().numpy() - mg.vcycle(ops, r64))
    bound = vcycle_abs(ops, np.abs(r64))
    assert np.all(err <= 2e-5 * bound), float(np.max(err / bound))


@pytest.mark.parametrize("shape,kb", [((24, 20, 40), 6), ((40, 48, 72), 1), ((7, 10, 12), 4), ((17, 17, 20), 8),
                                      ((168, 176, 184), 0)])
def test_mg_solve_passes(gpu_lib, shape, kb):
    k, kd = None, None
    if kb:
        k = inputs.lognormal_blocks(*inputs.block_counts(shape[2], shape[1], shape[0], kb), 33).astype(np.float64)
        kd = torch.from_numpy(k).float().cuda()
    b = inputs.uniform_rhs(shape, 34, dtype=np.float64)
    x, res = gpu_lib.mg_pcg_solve(torch.from_numpy(b).cuda(), tol=1e-6, maxit=500, k_block=kd, kb=kb or 8)
    assert res["status"] == gpu_lib.OK, res
    tr = oracle.true_relres(b, x.cpu().numpy(), k, kb or 8)
    assert tr <= 1e-6 and abs(res["rel_res_true"] - tr) <= 1e-3 * tr
