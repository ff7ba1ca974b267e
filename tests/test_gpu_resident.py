"""The on-chip solver against the streaming passes and the oracle.

A constant-coefficient problem that fits the chip is solved by the on-chip
kernel; the same call with tile_cfg set runs the streaming passes.  Both are
Jacobi-PCG with FP32 vectors, FP64 replacements and the same stopping test,
so iterations agree within 2 of the FP64 oracle's, the true residual meets
the tolerance, and x agrees with the passes' to the solves' accuracy.  The
shapes sit at the edges of the bricks: one CTA; rows that are no multiple of
four; fewer rows or planes than bricks have; halos in x; the deepest bricks;
grids one step either side of what fits.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_23343_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [(8, 8, 8), (1, 1, 9), (2, 3, 11), (30, 29, 31), (32, 32, 33), (5, 64, 130), (64, 5, 127),
          (40, 41, 42), (61, 62, 63), (7, 300, 40), (300, 7, 40)]


# FP32 x: grids on which its rounding (about lambda_max 2^-24 |x| / |b|, a few 1e-6 at 300 points along
# an axis of a flat grid) stays well below the tolerance, so that a solve can meet it
SHAPES32 = [s for s in SHAPES if max(s) <= 64]


@pytest.mark.parametrize("shape,io", [(s, np.float64) for s in SHAPES] + [(s, np.float32) for s in SHAPES32])
def test_on_chip_solve_against_oracle_and_passes(gpu_lib, shape, io):
    tol = 1e-5 if io == np.float32 else 1e-7
    b = inputs.uniform_rhs(shape, 301, dtype=io)
    bd = torch.from_numpy(b).cuda()
    x, res = gpu_lib.pcg_solve(bd, tol=tol, maxit=20000)
    b64 = b.astype(np.float64)
    ref = oracle.pcg(b64, tol=tol, maxit=20000)
    assert res["status"] == gpu_lib.OK and abs(res["iters"] - ref["iters"]) <= 2, (res, ref["iters"])
    true_rel = oracle.true_relres(b64, x.cpu().double().numpy())
    assert true_rel <= tol and abs(res["rel_res_true"] - true_rel) <= 1e-3 * true_rel
    cfgs = gpu_lib.tile_configs()
    code = gpu_lib.tile_cfg_code(cfgs.index((64, 16, 4)), cfgs.index((64, 16, 4)))
    xp, rp = gpu_lib.pcg_solve(bd, tol=tol, maxit=20000, tile_cfg=code)
    assert rp["status"] == gpu_lib.OK and abs(res["iters"] - rp["iters"]) <= 2
    # two solutions within tol of the same right-hand side; the oracle tests' accuracy bound
    assert float((x - xp).double().norm()) <= 50 * tol * float(xp.double().norm())


@pytest.mark.parametrize("shape", [(64, 112, 512), (160, 160, 160), (128, 128, 128), (176, 176, 176), (3, 2, 2050)])
def test_on_chip_solve_of_large_and_wide_grids(gpu_lib, shape):
    """The deepest bricks, the whole chip, (176^3) a grid that no longer fits, and rows cut into many
    bricks (so anisotropic that FP32 vectors cannot follow the FP64 iteration to the end, on chip or
    streamed): the first iterations against the oracle's residual history, and a repeated solve bit
    for bit."""
    b = inputs.uniform_rhs(shape, 302, dtype=np.float64)
    bd = torch.from_numpy(b).cuda()
    x, res = gpu_lib.pcg_solve(bd, tol=1e-12, maxit=12)
    ref = oracle.pcg(b, tol=1e-12, maxit=12, history=True)
    assert res["iters"] == 12 and res["status"] == gpu_lib.NOT_CONVERGED
    assert abs(res["rel_res_recursive"] - ref["hist"][12]) <= 1e-4 * ref["hist"][12]
    np.testing.assert_allclose(x.cpu().numpy(), ref["x"], rtol=0, atol=1e-5 * np.max(np.abs(ref["x"])))
    x2, _ = gpu_lib.pcg_solve(bd, tol=1e-12, maxit=12)
    assert torch.equal(x, x2)


@pytest.mark.parametrize("shape", [(20, 20, 23), (64, 64, 96), (80, 112, 256)])
def test_host_loop_on_chip_equals_the_single_launch(gpu_lib, shape):
    """Host-driven iterations save and restore the on-chip state: one build of the kernel per shape
    (up to 4, up to 7, up to 14 planes per thread)."""
    b = torch.from_numpy(inputs.uniform_rhs(shape, 303, dtype=np.float64)).cuda()
    xg, rg = gpu_lib.pcg_solve(b, tol=1e-3, maxit=3000)
    xh, rh = gpu_lib.pcg_solve(b, tol=1e-3, maxit=3000, mode="host_loop")
    assert rg["status"] == rh["status"] == gpu_lib.OK
    assert rg["iters"] == rh["iters"] and rg["replacements"] == rh["replacements"]
    assert torch.equal(xg, xh)


def test_special_values_and_breakdown_agree_with_the_passes(gpu_lib):
    """NaN and infinity in b, an initial guess that already solves, a zero right-hand side: the on-chip
    solve ends with the status and iterations of the passes."""
    shape = (16, 20, 24)
    cfgs = gpu_lib.tile_configs()
    code = gpu_lib.tile_cfg_code(cfgs.index((32, 16, 4)), cfgs.index((32, 16, 4)))
    b0 = inputs.uniform_rhs(shape, 304, dtype=np.float64)
    for bad in (np.nan, np.inf, -np.inf):
        b = b0.copy()
        b[3, 4, 5] = bad
        bd = torch.from_numpy(b).cuda()
        r = [gpu_lib.pcg_solve(bd, tol=1e-6, maxit=50, tile_cfg=c)[1] for c in (0, code)]
        assert r[0]["status"] == r[1]["status"] and r[0]["iters"] == r[1]["iters"], (bad, r)
    bd = torch.from_numpy(b0).cuda()
    x, _ = gpu_lib.pcg_solve(bd, tol=1e-10, maxit=2000)
    _, r = gpu_lib.pcg_solve(bd, x=x.clone(), tol=1e-6, maxit=2000)
    assert r["status"] == gpu_lib.OK and r["iters"] == 0
    z, r = gpu_lib.pcg_solve(torch.zeros_like(bd), x=torch.ones_like(bd))
    assert r["status"] == gpu_lib.OK and r["iters"] == 0 and not torch.any(z)


@pytest.mark.parametrize("io", [torch.float32, torch.float64])
def test_mixed_batch_on_chip_and_streamed(gpu_lib, io):
    """A batch of problems that share a launch, one that fills the chip alone, rows of no multiple of
    four among them: every problem against its own standalone solve."""
    shapes = [(24, 20, 36), (17, 19, 23), (48, 48, 48), (120, 128, 128), (9, 9, 9), (24, 20, 36)]
    tol = 1e-5 if io == torch.float32 else 1e-6
    bs = [torch.from_numpy(inputs.uniform_rhs(sh, 310 + i)).to(io).cuda() for i, sh in enumerate(shapes)]
    xs, res = gpu_lib.pcg_solve_batched(bs, tol=tol, maxit=3000)
    for b, x, r in zip(bs, xs, res):
        x1, r1 = gpu_lib.pcg_solve(b, tol=tol, maxit=3000)
        assert r["status"] == r1["status"] == gpu_lib.OK and abs(r["iters"] - r1["iters"]) <= 2
        assert oracle.true_relres(b.cpu().double().numpy(), x.cpu().double().numpy()) <= tol
        assert float((x - x1).double().norm()) <= 50 * tol * float(x1.double().norm())


def test_batch_waits_for_longer_problems(gpu_lib):
    """Problems that end at once beside problems that iterate for seconds: a problem whose CTAs come from
    both kinds waits for as long as the longer ones take (the limit of its wait counts from the last step
    any problem made).  Twenty flat grids, every second right-hand side zero, fill the chip; the cubes
    after them are larger and expected to take half the time, so each shares its CTAs with several."""
    flat, cube = (20, 30, 201), (59, 60, 61)
    shapes = [flat] * 20 + [cube] * 6
    zero = [i % 2 == 1 for i in range(20)] + [True] * 6
    bs = [torch.from_numpy(inputs.uniform_rhs(s, 320 + i, dtype=np.float64)).cuda() for i, s in enumerate(shapes)]
    for b, z in zip(bs, zero):
        if z:
            b.zero_()
    maxit = 400000
    xs, res = gpu_lib.pcg_solve_batched(bs, tol=1e-30, maxit=maxit)
    for x, r, z in zip(xs, res, zero):
        if z:
            assert r["status"] == gpu_lib.OK and r["iters"] == 0 and not torch.any(x), r
        else:
            assert r["status"] == gpu_lib.NOT_CONVERGED and r["iters"] == maxit, r
    assert res[0]["time_ms"] > 2000.0  # long enough for the limit to matter


@pytest.mark.parametrize("shape", [(32, 32, 32), (64, 64, 64), (3, 5, 9)])
def test_sums_beyond_single_precision_range(gpu_lib, shape):
    """An initial guess so far off that r.r exceeds FP32's largest number, though no thread's part does:
    the grid sums are taken in FP64 there, and the iterations are those of the passes."""
    cfgs = gpu_lib.tile_configs()
    code = gpu_lib.tile_cfg_code(cfgs.index((32, 16, 4)), cfgs.index((32, 16, 4)))
    b = torch.from_numpy(inputs.uniform_rhs(shape, 330, dtype=np.float64)).cuda()
    x0 = torch.from_numpy(inputs.uniform_rhs(shape, 331, dtype=np.float64)).cuda()
    r0 = float(gpu_lib.stencil_apply(x0).norm())
    x0 *= np.sqrt(2e39 if min(shape) > 8 else 1e37) / r0
    its = 12 if min(shape) > 8 else 4
    (xr, r), (xp, p) = [gpu_lib.pcg_solve(b, x0.clone(), tol=1e-6, maxit=its, tile_cfg=c) for c in (0, code)]
    assert r["status"] == p["status"] == gpu_lib.NOT_CONVERGED and r["iters"] == p["iters"] == its, (r, p)
    assert abs(r["rel_res_recursive"] - p["rel_res_recursive"]) <= 1e-3 * p["rel_res_recursive"]
    assert float((xr - xp).norm()) <= 1e-4 * float(xp.norm())


def test_batch_with_a_grid_that_does_not_fit_streams_as_one(gpu_lib):
    """One grid must stream; the others fill the gaps it leaves, in the same launch, rather than going
    before it on chip."""
    shapes = [(160, 160, 160), (32, 32, 32), (64, 64, 64), (192, 192, 192), (48, 48, 48)]
    bs = [torch.from_numpy(inputs.uniform_rhs(sh, 340 + i)).cuda() for i, sh in enumerate(shapes)]
    _, res = gpu_lib.pcg_solve_batched(bs, tol=1e-3, maxit=3000)
    assert all(r["status"] == gpu_lib.OK for r in res) and res[0]["pass_launches"][0] == 1
