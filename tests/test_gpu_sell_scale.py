"""Sliced-ELL PCG of right-hand sides of any scale: a solve of 2^k b from 2^k x0 returns 2^k times the
solution of b, bit for bit, where max |b| lies outside [2^-21, 2^20) (the solve then works on the same
scaled system), and to the tolerance within; products of the unscaled FP32 vectors would under- or
overflow at the outer scales."""
import numpy as np
import pytest
import torch

from paper_2603_23343_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("guess", [False, True])
def test_any_scale_of_b(gpu_lib, guess):
    shape = (13, 20, 31)
    m = gpu_lib.sell_from_stencil(shape)
    b = torch.from_numpy(inputs.uniform_rhs(shape, 91, dtype=np.float64)).cuda().ravel()
    x0 = torch.from_numpy(inputs.uniform_rhs(shape, 92, dtype=np.float64)).cuda().ravel() * 1e-3 * float(guess)
    tol = 1e-9
    x1, r1 = gpu_lib.sell_pcg_solve(m, b, x0.clone(), tol=tol, maxit=2000)
    assert r1["status"] == gpu_lib.OK
    ref = None
    for k in (-300, -80, -40, 40, 80, 300):
        s = 2.0 ** k
        x, r = gpu_lib.sell_pcg_solve(m, b * s, x0 * s, tol=tol, maxit=2000)
        assert r["status"] == gpu_lib.OK and r["rel_res_true"] <= tol, (k, r)
        assert abs(r["iters"] - r1["iters"]) <= 2, (k, r["iters"], r1["iters"])
        x = x / s
        assert float((x - x1).norm()) <= 50 * tol * float(x1.norm()), k
        if ref is None:
            ref = x
        assert torch.equal(x, ref), k
    z, r = gpu_lib.sell_pcg_solve(m, torch.zeros_like(b), x0.clone() + 1.0, tol=tol)
    assert r["status"] == gpu_lib.OK and r["iters"] == 0 and not torch.any(z)


def test_a_small_b_and_a_guess_far_off(gpu_lib):
    """The residual of the guess, not b, bounds the scale: the iterations are those of the same guess with b
    within range (whose share of the residual is 1e-14 and less either way)."""
    shape = (13, 20, 31)
    m = gpu_lib.sell_from_stencil(shape)
    b = torch.from_numpy(inputs.uniform_rhs(shape, 93, dtype=np.float64)).cuda().ravel()
    x0 = torch.from_numpy(inputs.uniform_rhs(shape, 94, dtype=np.float64)).cuda().ravel() * 1e13
    xs = []
    for s in (1.0, 2.0 ** -100, 2.0 ** -300):
        x, r = gpu_lib.sell_pcg_solve(m, b * s, x0.clone(), tol=1e-6, maxit=20)
        assert r["status"] == gpu_lib.NOT_CONVERGED and r["iters"] == 20, (s, r)
        xs.append(x)
    for x in xs[1:]:
        assert float((x - xs[0]).norm()) <= 1e-4 * float(xs[0].norm())
